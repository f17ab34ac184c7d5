// Forward and back substitution (paper section 2: L y = b, U x = y; and the
// transposed systems used by the gradient and by Cholesky's L^t x = y).
//
// The n rows are cut into 64-row blocks. Each CTA draws a ticket (atomic, in
// start order) that names the block it solves, so a CTA only ever waits on
// blocks owned by CTAs that started before it. For its block b it streams the
// 64 x 64 tiles M(b, q) of every earlier block q in solve order (coalesced
// loads into shared memory in either orientation), waits (bounded) for block
// q's flag, and accumulates M(b, q) x_q; then it solves its diagonal block
// in shared memory (one warp per right-hand side, lanes own rows), writes
// x_b and releases its flag. This kernel takes the systems of one block and
// those with a diagonal block whose inverse is not safe to use; the others go
// to the cluster kernel below.
#include <mutex>

#include "cluster.cuh"
#include "common.cuh"
#include "internal.h"

namespace gbla {

constexpr int kTsBS = 64;
constexpr int kTsNR = 16;

// Right-hand sides are split over two independent chains (the columns of X
// are solved independently), each with its own flags: the FP64 work of a
// chain step halves, and two chains share the SMs without crowding them
// (measured: 16 columns as 2 x 8 beat 4 x 4 and 8 x 2; 8 columns as 2 x 4
// beat 1 x 8).
constexpr int kTsChains = 2;
static int trsv_chains(int nrhs) { return nrhs < 2 ? 1 : kTsChains; }
static size_t trsv_flags_count(int n, int nrhs) {
  return (size_t)trsv_chains(nrhs) * (size_t)((n + kTsBS - 1) / kTsBS) + 1;
}

template <bool LOWER, bool TRANS, bool UNIT>
__global__ void __launch_bounds__(256)
    trsv_chain_kernel(int n, int ncols, int G, int C, const double* __restrict__ T, int ldt,
                      const double* rhs, int ldr, double* X, int ldx, unsigned* flags,
                      const unsigned* gate, int* info, uint64_t wait_ns) {
  if (gate && *gate == 0u) return;  // the inverted diagonal blocks were good: nothing left to do
  constexpr bool FWD = (LOWER != TRANS);
  __shared__ double tile[kTsBS][kTsBS + 1];
  __shared__ double xq[kTsBS][kTsNR];
  __shared__ int s_t, s_abort;
  const int tid = threadIdx.x;
  const int nblk = (n + kTsBS - 1) / kTsBS;
  if (tid == 0) {
    s_t = (int)atomicAdd(&flags[(size_t)C * nblk], 1u);
    s_abort = 0;
  }
  __syncthreads();
  // ticket -> (chain, position in that chain's solve order): a CTA waits only
  // for earlier positions of its own chain, which hold smaller tickets
  const int chain = s_t % C;
  const int t_ord = s_t / C;
  if (t_ord >= nblk) return;
  flags += (size_t)chain * nblk;
  X += (size_t)chain * G * ldx;
  rhs += (size_t)chain * G * ldr;
  const int nrhs = min(G, ncols - chain * G);
  if (nrhs <= 0) return;
  const int b = FWD ? t_ord : nblk - 1 - t_ord;
  const int r0 = b * kTsBS;
  const int nr = min(kTsBS, n - r0);
  const int r = tid & 63, g = tid >> 6;

  auto load_tile = [&](int c0, int nc) {
    for (int idx = tid; idx < kTsBS * kTsBS; idx += blockDim.x) {
      int rr, jj;
      if (!TRANS) {
        rr = idx & 63;
        jj = idx >> 6;
      } else {
        jj = idx & 63;
        rr = idx >> 6;
      }
      double v = 0.0;
      if (rr < nr && jj < nc)
        v = TRANS ? T[(c0 + jj) + (size_t)(r0 + rr) * ldt] : T[(r0 + rr) + (size_t)(c0 + jj) * ldt];
      tile[rr][jj] = v;
    }
  };

  double acc[kTsNR];
#pragma unroll
  for (int c = 0; c < kTsNR; ++c) acc[c] = 0.0;

  for (int st = 0; st < t_ord; ++st) {
    const int q = FWD ? st : nblk - 1 - st;
    const int c0 = q * kTsBS;
    const int nc = min(kTsBS, n - c0);
    __syncthreads();
    load_tile(c0, nc);
    if (tid == 0) {
      if (!gbla_wait_geq(&flags[q], 1u, wait_ns)) {
        gbla_flag_timeout(info);
        s_abort = 1;
      }
      __threadfence();
    }
    __syncthreads();
    if (s_abort) return;
    for (int idx = tid; idx < kTsBS * nrhs; idx += blockDim.x) {
      const int jj = idx & 63, c = idx >> 6;
      xq[jj][c] = jj < nc ? __ldcg(&X[(c0 + jj) + (size_t)c * ldx]) : 0.0;
    }
    __syncthreads();
#pragma unroll 4
    for (int jj = g * 16; jj < g * 16 + 16; ++jj) {
      const double tv = tile[r][jj];
#pragma unroll
      for (int c = 0; c < kTsNR; ++c)
        if (c < nrhs) acc[c] = fma(tv, xq[jj][c], acc[c]);
    }
  }
  // reduce the four partial sums of each row; the right-hand side of block b
  __syncthreads();
  double* part = &tile[0][0];
#pragma unroll
  for (int c = 0; c < kTsNR; ++c)
    if (c < nrhs) part[(g * kTsBS + r) * kTsNR + c] = acc[c];
  __syncthreads();
  for (int idx = tid; idx < kTsBS * nrhs; idx += blockDim.x) {
    const int rr = idx & 63, c = idx >> 6;
    double v = 0.0;
    if (rr < nr) {
      const double sum = (part[(0 * kTsBS + rr) * kTsNR + c] + part[(1 * kTsBS + rr) * kTsNR + c]) +
                         (part[(2 * kTsBS + rr) * kTsNR + c] + part[(3 * kTsBS + rr) * kTsNR + c]);
      v = rhs[(r0 + rr) + (size_t)c * ldr] - sum;
    }
    xq[rr][c] = v;
  }
  __syncthreads();
  load_tile(r0, nr);  // diagonal block
  __syncthreads();
  const int warp = tid >> 5, lane = tid & 31;
  for (int c = warp; c < nrhs; c += (int)(blockDim.x >> 5)) {
    double y0 = xq[lane][c], y1 = xq[lane + 32][c];
    if (FWD) {
      for (int i = 0; i < nr; ++i) {
        double xi = __shfl_sync(0xffffffffu, i < 32 ? y0 : y1, i & 31);
        if (!UNIT) xi = xi / tile[i][i];
        if (lane == (i & 31)) {
          if (i < 32) y0 = xi;
          else y1 = xi;
        }
        if (lane > i) y0 = fma(-tile[lane][i], xi, y0);
        if (lane + 32 > i) y1 = fma(-tile[lane + 32][i], xi, y1);
      }
    } else {
      for (int i = nr - 1; i >= 0; --i) {
        double xi = __shfl_sync(0xffffffffu, i < 32 ? y0 : y1, i & 31);
        if (!UNIT) xi = xi / tile[i][i];
        if (lane == (i & 31)) {
          if (i < 32) y0 = xi;
          else y1 = xi;
        }
        if (lane < i) y0 = fma(-tile[lane][i], xi, y0);
        if (lane + 32 < i) y1 = fma(-tile[lane + 32][i], xi, y1);
      }
    }
    xq[lane][c] = y0;
    xq[lane + 32][c] = y1;
  }
  __syncthreads();
  for (int idx = tid; idx < kTsBS * nrhs; idx += blockDim.x) {
    const int rr = idx & 63, c = idx >> 6;
    if (rr < nr) X[(r0 + rr) + (size_t)c * ldx] = xq[rr][c];
  }
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    st_release_u32(&flags[b], 1u);
  }
}

}  // namespace gbla

// ----------------------------------------------------------------------------
// Substitution with inverted diagonal blocks, the chain in one thread-block
// cluster. With D_s the inverse of the 64 x 64 diagonal block s (s counts in
// solve order, block b = s forward and nblk-1-s backward):
//   y_s = rhs_s - sum_{t < s} T(s, t) x_t,   x_s = D_s y_s.
//
// What bounds it: the dependence from x_{s-1} to x_s. This GPU's FP64 pipe does
// two multiply-adds per clock and SM (a warp's FP64 instruction holds its
// scheduler for 64 clocks), so a 64-row substitution by one warp, or a 64 x 64
// product on one SM, costs microseconds, and so does a round trip through L2.
// Hence: the CTAs of a cluster (8 for one right-hand side, 4 for several) share
// the rows of every block; four warps per right-hand side do the products of a
// step, 2 or 4 rows each (a few multiply-adds and shuffle-adds per lane); y_s and
// x_s are exchanged through the cluster's shared memory (st.async completing bytes
// on the receivers' mbarriers: 200 to 400 clocks); operands are loaded a step
// ahead, from L2, where they were prefetched; one warp fetches the start values of
// y. The chain multiplies the two nearest blocks itself. The blocks before those go
// to helper tasks (32 rows by up to 16 blocks, all right-hand sides of a chain) run
// by all other CTAs, which add their part to the previous task's and pass it on;
// the last one's result starts y_s. They wait for x_t and partial sums in global
// memory, which announce themselves: they start as an all-ones bit pattern (a NaN
// that arithmetic does not produce) and a consumer polls the values it needs.
//
// Split. Up to four chains of right-hand sides, each with its own cluster and
// tasks. Clusters of 8 are the shortest chain (2.5 against 3.2 thousand clocks a
// step), but only 120 of the 152 SMs hold one; 144 hold clusters of 4, and with
// several right-hand sides the helpers' FP64 work counts (n = 8192, 16 columns:
// 5.2 ms for both factors with clusters of 8, 3.2 with 4).
//
// Measured (both factors of one solve): n = 4096, 16 right-hand sides 6.5 -> 1.04
// ms; n = 8192 16.2 -> 3.1 ms; the preconditioner of n = 2500 0.25 -> 0.14 ms.
//
// Progress. Tasks are drawn by ticket, per chain, in solve order, so a task only
// waits for x values and partial sums of tasks already drawn by running CTAs.
// The chain's own CTAs draw tickets too whenever the chain has waited for a
// while, so a chain finishes even if no other CTA of the grid is ever scheduled
// beside it. All waits are bounded.
//
// The operations on a right-hand side and their order depend on n alone: for a given
// factor this is a fixed linear map of rhs (as GMRES requires), whatever CTAs do the
// tasks and whatever other right-hand sides share the launch.
//
// Accuracy. With g = || |D||T_ss| || the product x_s = D_s y_s leaves a residual of
// up to g u |T_ss||x_s| where a substitution leaves u |T_ss||x_s|. g is a few hundred
// for most blocks of U of a dense matrix, less for L and Cholesky factors, and now and
// then thousands (a small pivot inside a block). The set-up computes a bound of it:
// the four CTAs that share a block each leave the largest row sum over their 16
// columns of |D||T_ss|, and g is at most the sum of the four. Blocks whose bound is
// above a limit get one step of refinement, x_s += D_s (y_s - T_ss x_s), which brings
// the residual down by another factor g u; with a block of which one part is above
// kTcMaxPart, or not finite (a zero pivot), the FP64 solves take the substitution
// kernel above instead. The preconditioner needs neither.
// The limit is where the solution is no further from the exact one than that of the
// substitution kernel for the same factors (LU of uniform random matrices, extended
// precision, ratio of the errors' 2-norms, geometric mean over seeds, A and A^t):
//   n                  100        200        300        512        1000       2500
//   limit 1024      1.62 1.57  1.84 1.57  1.36 1.33  1.29 1.02  0.88 0.73  0.68 0.41
//   limit 128       0.91 0.83  0.96 0.95  0.88 0.82  0.80 0.79  0.77 0.60  0.72 0.39
// With few blocks their own residuals are what counts, with many the sums over the
// blocks before them, which are shorter here than in that kernel's chains. The
// refinement of most blocks costs the solve of n = 512 180 -> 214 us, 1000 211 -> 267
// and would cost 4096 451 -> 752.
namespace gbla {

constexpr int kTcWarps = 4;               // chain warps of a CTA per right-hand side
constexpr int kTcRing = 4;                // steps the start values of y may be ahead
constexpr int kTcMaxG = 4;                // right-hand sides of a chain
constexpr int kTcMaxC = 4;                // chains of a launch
constexpr int kTcChunk = 16;              // blocks per helper task
constexpr int kTcNear = 2;                // blocks the chain multiplies itself
constexpr int kTcLone = 4;                // blocks before those that a task takes one by one
constexpr float tc_refine_limit(int n) { return n <= 1024 ? 128.0f : 1024.0f; }
constexpr float kTcMaxPart = 0.25e8f;     // a quarter of the growth that one refinement step is good for
constexpr unsigned long long kXUnset = 0xffffffffffffffffull;

// helper tasks of block s (two row halves by chunks) and of the blocks before it
__host__ __device__ inline int tc_chunks(int s) {
  return s > kTcNear ? (s - kTcNear + kTcChunk - 1) / kTcChunk : 0;
}
__host__ __device__ inline int tc_first(int s) {
  const int m = s - 1 - kTcNear;  // blocks before s that have tasks: 1 .. m far blocks
  if (m <= 0) return 0;
  const int q = m / kTcChunk, r = m % kTcChunk;
  return 2 * (kTcChunk * q * (q + 1) / 2 + r * (q + 1));
}

struct TcShape {
  int C, G;  // chains, right-hand sides of a chain
};
static TcShape tc_shape(int nrhs) {
  TcShape t;
  t.C = nrhs < kTcMaxC ? nrhs : kTcMaxC;
  t.G = (nrhs + t.C - 1) / t.C;
  if (t.G > kTcMaxG) t.G = kTcMaxG;
  return t;
}

// control words: [0, kTcMaxC) tickets, [kTcMaxC] set when a diagonal block's
// inverse is not safe, from kTcCtrl on four per block with the parts of its growth
// (floats; 16-byte aligned), then the substitution kernel's flags
constexpr int kTcCtrl = 2 * kTcMaxC;
static size_t tc_ctrl_words(int n, int nrhs) {
  const int per = nrhs < kTsChains * kTsNR ? nrhs : kTsChains * kTsNR;
  return (kTcCtrl + (size_t)4 * ((n + kTsBS - 1) / kTsBS) + trsv_flags_count(n, per) + 31) / 32 * 32;
}
size_t diag_inv_doubles(int n) {
  return (size_t)((n + kTsBS - 1) / kTsBS) * kTsBS * kTsBS;
}
size_t trsv_scratch_bytes(int n, int nrhs) {
  const int nblk = (n + kTsBS - 1) / kTsBS;
  const TcShape t = tc_shape(nrhs);
  return tc_ctrl_words(n, nrhs) * sizeof(unsigned) +
         (size_t)tc_first(nblk) * t.C * t.G * 32 * sizeof(double);
}

// Tickets to zero, the values that announce themselves to "not yet".
__global__ void __launch_bounds__(256)
    tc_fill_kernel(int n, int ncols, double* X, int ldx, double* P, size_t np, unsigned* ctrl, int ctrl0,
                   int ctrl1) {
  const size_t t0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x, nt = (size_t)gridDim.x * blockDim.x;
  const double unset = __longlong_as_double((long long)kXUnset);
  for (size_t i = t0; i < (size_t)n * ncols; i += nt) X[i % n + (i / n) * ldx] = unset;
  for (size_t i = t0; i < np; i += nt) P[i] = unset;
  // what the set-up found, the words [kTcMaxC, ctrl0), is kept
  for (size_t i = t0; i < (size_t)kTcMaxC; i += nt) ctrl[i] = 0u;
  for (size_t i = ctrl0 + t0; i < (size_t)ctrl1; i += nt) ctrl[i] = 0u;
}

// D_b (row-major, block b of the matrix) of every diagonal block of op(T).
// Bound by the FP64 pipe's latency: 16 x 16 diagonal blocks are inverted by
// columns in registers, the rest of 16 columns per CTA by 16 x 16 products; four
// CTAs share a block, one per 16 columns of the inverse. An upper triangular
// block is handled in reversed index order, which makes it lower triangular. A
// short last block is padded with the identity. Measured: 41 us at n = 4096 (in
// FP64), 75 us at n = 8192; a thread per column took 130.
template <typename Ts, bool TRANS>
__global__ void __launch_bounds__(256)
    tc_diag_inv_kernel(int n, const Ts* __restrict__ T, int ldt, bool fwd, bool unit, double* __restrict__ D,
                       unsigned* bad) {
  __shared__ double E[10][16][17];   // lower triangle of 16 x 16 blocks: (i, k) at i (i + 1) / 2 + k
  __shared__ double I[4][16][17];    // inverses of the diagonal ones
  __shared__ double Xc[4][16][17];   // the CTA's 16 columns of the inverse
  __shared__ double S[16][17];
  __shared__ double rd[64];          // 1 / diagonal
  __shared__ float rs[64];           // sum_k |E_jk / E_jj|
  const int b = blockIdx.x >> 2, g = blockIdx.x & 3;
  const int r0 = b * kTsBS, nr = min(kTsBS, n - r0);
  const int tid = threadIdx.x;
  for (int idx = tid; idx < kTsBS * kTsBS; idx += 256) {
    const int u = idx & 63, v = idx >> 6;  // stored row and column
    const int row = TRANS ? v : u, col = TRANS ? u : v;
    const int i = fwd ? row : 63 - row, j = fwd ? col : 63 - col;
    if (i < j) continue;
    double x;
    if (row >= nr || col >= nr) x = i == j ? 1.0 : 0.0;
    else if (i == j && unit) x = 1.0;
    else x = (double)T[(r0 + u) + (size_t)(r0 + v) * ldt];
    const int bi = i >> 4, bj = j >> 4;
    E[bi * (bi + 1) / 2 + bj][i & 15][j & 15] = x;
  }
  __syncthreads();
  if (tid < 64) rd[tid] = 1.0 / E[(tid >> 4) * ((tid >> 4) + 3) / 2][tid & 15][tid & 15];
  __syncthreads();
  {
    const int w = tid >> 5, j = tid & 31;
    if (w < 4 && w >= g && j < 16) {
      const double(*Ed)[17] = E[w * (w + 3) / 2];
      double s[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) s[i] = i == j ? 1.0 : 0.0;
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        s[i] *= rd[16 * w + i];
#pragma unroll
        for (int k = i + 1; k < 16; ++k) s[k] = fma(-Ed[k][i], s[i], s[k]);
      }
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const double x = i >= j ? s[i] : 0.0;
        I[w][i][j] = x;
        if (w == g) Xc[w][i][j] = x;
      }
    } else if (bad && w >= 4) {
      // scaled row sums, for the growth check: FP32 is enough, and anything that
      // does not fit it is not safe
      const int t = tid - 128, row = t >> 1, q = t & 1;
      float f = 0.f;
      for (int k = q; k < row; k += 2)
        f += fabsf((float)(E[(row >> 4) * ((row >> 4) + 1) / 2 + (k >> 4)][row & 15][k & 15] * rd[row]));
      f += __shfl_xor_sync(0xffffffffu, f, 1);
      if (q == 0) rs[row] = f + 1.f;
    }
  }
  __syncthreads();
  const int r = tid >> 4, c = tid & 15;
  for (int i = g + 1; i < 4; ++i) {
    double a = 0.0;
    for (int k = g; k < i; ++k) {
      const double(*Eik)[17] = E[i * (i + 1) / 2 + k];
#pragma unroll
      for (int q = 0; q < 16; ++q) a = fma(Eik[r][q], Xc[k][q][c], a);
    }
    S[r][c] = a;
    __syncthreads();
    double z = 0.0;
#pragma unroll
    for (int q = 0; q < 16; ++q) z = fma(-I[i][r][q], S[q][c], z);
    Xc[i][r][c] = z;
    __syncthreads();
  }
  if (bad) {
    const int row = tid >> 2, q = tid & 3;
    float f = 0.f;
    if (row >= 16 * g)
      for (int cc = q; cc < 16; cc += 4) {
        const int col = 16 * g + cc;
        const double d = E[g * (g + 3) / 2][cc][cc];
        f += fabsf((float)(Xc[row >> 4][row & 15][cc] * d)) * rs[col];
      }
    f += __shfl_xor_sync(0xffffffffu, f, 1);
    f += __shfl_xor_sync(0xffffffffu, f, 2);
    if (!(f <= kTcMaxPart)) *bad = 1u;
    // floats >= 0 order like their bits
    const unsigned top = __reduce_max_sync(0xffffffffu, __float_as_uint(f));
    if ((tid & 31) == 0) atomicMax(&bad[kTcCtrl - kTcMaxC + blockIdx.x], top);
  }
  double* Db = D + (size_t)b * kTsBS * kTsBS;
  for (int idx = tid; idx < kTsBS * 16; idx += 256) {
    const int i = idx >> 4, cc = idx & 15;
    const int j = 16 * g + cc;
    const double x = (i >> 4) >= g ? Xc[i >> 4][i & 15][cc] : 0.0;
    const int row = fwd ? i : 63 - i, col = fwd ? j : 63 - j;
    Db[row * kTsBS + col] = x;
  }
}

// poll one announced FP64 value (bounded); false on timeout
GBLA_DEVINL unsigned long long tc_load(const double* p) {
  unsigned long long bits;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(bits) : "l"(p) : "memory");
  return bits;
}
GBLA_DEVINL bool tc_poll(const double* p, uint64_t wait_ns, double* out) {
  unsigned long long bits = tc_load(p);
  if (bits == kXUnset) {
    const uint64_t t0 = gbla_now_ns();
    do {
      __nanosleep(32);  // many CTAs may be asking for the same line
      bits = tc_load(p);
      if (gbla_now_ns() - t0 > wait_ns) return false;
    } while (bits == kXUnset);
  }
  *out = __longlong_as_double((long long)bits);
  return true;
}
GBLA_DEVINL void tc_announce(double* p, double v) {
  unsigned long long bits = (unsigned long long)__double_as_longlong(v);
  if (bits == kXUnset) bits = 0x7ff8000000000000ull;  // a NaN handed in by the caller
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(bits) : "memory");
}
GBLA_DEVINL void tc_prefetch(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
// v to another CTA's shared memory, completing 8 bytes on that CTA's mbarrier
GBLA_DEVINL void tc_push(uint32_t raddr, double v, uint32_t rbar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(raddr),
               "l"(__double_as_longlong(v)), "r"(rbar)
               : "memory");
}
// barrier of the helper part; the first, true in every thread if f was in any
template <int H>
GBLA_DEVINL bool tc_help_sync_or(bool f) {
  uint32_t r;
  asm volatile("{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.or.pred q, 1, %2, p;\n selp.u32 %0, 1, 0, q;\n}\n"
               : "=r"(r)
               : "r"((uint32_t)f), "n"(H)
               : "memory");
  return r != 0;
}
template <int H>
GBLA_DEVINL void tc_help_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(H) : "memory");
}

struct TcArgs {
  int n, nblk, ncols, G, C, ldt, ldr, ldx;
  bool fwd, unit;
  const double* D;
  const double* rhs;
  double* X;
  double* P;
  unsigned* ctrl;
  bool gated;
  float refine;  // blocks of larger growth are refined
  int* info;
  uint64_t wait_ns;
};

// threads: helpers, chain warps, the warp that fetches the start values of y
// H helper threads: 256, or 128 in the variant that leaves room for others. The
// latter, also held to 64 registers, is for the preconditioner of systems above 4096
// rows: 288 threads leave an SM room for the 512 threads of 91 registers of such a
// system's panel kernel, which needs 16 SMs of one GPC at the same time and would
// otherwise wait for the whole substitution of another stream's system, and for the
// updates, of LU and Cholesky alike. Three systems of n = 16384 on three streams
// (python bench.py): 185.0 -> 180.6 ms a step; three mixed Cholesky solves of n = 16384
// 64.3 -> 58.2 ms, of 8192 17.6 -> 16.1. One alone pays: mixed LU of n = 8192 23.0 ->
// 23.4 ms, mixed Cholesky 10.6 -> 11.0, of n = 16384 30.4 -> 31.7. The panels of
// smaller systems fit beside the other variant, which is faster (n = 2500, 4
// right-hand sides: 22.5 -> 19.7 ms).
template <int NR, int H>
constexpr int tc_threads() {
  return H + 32 * kTcWarps * NR + 32;
}
constexpr int kTcRoomy = 4096;  // rows up to which the panels fit beside 256 helper threads

template <typename Ts, bool TRANS, int NR, int CL, int H>
__global__ void __launch_bounds__(H == 128 ? 320 : tc_threads<NR, H>(), H == 128 ? 3 : 1)
    tc_solve_kernel(const Ts* __restrict__ T, const TcArgs a) {
  constexpr int kHelp = H;
  constexpr int kHw = kHelp / 32;               // helper warps
  constexpr int kEl = 32 * kTsBS / kHelp;       // elements of a 32 x 64 tile per helper thread
  constexpr int kRows = kTsBS / CL / kTcWarps;  // rows of every block per chain warp
  constexpr int kGrp = 32 / kRows;              // lanes that share a row
  constexpr int kCols = kTsBS / kGrp;           // columns of a block per lane
  constexpr int kAcc = 16 / kGrp;               // of the 16 sums of a row (column mod 16) a lane's
  static_assert(kAcc == 1 || kAcc == 2, "clusters of 8 or 4");
  constexpr int kOwn = kTsBS / CL;              // rows of every block per CTA
  __shared__ double s_x[2][NR][kTsBS];        // x_s, by parity of s
  __shared__ double s_y[2][NR][kTsBS];        // y_s
  __shared__ alignas(8) uint64_t s_bar[2][2][NR];
  __shared__ double s_xq[NR == 1 ? 1 : 2][NR][kTsBS];  // helpers: the x values of a block
  __shared__ double s_xs[2][kHelp / 64][kTsBS];          // or (one right-hand side) of several
  __shared__ double s_part[TRANS ? 32 * 33 : kHw * NR * 32];
  __shared__ volatile double s_y0[kTcRing][NR][kOwn];  // start values of y_s, by s mod kTcRing
  __shared__ volatile int s_have[NR][kOwn];   // steps whose start value is there
  __shared__ volatile int s_step[NR];         // the step the chain's first warp is at
  __shared__ int s_t;
  __shared__ volatile int s_stuck[NR];        // s + 1: chain warp c waits for y_s
  __shared__ int s_done;                      // chain warps that have finished
  __shared__ unsigned s_fail[CL];          // per CTA of the cluster: a wait gave up
  if (a.gated && a.ctrl[kTcMaxC] != 0u) return;  // the substitution kernel takes this system
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int cluster = blockIdx.x / CL;
  const bool in_chain = cluster < a.C;
  const int nblk = a.nblk, n = a.n;
  const int ntask = tc_first(nblk);
  __shared__ int s_failed;

  if (in_chain) {
    if (tid == 0) {
      for (int k = 0; k < 2; ++k)
        for (int p = 0; p < 2; ++p)
          for (int c = 0; c < NR; ++c) {
            cl_mbar_init(cl_smem_u32(&s_bar[k][p][c]), 1);
            cl_mbar_arm(cl_smem_u32(&s_bar[k][p][c]), kTsBS * 8);
          }
      s_done = 0;
      s_failed = 0;
      for (int c = 0; c < NR; ++c) {
        s_stuck[c] = s_step[c] = 0;
        for (int r = 0; r < kOwn; ++r) s_have[c][r] = 0;
      }
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    cl_sync();  // every mbarrier of the cluster is ready for the first push
  }

  if (warp == kHelp / 32 + kTcWarps * NR) {
    // ---- start values of y: rhs, or what the last helper task of the block left;
    // polled here so that the chain never waits for a load it issued too late ------
    if (in_chain) {
      constexpr int kItems = (NR * kOwn + 31) / 32;
      int s[kItems];
#pragma unroll
      for (int i = 0; i < kItems; ++i) s[i] = 0;
      bool more = true;
      while (more) {
        more = false;
#pragma unroll
        for (int i = 0; i < kItems; ++i) {
          const int it = lane + 32 * i, c = it / kOwn, rr = it % kOwn;
          const int col = cluster * a.G + c;
          if (c >= a.G || col >= a.ncols || s[i] >= nblk) continue;
          more = true;
          // the slot's last value has been used: the other warps of the chain are at
          // most one step from its first
          if (s[i] > s_step[c] + kTcRing - 2) continue;
          const int rb = kOwn * (int)cl_ctarank() + rr;
          const int nch = tc_chunks(s[i]);
          unsigned long long bits = 0ull;
          if (nch == 0) {
            const int r = (a.fwd ? s[i] : nblk - 1 - s[i]) * kTsBS + rb;
            if (r < n) bits = tc_load(a.rhs + r + (size_t)col * a.ldr);
          } else {
            const int task = tc_first(s[i]) + 2 * (nch - 1) + (rb >> 5);
            bits = tc_load(a.P + (((size_t)cluster * ntask + task) * a.G + c) * 32 + (rb & 31));
            if (bits == kXUnset) continue;
          }
          s_y0[s[i] % kTcRing][c][rr] = __longlong_as_double((long long)bits);
          __threadfence_block();
          s_have[c][rr] = ++s[i];
        }
        // one decision for the warp; a chain that gave up ends it too
        const bool over = *(volatile int*)&s_done == NR * kTcWarps;
        more = __any_sync(0xffffffffu, more) && !__any_sync(0xffffffffu, over);
      }
    }
  } else if (warp >= kHelp / 32) {
    // ---- chain: four warps per right-hand side, each with its own rows ----------
    const int c = (warp - kHelp / 32) / kTcWarps, wr = (warp - kHelp / 32) % kTcWarps;
    const int col = cluster * a.G + c;
    if (in_chain) {
      bool ok = true;
      if (c < a.G && col < a.ncols) {
        const int row = lane % kRows, grp = lane / kRows;
        const int ro = kRows * wr + row;                     // row among the CTA's
        const int rb = kOwn * (int)cl_ctarank() + ro;        // and in its block
        double* X = a.X + (size_t)col * a.ldx;
        // parity 0 of the row's x and y in the CTA that this lane (of the first
        // kRows CL) serves
        const int to = grp % CL;
        const uint32_t dst_x = cl_mapa(cl_smem_u32(&s_x[0][c][rb]), to), dbar_x = cl_mapa(cl_smem_u32(&s_bar[0][0][c]), to);
        const uint32_t dst_y = cl_mapa(cl_smem_u32(&s_y[0][c][rb]), to), dbar_y = cl_mapa(cl_smem_u32(&s_bar[1][0][c]), to);
        const bool pushes = lane < kRows * CL;
        constexpr uint32_t kBuf = NR * kTsBS * 8, kBar = NR * 8;
        // T(s, s - back), the lane's columns of its row; D_s; where y_s starts from.
        // Only the last block of the matrix can be short: a row block forward in the
        // last step, a column block backward in the first steps.
        auto load_t = [&](int s, int back, Ts (&v)[kCols]) {
          const bool in = s < nblk && s >= back;
          const int b = a.fwd ? s : nblk - 1 - s, q = a.fwd ? s - back : nblk - 1 - s + back;
          const int r = b * kTsBS + rb, c0 = q * kTsBS + grp;
          const Ts* p = TRANS ? T + c0 + (size_t)r * a.ldt : T + r + (size_t)c0 * a.ldt;
          const size_t step = TRANS ? kGrp : (size_t)kGrp * a.ldt;
          if (in && max(b, q) < nblk - 1) {
#pragma unroll
            for (int j = 0; j < kCols; ++j) v[j] = p[j * step];
          } else {
#pragma unroll
            for (int j = 0; j < kCols; ++j) v[j] = (in && r < n && c0 + kGrp * j < n) ? p[j * step] : (Ts)0;
          }
        };
        auto load_d = [&](int s, double (&v)[kCols]) {
          if (s >= nblk) return;
          const double* d = a.D + ((size_t)(a.fwd ? s : nblk - 1 - s) * kTsBS + rb) * kTsBS + grp;
#pragma unroll
          for (int j = 0; j < kCols; ++j) v[j] = d[kGrp * j];
        };
        Ts t1[kCols], t2[kCols];
        double d[kCols];
        load_t(0, 1, t1);
        load_t(0, 2, t2);
        load_d(0, d);
        auto load_growth = [&](int s) {
          return a.gated && s < nblk ? reinterpret_cast<const float4*>(a.ctrl + kTcCtrl)[a.fwd ? s : nblk - 1 - s]
                                     : make_float4(0.f, 0.f, 0.f, 0.f);
        };
        float4 growth = load_growth(0);
        int ny = 0;  // exchanges through s_y so far: one per step, three in a refined one
        // v of every row to every CTA; false if a wait gave up
        auto exchange_y = [&](double v) -> bool {
          const int p = ny & 1;
          if (pushes) tc_push(dst_y + p * kBuf, v, dbar_y + p * kBar);
          const uint32_t ybar = cl_smem_u32(&s_bar[1][p][c]);
          const bool got = cl_mbar_wait(ybar, (uint32_t)(ny >> 1) & 1u, a.wait_ns);
          if (!__all_sync(0xffffffffu, got)) return false;
          if (wr == 0 && lane == 0) cl_mbar_arm(ybar, kTsBS * 8);
          ++ny;
          return true;
        };
        // The 16 sums of a row, added in one order whatever the cluster's size: h and h + 8
        // first (one lane's two, or two lanes'), then the bits of h from the lowest.
        auto row_sum = [&](const double (&p)[kAcc]) {
          double v = p[0] + (kAcc == 2 ? p[kAcc - 1] : __shfl_xor_sync(0xffffffffu, p[0], 16));
#pragma unroll
          for (int o = kRows; o < 8 * kRows; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
          return v;
        };
        auto times_d = [&](double (&dd)[kCols]) {  // D_s times what the last exchange brought
          const double* yv = s_y[(ny - 1) & 1][c];
          double v[kAcc] = {};
#pragma unroll
          for (int j = 0; j < kCols; ++j) v[j % kAcc] = fma(dd[j], yv[grp + kGrp * j], v[j % kAcc]);
          return row_sum(v);
        };
        for (int s = 0; s < nblk; ++s) {
          // every operand is loaded for the next step as soon as this one has used it
          const int par = s & 1;
          double part[kAcc] = {};
          if (s >= 2) {
#pragma unroll
            for (int j = 0; j < kCols; ++j) part[j % kAcc] = fma(-to_f64(t2[j]), s_x[par][c][grp + kGrp * j], part[j % kAcc]);
          }
          load_t(s + 1, 2, t2);
          if (wr == 0 && lane == 0) s_step[c] = s;
          if (!__all_sync(0xffffffffu, s_have[c][ro] > s)) {
            // the helpers are behind
            const uint64_t t0 = gbla_now_ns();
            bool told = false;
            while (!__all_sync(0xffffffffu, s_have[c][ro] > s)) {
              const uint64_t dt = gbla_now_ns() - t0;
              if (__any_sync(0xffffffffu, dt > a.wait_ns)) {
                ok = false;
                break;
              }
              if (__any_sync(0xffffffffu, dt > 4000)) {
                told = true;
                if (lane == 0) s_stuck[c] = s + 1;  // again each time: another warp may have cleared it
              }
            }
            if (told && lane == 0) s_stuck[c] = 0;
            if (!ok) break;
          }
          __threadfence_block();  // s_have before s_y0, as they were written
          if (grp == 0) part[0] += s_y0[s % kTcRing][c][ro];
          if (s >= 1) {
            const uint32_t bar = cl_smem_u32(&s_bar[0][par ^ 1][c]);
            ok = cl_mbar_wait(bar, (uint32_t)((s - 1) >> 1) & 1u, a.wait_ns);
            if (!__all_sync(0xffffffffu, ok)) {
              ok = false;
              break;
            }
            if (wr == 0 && lane == 0) cl_mbar_arm(bar, kTsBS * 8);
#pragma unroll
            for (int j = 0; j < kCols; ++j)
              part[j % kAcc] = fma(-to_f64(t1[j]), s_x[par ^ 1][c][grp + kGrp * j], part[j % kAcc]);
          }
          const double acc = row_sum(part);
          load_t(s + 1, 1, t1);
          ok = exchange_y(acc);
          if (!ok) break;
          double x = times_d(d);
          if ((growth.x + growth.y) + (growth.z + growth.w) > a.refine) {
            // x += D (y - T_ss x)
            ok = exchange_y(x);
            if (!ok) break;
            const int b0 = (a.fwd ? s : nblk - 1 - s) * kTsBS, r = b0 + rb;
            const double* xv = s_y[(ny - 1) & 1][c];
            double rp[kAcc] = {};
            if (grp == 0) rp[0] = acc;
#pragma unroll
            for (int j = 0; j < kCols; ++j) {
              const int cc = grp + kGrp * j, gc = b0 + cc;
              if (r >= n || gc >= n || (a.fwd ? cc > rb : cc < rb)) continue;
              const double tv = cc == rb && a.unit ? 1.0 : (double)(TRANS ? T[gc + (size_t)r * a.ldt] : T[r + (size_t)gc * a.ldt]);
              rp[j % kAcc] = fma(-tv, xv[cc], rp[j % kAcc]);
            }
            ok = exchange_y(row_sum(rp));
            if (!ok) break;
            x += times_d(d);
          }
          if (s + 1 < nblk && pushes) tc_push(dst_x + par * kBuf, x, dbar_x + par * kBar);
          const int r = (a.fwd ? s : nblk - 1 - s) * kTsBS + rb;
          if (grp == 0 && r < n) tc_announce(X + r, x);
          load_d(s + 1, d);
          growth = load_growth(s + 1);
        }
      }
      __syncwarp();
      if (lane == 0) {
        if (!ok) {
          gbla_flag_timeout(a.info);
          atomicExch(&s_failed, 1);
        }
        atomicAdd(&s_done, 1);
      }
      __syncwarp();
    }
  } else {
    // ---- helper tasks ------------------------------------------------------------
    constexpr int kLine = 128 / (int)sizeof(Ts);  // elements of a cache line
    if (in_chain) {
      // the chain's operands (its rows of the blocks (s, s - 1) and (s, s - 2)), in
      // solve order: it loads them only one step ahead, less than HBM's latency
      constexpr int kU = TRANS ? kOwn * 2 * kTsBS / kLine : 2 * kTsBS;  // lines of a step
      for (int i = tid; i < nblk * kU; i += kHelp) {
        const int s = i / kU, u = i % kU;
        const int r = (a.fwd ? s : nblk - 1 - s) * kTsBS + kOwn * (int)cl_ctarank() + (TRANS ? u % kOwn : 0);
        const int off = TRANS ? u / kOwn * kLine : u;  // column among those of the two blocks
        const int cc = a.fwd ? (s - 2) * kTsBS + off : (nblk - s) * kTsBS + off;
        if (r < n && cc >= 0 && cc < n) tc_prefetch(TRANS ? T + cc + (size_t)r * a.ldt : T + r + (size_t)cc * a.ldt);
      }
    }
    for (int q = 0; q < (in_chain ? 1 : a.C); ++q) {
      const int ch = in_chain ? cluster : (int)((blockIdx.x + q) % a.C);
      const int nc = min(a.G, a.ncols - ch * a.G);
      const double* rhs = a.rhs + (size_t)ch * a.G * a.ldr;
      const double* X = a.X + (size_t)ch * a.G * a.ldx;
      double* P = a.P + (size_t)ch * ntask * a.G * 32;
      int s = 0;
      bool stop = false;
      while (nc > 0 && !stop) {
        tc_help_sync<kHelp>();  // the previous task's shared memory is no longer read
        if (tid == 0) {
          bool draw = true;
          if (in_chain) {
            // only while the chain of this CTA is held up by tasks nobody has drawn
            while (true) {
              if (*(volatile int*)&s_done == NR * kTcWarps) {
                draw = false;
                break;
              }
              int st = 0;
              for (int c = 0; c < NR; ++c) st = max(st, s_stuck[c]);
              if (st && *(volatile unsigned*)&a.ctrl[ch] < (unsigned)tc_first(st)) break;
              __nanosleep(500);
            }
          }
          const unsigned t = draw ? atomicAdd(&a.ctrl[ch], 1u) : 0xffffffffu;
          s_t = t < (unsigned)ntask ? (int)t : -1;
        }
        tc_help_sync<kHelp>();
        const int t = s_t;
        if (t < 0) break;
        while (tc_first(s + 1) <= t) ++s;
        const int idx = t - tc_first(s), chunk = idx >> 1, half = idx & 1;
        const int lo = chunk * kTcChunk, hi = min(lo + kTcChunk, s - kTcNear);
        const int r0 = (a.fwd ? s : nblk - 1 - s) * kTsBS + 32 * half;  // first of the 32 rows
        constexpr int NA = TRANS ? kEl / 2 : 1;  // rows of a thread
        double acc[NA][NR];
#pragma unroll
        for (int i = 0; i < NA; ++i)
#pragma unroll
          for (int c = 0; c < NR; ++c) acc[i][c] = 0.0;
        // a thread's elements of a 32 x 64 tile: one row and columns warp + kHw j,
        // or (stored transposed) rows NA warp + i and columns lane + 32 h
        auto load = [&](int sp, Ts (&v)[kEl]) {
          const int c0 = (a.fwd ? sp : nblk - 1 - sp) * kTsBS;
#pragma unroll
          for (int j = 0; j < kEl; ++j) {
            const int rr = TRANS ? r0 + NA * warp + (j >> 1) : r0 + lane;
            const int cc = TRANS ? c0 + lane + 32 * (j & 1) : c0 + warp + kHw * j;
            v[j] = (rr < n && cc < n) ? (TRANS ? T[cc + (size_t)rr * a.ldt] : T[rr + (size_t)cc * a.ldt]) : (Ts)0;
          }
        };
        {
          // the whole task to L2 at once: the loads below reach only one or two tiles
          // ahead, too little for HBM's latency
          const int c0 = (a.fwd ? lo : nblk - hi) * kTsBS, ncol = (hi - lo) * kTsBS;
          constexpr int kPer = 32 / kLine > 0 ? 32 / kLine : 1;  // lines of a 32-row column
          const int lines = TRANS ? 32 * (ncol / kLine) : ncol * kPer;
          for (int i = tid; i < lines; i += kHelp) {
            const int rr = r0 + (TRANS ? i & 31 : i % kPer * kLine), cc = c0 + (TRANS ? (i >> 5) * kLine : i / kPer);
            if (rr < n && cc < n) tc_prefetch(TRANS ? T + cc + (size_t)rr * a.ldt : T + rr + (size_t)cc * a.ldt);
          }
        }
        // one x value per thread: right-hand side xc, row xj of the block (a single
        // right-hand side: of kU blocks at once)
        const int xj = tid & 63, xc = tid >> 6;
        if constexpr (NR == 1) {
          // Little work per tile: a round trip to L2 for x and a barrier per tile would
          // be most of the time. kU blocks share them, but for the last ones of the
          // row, which are waited for one by one.
          const int lone = hi == s - kTcNear ? kTcLone : 0;  // blocks at the end taken singly
          constexpr int kU = kHelp / 64;  // blocks of a group
          Ts cur[kU][kEl];
          int sp = lo, step = hi - lone - lo >= kU ? kU : 1;
          auto fetch = [&](int b0, int nb) {
#pragma unroll
            for (int u = 0; u < kU; ++u)
              if (u < nb) load(b0 + u, cur[u]);
          };
          fetch(sp, step);
          for (int par = 0; sp < hi; par ^= 1) {
            bool late = false;
            const int r = (a.fwd ? sp + xc : nblk - 1 - sp - xc) * kTsBS + xj;
            double xv = 0.0;
            if (xc < step && r < n) late = !tc_poll(X + r, a.wait_ns, &xv);
            s_xs[par][xc][xj] = xv;
            stop = tc_help_sync_or<kHelp>(late);
            if (stop) break;
            const int next = sp + step, nstep = hi - lone - next >= kU ? kU : 1;
#pragma unroll
            for (int u = 0; u < kU; ++u) {
              if (u < step) {
#pragma unroll
                for (int j = 0; j < kEl; ++j) {
                  const int i = TRANS ? j >> 1 : 0, jj = TRANS ? lane + 32 * (j & 1) : warp + kHw * j;
                  acc[i][0] = fma(to_f64(cur[u][j]), s_xs[par][u][jj], acc[i][0]);
                }
              }
              // straight into the registers just used: a move would wait for the load
              if (u < nstep && next + u < hi) load(next + u, cur[u]);
            }
            sp = next;
            step = nstep;
          }
        } else {
          auto x_ptr = [&](int sp) -> const double* {
            const int r = (a.fwd ? sp : nblk - 1 - sp) * kTsBS + xj;
            return xc < nc && r < n ? X + r + (size_t)xc * a.ldx : nullptr;
          };
          // x and tiles are loaded one block ahead, which the work on a tile covers
          Ts cur[kEl], n1[kEl];
          load(lo, cur);
          const double* xp = x_ptr(lo);
          unsigned long long xb = xp ? tc_load(xp) : 0ull;
          for (int sp = lo; sp < hi; ++sp) {
            double(*xq)[kTsBS] = s_xq[sp & 1];
            bool late = false;
            double xv = __longlong_as_double((long long)xb);
            if (xp && xb == kXUnset) late = !tc_poll(xp, a.wait_ns, &xv);
            if (xc < NR) xq[xc][xj] = xv;
            // after the use of x: a wait for it would also wait for loads issued before it
            if (sp + 1 < hi) {
              xp = x_ptr(sp + 1);
              xb = xp ? tc_load(xp) : 0ull;
              load(sp + 1, n1);
            }
            stop = tc_help_sync_or<kHelp>(late);
            if (stop) break;
#pragma unroll
            for (int j = 0; j < kEl; ++j) {
              const double v = to_f64(cur[j]);
              const int i = TRANS ? j >> 1 : 0, jj = TRANS ? lane + 32 * (j & 1) : warp + kHw * j;
#pragma unroll
              for (int c = 0; c < NR; ++c)
                if (c < nc) acc[i][c] = fma(v, xq[c][jj], acc[i][c]);
            }
#pragma unroll
            for (int j = 0; j < kEl; ++j) cur[j] = n1[j];
          }
        }
        if (stop) {
          if (tid == 0) gbla_flag_timeout(a.info);
          break;
        }
        // what was known before this chunk, minus this chunk's sum
        bool late = false;
        auto publish = [&](int rr, int c, double sum) {
          double prev = 0.0;
          if (chunk == 0) {
            if (r0 + rr < n) prev = rhs[r0 + rr + (size_t)c * a.ldr];
          } else if (!tc_poll(P + ((size_t)(t - 2) * a.G + c) * 32 + rr, a.wait_ns, &prev)) {
            late = true;
            return;
          }
          tc_announce(P + ((size_t)t * a.G + c) * 32 + rr, prev - sum);
        };
        if constexpr (!TRANS) {
          double(*part)[NR][32] = reinterpret_cast<double(*)[NR][32]>(s_part);
#pragma unroll
          for (int c = 0; c < NR; ++c)
            if (c < nc) part[warp][c][lane] = acc[0][c];
          tc_help_sync<kHelp>();
          for (int i = tid; i < 32 * nc; i += kHelp) {
            const int rr = i & 31, c = i >> 5;
            double sum = (part[0][c][rr] + part[1][c][rr]) + (part[2][c][rr] + part[3][c][rr]);
            if constexpr (kHw == 8)
              sum += (part[4][c][rr] + part[5][c][rr]) + (part[6][c][rr] + part[7][c][rr]);
            publish(rr, c, sum);
          }
        } else {
          double(*part)[33] = reinterpret_cast<double(*)[33]>(s_part);
#pragma unroll
          for (int c = 0; c < NR; ++c)
            if (c < nc) {
#pragma unroll
              for (int i = 0; i < NA; ++i) part[NA * warp + i][lane] = acc[i][c];
              tc_help_sync<kHelp>();
              constexpr int kPer = kHelp / 32;  // threads of a row
              const int rr = tid / kPer, e = tid % kPer;
              double sum = 0.0;
#pragma unroll
              for (int q = 0; q < 32 / kPer; ++q) sum += part[rr][e + kPer * q];
#pragma unroll
              for (int o = 1; o < kPer; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
              if (e == 0) publish(rr, c, sum);
              tc_help_sync<kHelp>();
            }
        }
        if (tc_help_sync_or<kHelp>(late)) {
          if (tid == 0) gbla_flag_timeout(a.info);
          break;
        }
      }
    }
  }
  if (!in_chain) return;
  // Leaving. On the way through, every push into a CTA was waited for by it. If a
  // wait gave up anywhere in the cluster, pushes may still be on their way: all
  // CTAs learn of it at the first barrier, give them time to land, and leave
  // together after a second one.
  __syncthreads();
  if (tid < CL) cl_store_remote_u32(cl_mapa(cl_smem_u32(&s_fail[cl_ctarank()]), tid), (unsigned)s_failed);
  __syncwarp();
  cl_sync();
  unsigned any = 0;
  for (int q = 0; q < CL; ++q) any |= s_fail[q];
  if (!any) return;
  const uint64_t t0 = gbla_now_ns();
  while (gbla_now_ns() - t0 < 200000) __nanosleep(1000);
  __syncwarp();
  cl_sync();
}

// clusters of CL CTAs that the device can hold at once (0: none)
template <typename Ts, bool TRANS, int NR, int CL, int H>
static cudaError_t tc_max_clusters(int* out) {
  static std::mutex mu;
  static int known[64];
  static bool init = false;
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(mu);
  if (!init) {
    for (int& v : known) v = -1;
    init = true;
  }
  if (known[dev] < 0) {
    cudaLaunchConfig_t q = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CL;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    q.gridDim = dim3(CL);
    q.blockDim = dim3(tc_threads<NR, H>());
    q.attrs = at;
    q.numAttrs = 1;
    int k = 0;
    e = cudaOccupancyMaxActiveClusters(&k, tc_solve_kernel<Ts, TRANS, NR, CL, H>, &q);
    if (e != cudaSuccess) return e;
    known[dev] = k;
  }
  *out = known[dev];
  return cudaSuccess;
}

template <typename Ts, bool TRANS, int NR, int CL, int H>
static cudaError_t tc_launch_solve(const Ts* T, TcArgs a, cudaStream_t s) {
  int maxc = 0;
  cudaError_t e = tc_max_clusters<Ts, TRANS, NR, CL, H>(&maxc);
  if (e != cudaSuccess) return e;
  if (maxc < 1) return cudaErrorNotSupported;
  // one CTA per SM: the FP64 units of an SM, which chain and tasks are bound by,
  // are not shared between two of them. Capped by gbla_set_substitution_ctas.
  int clusters = a.C + (a.C * tc_first(a.nblk) + CL - 1) / CL;
  const int sms = device_props().num_sms / CL;
  if (clusters > maxc) clusters = maxc;
  if (sms > 0 && clusters > sms) clusters = sms;
  const int cap = substitution_ctas();
  if (cap > 0 && clusters > cap / CL) clusters = cap / CL;
  if (clusters < a.C) clusters = a.C;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CL;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)(clusters * CL));
  cfg.blockDim = dim3(tc_threads<NR, H>());
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  count_launch();
  return cudaLaunchKernelEx(&cfg, tc_solve_kernel<Ts, TRANS, NR, CL, H>, T, a);
}

template <typename Ts, bool TRANS>
static cudaError_t tc_launch_diag_inv(bool fwd, bool unit, int n, const Ts* T, int ldt, double* D, unsigned* bad,
                                      cudaStream_t s) {
  tc_diag_inv_kernel<Ts, TRANS><<<4 * ((n + kTsBS - 1) / kTsBS), 256, 0, s>>>(n, T, ldt, fwd, unit, D, bad);
  count_launch();
  return cudaGetLastError();
}

// One group of at most kTcMaxC * kTcMaxG right-hand sides.
template <typename Ts, bool TRANS>
static cudaError_t tc_apply(bool fwd, bool unit, int n, int ncols, TcShape sh, const Ts* T, int ldt, const double* D, const double* rhs,
                            int ldr, double* X, int ldx, char* scratch, size_t ctrl_words, bool gated, int* info,
                            cudaStream_t s) {
  TcArgs a;
  a.n = n;
  a.nblk = (n + kTsBS - 1) / kTsBS;
  a.ncols = ncols;
  a.G = sh.G;
  a.C = (ncols + sh.G - 1) / sh.G;
  a.ldt = ldt;
  a.ldr = ldr;
  a.ldx = ldx;
  a.fwd = fwd;
  a.unit = unit;
  a.D = D;
  a.rhs = rhs;
  a.X = X;
  a.ctrl = reinterpret_cast<unsigned*>(scratch);
  a.P = reinterpret_cast<double*>(scratch + ctrl_words * sizeof(unsigned));
  a.gated = gated;
  a.refine = tc_refine_limit(n);
  a.info = info;
  a.wait_ns = wait_timeout_ns();
  const bool one = ncols == 1;
  if constexpr (sizeof(Ts) == 4) {
    if (n > kTcRoomy && sh.G == 1)
      return one ? tc_launch_solve<Ts, TRANS, 1, 8, 128>(T, a, s) : tc_launch_solve<Ts, TRANS, 1, 4, 128>(T, a, s);
  }
  if (one) return tc_launch_solve<Ts, TRANS, 1, 8, 256>(T, a, s);
  if (sh.G == 1) return tc_launch_solve<Ts, TRANS, 1, 4, 256>(T, a, s);
  if constexpr (sizeof(Ts) == 8) {
    if (sh.G == 2) return tc_launch_solve<Ts, TRANS, 2, 4, 256>(T, a, s);
    return tc_launch_solve<Ts, TRANS, 4, 4, 256>(T, a, s);
  }
  return cudaErrorInvalidValue;  // the preconditioner takes at most kTcMaxC columns
}

// keep_bad: what the set-up found about the inverses is left as it is.
static cudaError_t tc_fill(int n, int ncols, TcShape sh, double* X, int ldx, char* scratch, size_t ctrl_words,
                           bool keep_bad, cudaStream_t s) {
  const size_t np = (size_t)tc_first((n + kTsBS - 1) / kTsBS) * sh.C * sh.G * 32;
  const size_t work = (size_t)n * ncols + np + ctrl_words;
  size_t grid = (work + 1023) / 1024;
  if (grid > 608) grid = 608;
  tc_fill_kernel<<<(unsigned)grid, 256, 0, s>>>(n, ncols, X, ldx,
                                                reinterpret_cast<double*>(scratch + ctrl_words * sizeof(unsigned)), np,
                                                reinterpret_cast<unsigned*>(scratch),
                                                keep_bad ? kTcCtrl + 4 * ((n + kTsBS - 1) / kTsBS) : kTcMaxC,
                                                (int)ctrl_words);
  count_launch();
  return cudaGetLastError();
}

// X = op(T)^-1 rhs (distinct buffers), FP64. D: diag_inv_doubles(n) doubles.
cudaError_t launch_trsv(bool lower, bool trans, bool unit, int n, int nrhs, const double* T, int ldt,
                        const double* rhs, int ldr, double* X, int ldx, double* D, void* scratch, int* info,
                        cudaStream_t s) {
  if (n <= 0 || nrhs <= 0) return cudaSuccess;
  if (!lower && unit) return cudaErrorInvalidValue;  // no factorisation leaves one
  const int nblk = (n + kTsBS - 1) / kTsBS;
  const uint64_t wait_ns = wait_timeout_ns();
  const bool fwd = lower != trans;
  const size_t cw = tc_ctrl_words(n, nrhs);
  char* sc = static_cast<char*>(scratch);
  unsigned* ctrl = reinterpret_cast<unsigned*>(sc);
  // A system of one block has no chain: its substitution alone is shorter than
  // inverting the block first, and takes kTsChains x kTsNR columns a launch with
  // nothing to prepare but its flags (measured, n = 32, 256 columns: 863 -> 660 us; n
  // = 1 434 -> 240).
  const bool blocks = nblk > 1;
  const TcShape sh = tc_shape(nrhs);
  const int per = blocks ? sh.C * sh.G : kTsChains * kTsNR;
  unsigned* flags = ctrl + kTcCtrl + 4 * nblk;
  for (int c0 = 0; c0 < nrhs; c0 += per) {
    const int ncols = nrhs - c0 < per ? nrhs - c0 : per;
    const double* R = rhs + (size_t)c0 * ldr;
    double* Xc = X + (size_t)c0 * ldx;
    cudaError_t e = blocks ? tc_fill(n, ncols, sh, Xc, ldx, sc, cw, c0 > 0, s)
                           : cudaMemsetAsync(flags, 0, sizeof(unsigned) * trsv_flags_count(n, ncols), s);
    if (e != cudaSuccess) return e;
    if (blocks) {
      if (c0 == 0) {
        e = trans ? tc_launch_diag_inv<double, true>(fwd, unit, n, T, ldt, D, ctrl + kTcMaxC, s)
                  : tc_launch_diag_inv<double, false>(fwd, unit, n, T, ldt, D, ctrl + kTcMaxC, s);
        if (e != cudaSuccess) return e;
      }
      e = trans ? tc_apply<double, true>(fwd, unit, n, ncols, sh, T, ldt, D, R, ldr, Xc, ldx, sc, cw, true, info, s)
                : tc_apply<double, false>(fwd, unit, n, ncols, sh, T, ldt, D, R, ldr, Xc, ldx, sc, cw, true, info, s);
      if (e != cudaSuccess) return e;
    }
    const int C = trsv_chains(ncols);
    const int G = (ncols + C - 1) / C;
    const int Cl = (ncols + G - 1) / G;  // chains that hold columns
    const int grid = Cl * nblk;
    const unsigned* gate = blocks ? ctrl + kTcMaxC : nullptr;
#define GBLA_TRSV(LW, TR, UN)                                                                         \
  trsv_chain_kernel<LW, TR, UN><<<grid, 256, 0, s>>>(n, ncols, G, Cl, T, ldt, R, ldr, Xc, ldx, flags, \
                                                     gate, info, wait_ns)
    if (lower && !trans && unit) GBLA_TRSV(true, false, true);
    else if (lower && !trans && !unit) GBLA_TRSV(true, false, false);
    else if (lower && trans && unit) GBLA_TRSV(true, true, true);
    else if (lower && trans && !unit) GBLA_TRSV(true, true, false);
    else if (!trans) GBLA_TRSV(false, false, false);
    else GBLA_TRSV(false, true, false);
#undef GBLA_TRSV
    count_launch();
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// The preconditioner's factors: the inverses once per set of factors ...
cudaError_t launch_diag_inv(bool lower, bool unit, int n, const float* T, int ldt, double* D, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  return tc_launch_diag_inv<float, false>(lower, unit, n, T, ldt, D, nullptr, s);
}

// ... and X = T^-1 rhs (at most kTcMaxC columns, distinct buffers) as a fixed
// linear map
cudaError_t launch_trsv_inv(bool lower, int n, int nrhs, const float* T, int ldt, const double* D, const double* rhs,
                            int ldr, double* X, int ldx, void* scratch, int* info, cudaStream_t s) {
  if (n <= 0 || nrhs <= 0) return cudaSuccess;
  if (nrhs > kTcMaxC) return cudaErrorInvalidValue;
  const size_t cw = tc_ctrl_words(n, nrhs);
  const TcShape sh = tc_shape(nrhs);
  char* sc = static_cast<char*>(scratch);
  cudaError_t e = tc_fill(n, nrhs, sh, X, ldx, sc, cw, false, s);
  if (e != cudaSuccess) return e;
  return tc_apply<float, false>(lower, false, n, nrhs, sh, T, ldt, D, rhs, ldr, X, ldx, sc, cw, false, info, s);
}

}  // namespace gbla
