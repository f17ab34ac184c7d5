// Batched LU with partial pivoting and solve for many small systems of uneven
// size in one persistent launch (paper section 2 -- factor, then forward and
// back substitution -- applied to every system of the batch), and the same
// for Cholesky.
//
// A fixed grid pulls system indices from an atomic counter in the caller's
// order (largest first balances the tail). One CTA of 128 or 256 threads takes one
// whole system at a time; the matrix stays in global memory (L2 holds the
// systems in flight) and is factored right-looking in panels of 16 columns:
//   * panel: one thread per row (two above 256 rows), its 16 values in
//     registers; LU picks the pivot with one warp reduction and one exchange
//     through shared memory per column, Cholesky factors the 16 x 16 diagonal
//     block in one warp and then solves the rows below, thread by row;
//   * LU: the panel's interchanges as one gather/scatter per other column
//     (every thread's row remembers where it came from), then the 16 rows of
//     U, thread by column, in shared memory;
//   * update of the trailing matrix, 32 x 16 tiles per warp, the panel and
//     the rows of U read from shared memory.
// Every element receives the operations of the unblocked elimination in the
// same order (a_ik <- fma(-l_ij, u_jk, a_ik) for ascending j), so blocking
// changes no bit of the result.
//
// What bounds it: in FP64 the FP64 pipe (2 fused multiply-adds per clock and
// SM), so the panel reciprocal is formed by one warp only and tiles are cut so
// that no warp multiplies padding; in FP32 the latency of the column chain,
// hidden by several CTAs per SM (the matrix is not kept in shared memory,
// which would leave room for one).
//
// Measured (4096 systems of order 16 .. 256, factor + solve; before: one
// rank-1 update of the whole matrix per column, three barriers each): LU FP64
// 62.2 -> 14.1 ms (the multiply-adds alone: 11.6 ms at the measured FP64 rate),
// LU FP32 33.1 -> 2.0 ms, Cholesky FP64 (2048 systems) 23.0 -> 4.7 ms.
//
// Systems larger than the launch's shared memory holds (n > 512, or n > max_n)
// are eliminated column by column in place in global memory.
// Nothing here waits on another CTA.
#include <climits>

#include "common.cuh"
#include "internal.h"

namespace gbla {

constexpr int kBatchMaxRhs = 4;

// CTAs per SM the register budget is cut for (256 threads: 3 rather than 2 measured
// 15.2 against 16.5 ms in FP64 LU and 5.7 against 6.6 ms in FP64 Cholesky, spills included).
template <typename T>
constexpr int bt_min_ctas(int nt) {
  return nt > 256 ? 1024 / nt : nt == 256 ? 3 : (sizeof(T) == 4 ? 6 : 5);
}

constexpr int kBtW = 16;  // panel width
constexpr int kBtCap = 512;  // largest order that is factored in panels

// Stride of one column of U in shared memory: 16-byte aligned rows of kBtW
// values, padded by one vector so that consecutive columns start in other banks.
template <typename T>
constexpr int bt_ldu() {
  return kBtW + 16 / (int)sizeof(T);
}

// Dynamic shared memory of one CTA for systems of up to `cap` rows: the panel
// (k-major, cap rows) and the rows of U (cap columns); the solve reuses the
// second part for the right-hand sides and the pivots.
template <typename T>
constexpr size_t bt_smem_bytes(int cap) {
  return (size_t)cap * (kBtW + bt_ldu<T>()) * sizeof(T);
}

template <typename T>
struct alignas(16) BtRow {
  T v[kBtW];
  unsigned hi, lo;  // pivot key: |v| as an integer that orders like the value, 0: no candidate
  int row, src;
};

template <typename T, int NT>
struct BtShared {
  BtRow<T> cand[2][NT / 32];
  BtRow<T> jrow[2];
  T rp;
  T rdiag[kBtW];
  int idx, ndisp, moved, bad;
  int top_src[kBtW];
  int disp[kBtW], disp_src[kBtW];
};

// |a| as two words that order like the value; NaN is no candidate (0, 0).
GBLA_DEVINL void bt_key(float a, unsigned& hi, unsigned& lo) {
  const unsigned b = __float_as_uint(a) & 0x7fffffffu;
  hi = b > 0x7f800000u ? 0u : b + 1u;
  lo = 0u;
}
GBLA_DEVINL void bt_key(double a, unsigned& hi, unsigned& lo) {
  const unsigned h = (unsigned)__double2hiint(a) & 0x7fffffffu;
  const unsigned l = (unsigned)__double2loint(a);
  const bool nan = h > 0x7ff00000u || (h == 0x7ff00000u && l != 0u);
  hi = nan ? 0u : h + 1u;
  lo = nan ? 0u : l;
}
// Warp maximum of the keys; ties go to the lowest row. Returns the winning row
// (INT_MAX when no lane has a candidate) and leaves its key in hi, lo.
template <typename T>
GBLA_DEVINL int bt_warp_argmax(unsigned& hi, unsigned& lo, int row) {
  const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
  unsigned ml = 0u;
  if (sizeof(T) == 8) ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
  const bool tie = mh != 0u && hi == mh && lo == ml;
  const int r = (int)__reduce_min_sync(0xffffffffu, tie ? (unsigned)row : (unsigned)INT_MAX);
  hi = mh;
  lo = ml;
  return r;
}
GBLA_DEVINL float bt_rcp(float x) { return __frcp_rn(x); }
GBLA_DEVINL double bt_rcp(double x) { return __drcp_rn(x); }

// v / d with rd = 1 / d, rounded to nearest. FP64: the quotient v rd corrected once by
// its own residual (Markstein, 1990), which is exact while no exponent is extreme: three
// dependent operations in place of the division's ten, at 64 clocks a warp each.
GBLA_DEVINL float bt_div(float v, float d, float) { return v / d; }
GBLA_DEVINL double bt_div(double v, double d, double rd) {
  const auto plain = [](double x) { return (((unsigned)__double2hiint(x) >> 20) & 0x7ffu) - 128u < 1792u; };
  const double q = v * rd;
  if (!(plain(v) && plain(d) && plain(q))) return v / d;
  return fma(fma(-d, q, v), rd, q);
}

template <typename T>
GBLA_DEVINL void bt_store_row(T* dst, const T (&v)[kBtW]) {
  constexpr int VE = 16 / (int)sizeof(T);
#pragma unroll
  for (int q = 0; q < kBtW / VE; ++q) {
    if constexpr (sizeof(T) == 4)
      reinterpret_cast<float4*>(dst)[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    else
      reinterpret_cast<double2*>(dst)[q] = make_double2(v[2 * q], v[2 * q + 1]);
  }
}
template <typename T>
GBLA_DEVINL void bt_load_row(T (&v)[kBtW], const T* src) {
  constexpr int VE = 16 / (int)sizeof(T);
#pragma unroll
  for (int q = 0; q < kBtW / VE; ++q) {
    if constexpr (sizeof(T) == 4) {
      const float4 x = reinterpret_cast<const float4*>(src)[q];
      v[4 * q] = x.x;
      v[4 * q + 1] = x.y;
      v[4 * q + 2] = x.z;
      v[4 * q + 3] = x.w;
    } else {
      const double2 x = reinterpret_cast<const double2*>(src)[q];
      v[2 * q] = x.x;
      v[2 * q + 1] = x.y;
    }
  }
}

// One LU panel: rows 0 .. m-1 (m <= RPT * NT) and w <= 16 columns of A, thread
// t holding rows t, t + NT. One barrier per column (two in FP64: the
// reciprocal of the pivot costs a dozen FP64 operations, so one warp forms it
// for all): every warp stages its candidate row next to its key, and after
// the barrier each warp picks the winner itself. Leaves L (all rows) k-major
// in Ls, the factored panel in A, and the net row movement in sh.
template <typename T, int NT, int RPT>
__device__ void bt_lu_panel(T* __restrict__ A, int lda, int m, int w, int k0, int* __restrict__ piv,
                            T* __restrict__ Ls, int ldl, BtShared<T, NT>& sh, int& info) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  T a[RPT][kBtW];
  int src[RPT];
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    const int r = tid + NT * i;
    src[i] = r;
#pragma unroll
    for (int k = 0; k < kBtW; ++k) a[i][k] = (r < m && k < w) ? A[r + (size_t)k * lda] : (T)0;
  }
  const bool live = warp * 32 < m;  // a warp without rows never offers a candidate
  if (!live && lane == 0) {
    sh.cand[0][warp].hi = sh.cand[1][warp].hi = 0u;
    sh.cand[0][warp].lo = sh.cand[1][warp].lo = 0u;
    sh.cand[0][warp].row = sh.cand[1][warp].row = INT_MAX;
  }
  if (tid == 0) sh.ndisp = sh.moved = 0;
#pragma unroll
  for (int j = 0; j < kBtW; ++j) {
    if (j < w) {
      const int par = j & 1;
      if (live) {
        unsigned hi = 0u, lo = 0u;
        int row = INT_MAX, ib = 0;
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
          const int r = tid + NT * i;
          if (r >= j && r < m) {
            unsigned h, l;
            bt_key(a[i][j], h, l);
            if (h > hi || (h == hi && l > lo)) {  // ties keep the lower row
              hi = h;
              lo = l;
              row = r;
              ib = i;
            }
          }
        }
        unsigned wh = hi, wl = lo;
        const int wr = bt_warp_argmax<T>(wh, wl, row);
        BtRow<T>& c = sh.cand[par][warp];
        if (wr != INT_MAX ? row == wr : lane == 0) {
#pragma unroll
          for (int i = 0; i < RPT; ++i)
            if (i == ib) {
              bt_store_row<T>(c.v, a[i]);
              c.src = src[i];
            }
          c.hi = wh;
          c.lo = wl;
          c.row = wr;
        }
        if (tid == j) {
          bt_store_row<T>(sh.jrow[par].v, a[0]);
          sh.jrow[par].src = src[0];
        }
      }
      __syncthreads();
      unsigned hi = 0u, lo = 0u;
      int row = INT_MAX;
      if (lane < (NT / 32)) {
        hi = sh.cand[par][lane].hi;
        lo = sh.cand[par][lane].lo;
        row = sh.cand[par][lane].row;
      }
      unsigned wh = hi, wl = lo;
      int p = bt_warp_argmax<T>(wh, wl, row);
      const unsigned bal = __ballot_sync(0xffffffffu, lane < (NT / 32) && row == p);
      const BtRow<T>* pr = p != INT_MAX ? &sh.cand[par][__ffs(bal) - 1] : &sh.jrow[par];
      if (p == INT_MAX) p = j;  // a column of NaN: no interchange
      const T pv = pr->v[j];
      T rp;
      if constexpr (sizeof(T) == 8) {
        if (warp == 0) {
          rp = pv != (T)0 ? bt_rcp(pv) : (T)0;
          if (lane == 0) sh.rp = rp;
        }
        __syncthreads();
        rp = sh.rp;
      } else {
        rp = pv != (T)0 ? bt_rcp(pv) : (T)0;
      }
      if (rp == (T)0 && info == 0) info = k0 + j + 1;
      if (tid == 0) piv[k0 + j] = k0 + p + 1;
      if (live) {
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
          const int r = tid + NT * i;
          if (p != j && (r == j || r == p)) {
            const BtRow<T>* s = r == j ? pr : &sh.jrow[par];
            bt_load_row<T>(a[i], s->v);
            src[i] = s->src;
          }
          if (r > j && r < m) {
            if (rp != (T)0) a[i][j] *= rp;
            const T l = a[i][j];
#pragma unroll
            for (int k = j + 1; k < kBtW; ++k) a[i][k] = fma(-l, pr->v[k], a[i][k]);
          }
        }
      }
    }
  }
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    const int r = tid + NT * i;
    if (r < m) {
#pragma unroll
      for (int k = 0; k < kBtW; ++k)
        if (k < w) {
          A[r + (size_t)k * lda] = a[i][k];
          Ls[r + k * ldl] = a[i][k];
        }
      if (r < w) {
        sh.top_src[r] = src[i];
      } else if (src[i] != r) {
        const int d = atomicAdd(&sh.ndisp, 1);  // at most w rows below the panel's top move
        sh.disp[d] = r;
        sh.disp_src[d] = src[i];
      }
      if (src[i] != r) sh.moved = 1;
    }
  }
  __syncthreads();
}

// The panel's row movement on the columns left of it (k0 of them, at A - k0
// columns) and right of it (nr): lanes 0-15 hold the top rows, lanes 16-31 the
// rows below that change; every load of a column precedes its stores. The top
// rows of the right columns go to Us (the U solve reads them there).
template <typename T, int NT>
__device__ void bt_move_rows(T* __restrict__ A, int lda, int k0, int nr, T* __restrict__ Us,
                             const BtShared<T, NT>& sh) {
  constexpr int LDU = bt_ldu<T>();
  constexpr int U = 4;  // columns in flight per warp
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool moved = sh.moved != 0;
  const int nd = sh.ndisp;
  int dst = -1, s = 0;
  if (lane < kBtW) {
    dst = lane;
    s = sh.top_src[lane];
  } else if (lane - kBtW < nd) {
    dst = sh.disp[lane - kBtW];
    s = sh.disp_src[lane - kBtW];
  }
  const int nl = moved ? k0 : 0;
  for (int q0 = U * warp; q0 < nl + nr; q0 += U * (NT / 32)) {
    T v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int q = q0 + u;
      const int col = q < nl ? q - k0 : kBtW + q - nl;
      v[u] = (q < nl + nr && dst >= 0) ? A[s + (ptrdiff_t)col * lda] : (T)0;
    }
    __syncwarp();
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int q = q0 + u;
      const int col = q < nl ? q - k0 : kBtW + q - nl;
      if (q < nl + nr && dst >= 0) {
        if (q >= nl && lane < kBtW)
          Us[(q - nl) * LDU + lane] = v[u];
        else if (dst != s)
          A[dst + (ptrdiff_t)col * lda] = v[u];
      }
    }
  }
  __syncthreads();
}

// The 16 rows of U over nr columns: u_i <- fma(-l_ik, u_k, u_i), k ascending,
// one thread per column; then back to A, two columns per warp access.
template <typename T, int NT>
__device__ void bt_solve_u(T* __restrict__ A, int lda, int nr, const T* __restrict__ Ls, int ldl,
                           T* __restrict__ Us) {
  constexpr int LDU = bt_ldu<T>();
  for (int c = threadIdx.x; c < nr; c += NT) {
    T u[kBtW];
    bt_load_row<T>(u, Us + c * LDU);
#pragma unroll
    for (int k = 0; k < kBtW; ++k) {
      asm volatile("" ::: "memory");  // keeps the 120 loads of L from being hoisted into registers
#pragma unroll
      for (int i = k + 1; i < kBtW; ++i) u[i] = fma(-Ls[i + k * ldl], u[k], u[i]);
    }
    bt_store_row<T>(Us + c * LDU, u);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < nr * kBtW; e += NT) {
    const int r = e % kBtW, c = e / kBtW;
    A[r + (size_t)(kBtW + c) * lda] = Us[c * LDU + r];
  }
}

// Trailing update of rows / columns 16 .. m-1 (relative to the panel): warp
// tiles of 32 x 16, lane (r, g) rows r and r + 16, columns 2c + g. A half tile
// without rows (or, LOWER, wholly above the diagonal) is skipped, so a warp
// multiplies padding only in the last 16 rows and at the diagonal. LU reads
// U from Us, 16 bytes (kVe values of k) at a time; Cholesky reads L^t from Ls.
template <typename T, bool LOWER, bool H0, bool H1>
GBLA_DEVINL void bt_tile(T* __restrict__ A, int lda, int m, int nr, int wk, const T* __restrict__ Ls,
                         int ldl, const T* __restrict__ Us, int m0, int c0) {
  constexpr int LDU = bt_ldu<T>();
  constexpr int VE = 16 / (int)sizeof(T);
  const int lane = threadIdx.x & 31;
  const int r0 = m0 + (lane & 15), g = lane >> 4;
  T x0[8], x1[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int col = c0 + 2 * c + g;
    const bool ok = col < nr;
    const T* p = A + (size_t)(kBtW + col) * lda;
    if (H0) x0[c] = ok && r0 < m && (!LOWER || r0 >= kBtW + col) ? p[r0] : (T)0;
    if (H1) x1[c] = ok && r0 + 16 < m && (!LOWER || r0 + 16 >= kBtW + col) ? p[r0 + 16] : (T)0;
  }
  const int ra = min(r0, m - 1), rb = min(r0 + 16, m - 1);
  if constexpr (!LOWER) {
#pragma unroll
    for (int k = 0; k < kBtW; k += VE) {
      T a0[VE], a1[VE];
#pragma unroll
      for (int e = 0; e < VE; ++e) {
        if (H0) a0[e] = -Ls[ra + (k + e) * ldl];
        if (H1) a1[e] = -Ls[rb + (k + e) * ldl];
      }
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const int col = min(c0 + 2 * c + g, nr - 1);
        T b[VE];
        if constexpr (sizeof(T) == 4) {
          const float4 v = *reinterpret_cast<const float4*>(Us + col * LDU + k);
          b[0] = v.x;
          b[1] = v.y;
          b[2] = v.z;
          b[3] = v.w;
        } else {
          const double2 v = *reinterpret_cast<const double2*>(Us + col * LDU + k);
          b[0] = v.x;
          b[1] = v.y;
        }
        if (c0 + 2 * c < nr) {
#pragma unroll
          for (int e = 0; e < VE; ++e) {
            if (H0) x0[c] = fma(a0[e], b[e], x0[c]);
            if (H1) x1[c] = fma(a1[e], b[e], x1[c]);
          }
        }
      }
    }
  } else {
#pragma unroll 2
    for (int k = 0; k < wk; ++k) {
      T a0 = (T)0, a1 = (T)0;
      if (H0) a0 = -Ls[ra + k * ldl];
      if (H1) a1 = -Ls[rb + k * ldl];
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const T b = Ls[min(kBtW + c0 + 2 * c + g, m - 1) + k * ldl];
        if (c0 + 2 * c < nr) {
          if (H0) x0[c] = fma(a0, b, x0[c]);
          if (H1) x1[c] = fma(a1, b, x1[c]);
        }
      }
    }
  }
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int col = c0 + 2 * c + g;
    T* p = A + (size_t)(kBtW + col) * lda;
    if (col < nr) {
      if (H0 && r0 < m && (!LOWER || r0 >= kBtW + col)) p[r0] = x0[c];
      if (H1 && r0 + 16 < m && (!LOWER || r0 + 16 >= kBtW + col)) p[r0 + 16] = x1[c];
    }
  }
}

template <typename T, int NT, bool LOWER>
__device__ void bt_update(T* __restrict__ A, int lda, int m, int nr, int wk, const T* __restrict__ Ls,
                          int ldl, const T* __restrict__ Us) {
  const int warp = threadIdx.x >> 5;
  const int tm = (m - kBtW + 31) / 32, tn = (nr + 15) / 16;
  for (int t = warp; t < tm * tn; t += (NT / 32)) {
    const int m0 = kBtW + 32 * (t % tm), c0 = 16 * (t / tm);
    // rows of the two halves; LOWER: a half is needed if its last row reaches the first column
    const bool h0 = !LOWER || m0 + 15 >= kBtW + c0;
    const bool h1 = m0 + 16 < m && (!LOWER || m0 + 31 >= kBtW + c0);
    if (h0 && h1)
      bt_tile<T, LOWER, true, true>(A, lda, m, nr, wk, Ls, ldl, Us, m0, c0);
    else if (h0)
      bt_tile<T, LOWER, true, false>(A, lda, m, nr, wk, Ls, ldl, Us, m0, c0);
    else if (LOWER && h1)
      bt_tile<T, LOWER, false, true>(A, lda, m, nr, wk, Ls, ldl, Us, m0, c0);
  }
}

// One Cholesky panel (rows 0 .. m-1, w <= 16 columns): warp 0 factors the
// diagonal block (lane = row), then thread t solves rows t, t + NT below it.
// d <= 0 (or NaN) in column j stops: columns 0 .. j-1 are done, the others of
// the panel have received their updates. Returns the finished columns.
template <typename T, int NT, int RPT>
__device__ int bt_chol_panel(T* __restrict__ A, int lda, int m, int w, T* __restrict__ Ls, int ldl,
                             BtShared<T, NT>& sh) {
  const int tid = threadIdx.x, lane = tid & 31;
  T x[RPT][kBtW];
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    const int r = tid + NT * i;
#pragma unroll
    for (int k = 0; k < kBtW; ++k) x[i][k] = (r < m && k < w && r >= k) ? A[r + (size_t)k * lda] : (T)0;
  }
  if (tid < 32) {
    int bad = w;
#pragma unroll
    for (int j = 0; j < kBtW; ++j) {
      if (j < w && bad == w) {
        const T d = __shfl_sync(0xffffffffu, x[0][j], j);
        if (!(d > (T)0)) {
          bad = j;
        } else {
          T l, rl;
          sqrt_rcp(d, &l, &rl);
          if (lane == j) x[0][j] = l;
          if (lane > j && lane < w) x[0][j] *= rl;
          if (lane == 0) sh.rdiag[j] = rl;
#pragma unroll
          for (int k = j + 1; k < kBtW; ++k) {
            if (k < w) {
              const T z = fma(-x[0][j], __shfl_sync(0xffffffffu, x[0][j], k), x[0][k]);
              if (lane >= k && lane < w) x[0][k] = z;
            }
          }
        }
      }
    }
    if (lane < w) {
#pragma unroll
      for (int k = 0; k < kBtW; ++k)
        if (k < w) Ls[lane + k * ldl] = x[0][k];
    }
    if (lane == 0) sh.bad = bad;
  }
  __syncthreads();
  const int wk = sh.bad;
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    const int r = tid + NT * i;
    if (r < m && r >= w) {
#pragma unroll
      for (int j = 0; j < kBtW; ++j) {
        if (j < wk) {
          x[i][j] *= sh.rdiag[j];
#pragma unroll
          for (int k = j + 1; k < kBtW; ++k)
            if (k < w) x[i][k] = fma(-x[i][j], Ls[k + j * ldl], x[i][k]);
        }
      }
    }
    if (r < m) {
#pragma unroll
      for (int k = 0; k < kBtW; ++k)
        if (k < w && r >= k) {
          A[r + (size_t)k * lda] = x[i][k];
          if (r >= w) Ls[r + k * ldl] = x[i][k];
        }
    }
  }
  __syncthreads();
  return wk;
}

// One triangular substitution on the n x nrhs right-hand sides b (shared
// memory), 32 rows at a time: a warp per right-hand side solves the diagonal
// block, then every thread updates the rows that remain. The operations on each
// element and their order are those of the row-by-row substitution. Bound, for a
// system alone, by the chain over the rows: the diagonal block is staged in D
// (32 x 32, shared memory), the steps have no branch, and a right-hand side to a
// warp keeps the FP64 operations of a step to one or four. Measured, solve of one
// system of n = 64 with two right-hand sides (before: one warp for both, with a load
// from L2 and a division per step): FP64 LU 131 -> 67 us, Cholesky 182 -> 72.
template <typename T, int NT, bool FWD, bool UNIT, bool TRANS>
__device__ void bt_substitute(const T* a, int ld, int n, int nrhs, T* __restrict__ b, int ldb, T* __restrict__ D) {
  const int tid = threadIdx.x, lane = tid & 31;
  const int nblk = (n + 31) / 32;
  for (int s = 0; s < nblk; ++s) {
    const int k0 = 32 * (FWD ? s : nblk - 1 - s);
    const int kb = min(32, n - k0);
    for (int e = tid; e < 32 * kb; e += NT) {  // D(i, j) of op(a) at [32 j + i]
      const int i = e & 31, j = e >> 5;
      if (TRANS) {
        if (i < kb) D[32 * i + (j ^ i)] = a[k0 + i + (size_t)(k0 + j) * ld];
      } else {
        if (i < kb) D[32 * j + (i ^ j)] = a[k0 + i + (size_t)(k0 + j) * ld];
      }
    }
    __syncthreads();
    const int c = tid >> 5;  // this warp's right-hand side
    if (c < nrhs) {
      T y = lane < kb ? b[k0 + lane + c * ldb] : (T)0;
      T dl = (T)1, rdl = (T)1;  // the lane's diagonal element and its reciprocal
      if (!UNIT && lane < kb) {
        dl = D[32 * lane];
        rdl = bt_rcp(dl);
      }
#pragma unroll 8
      for (int q = 0; q < kb; ++q) {
        const int jj = FWD ? q : kb - 1 - q;
        const T l = D[32 * jj + (lane ^ jj)];
        T x = __shfl_sync(0xffffffffu, y, jj);
        if (!UNIT) x = bt_div(x, __shfl_sync(0xffffffffu, dl, jj), __shfl_sync(0xffffffffu, rdl, jj));
        const T z = fma(-l, x, y);
        y = (FWD ? lane > jj : lane < jj) ? z : (lane == jj ? x : y);
      }
      if (lane < kb) b[k0 + lane + c * ldb] = y;
    }
    __syncthreads();
    const int i_lo = FWD ? k0 + kb : 0, i_hi = FWD ? n : k0;
    for (int i = i_lo + tid; i < i_hi; i += NT) {
      T y[kBatchMaxRhs];
#pragma unroll
      for (int c = 0; c < kBatchMaxRhs; ++c) y[c] = c < nrhs ? b[i + c * ldb] : (T)0;
      const T* col = TRANS ? a + k0 + (size_t)i * ld : a + i + (size_t)k0 * ld;
      const size_t step = TRANS ? 1 : (size_t)ld;
#pragma unroll 8
      for (int q = 0; q < kb; ++q) {
        const int jj = FWD ? q : kb - 1 - q;
        const T l = col[jj * step];
#pragma unroll
        for (int c = 0; c < kBatchMaxRhs; ++c)
          if (c < nrhs) y[c] = fma(-l, b[k0 + jj + c * ldb], y[c]);
      }
#pragma unroll
      for (int c = 0; c < kBatchMaxRhs; ++c)
        if (c < nrhs) b[i + c * ldb] = y[c];
    }
    __syncthreads();
  }
}

// ---- systems too large for the launch's shared memory: column by column in place
// c_i -= l_i u for rows i0, i0 + 32, .. < n of one column, by one warp. Bound by the
// latency of L2: four rows of a lane are loaded before the first is stored (one where
// 1024 threads share the FP64 pipe already). Measured (one LU of n = 1024, FP64; a flat
// index over the square before): 256 threads 467 -> 196 ms, 1024 threads 146 -> 122.
template <typename T, int NT>
GBLA_DEVINL void bt_column_update(T* c, const T* l, T u, int i0, int n) {
  constexpr int NR = sizeof(T) == 8 && NT == 1024 ? 1 : 4;
#pragma unroll 1
  for (int i = i0; i < n; i += 32 * NR) {
    T lv[NR], cv[NR];
#pragma unroll
    for (int q = 0; q < NR; ++q)
      if (i + 32 * q < n) {
        lv[q] = l[i + 32 * q];
        cv[q] = c[i + 32 * q];
      }
#pragma unroll
    for (int q = 0; q < NR; ++q)
      if (i + 32 * q < n) c[i + 32 * q] = fma(-lv[q], u, cv[q]);
  }
}

template <typename T, int NT>
__device__ int bt_lu_in_place(T* a, int ld, int n, int* piv, BtShared<T, NT>& sh) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int info = 0;
  for (int j = 0; j < n; ++j) {
    unsigned hi = 0u, lo = 0u;
    int row = INT_MAX;
    for (int i = j + tid; i < n; i += NT) {
      unsigned h, l;
      bt_key(a[i + (size_t)j * ld], h, l);
      if (h > hi || (h == hi && l > lo)) {
        hi = h;
        lo = l;
        row = i;
      }
    }
    unsigned wh = hi, wl = lo;
    const int wr = bt_warp_argmax<T>(wh, wl, row);
    if (lane == 0) {
      sh.cand[0][warp].hi = wh;
      sh.cand[0][warp].lo = wl;
      sh.cand[0][warp].row = wr;
    }
    __syncthreads();
    hi = lo = 0u;
    row = INT_MAX;
    if (lane < (NT / 32)) {
      hi = sh.cand[0][lane].hi;
      lo = sh.cand[0][lane].lo;
      row = sh.cand[0][lane].row;
    }
    int p = bt_warp_argmax<T>(hi, lo, row);
    if (p == INT_MAX) p = j;
    const T pv = a[p + (size_t)j * ld];
    const T rp = pv != (T)0 ? (T)1 / pv : (T)0;
    if (rp == (T)0 && info == 0) info = j + 1;
    if (tid == 0) piv[j] = p + 1;
    __syncthreads();
    if (p != j)
      for (int c = tid; c < n; c += NT) {
        const T t = a[j + (size_t)c * ld];
        a[j + (size_t)c * ld] = a[p + (size_t)c * ld];
        a[p + (size_t)c * ld] = t;
      }
    __syncthreads();
    if (rp != (T)0)
      for (int i = j + 1 + tid; i < n; i += NT) a[i + (size_t)j * ld] *= rp;
    __syncthreads();
    for (int k = j + 1 + warp; k < n; k += NT / 32)
      bt_column_update<T, NT>(a + (size_t)k * ld, a + (size_t)j * ld, a[j + (size_t)k * ld], j + 1 + lane, n);
    __syncthreads();
  }
  return info;
}

template <typename T, int NT>
__device__ int bt_chol_in_place(T* a, int ld, int n, BtShared<T, NT>& sh) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int j = 0; j < n; ++j) {
    const T d = a[j + (size_t)j * ld];
    if (!(d > (T)0)) return j + 1;  // the same decision in every thread
    const T l = sqrt(d), rl = (T)1 / l;
    __syncthreads();
    if (tid == 0) a[j + (size_t)j * ld] = l;
    for (int i = j + 1 + tid; i < n; i += NT) a[i + (size_t)j * ld] *= rl;
    __syncthreads();
    for (int k = j + 1 + warp; k < n; k += NT / 32)
      bt_column_update<T, NT>(a + (size_t)k * ld, a + (size_t)j * ld, a[k + (size_t)j * ld], k + lane, n);
    __syncthreads();
  }
  return 0;
}

// The next system of the caller's order, or -1.
template <typename T, int NT>
GBLA_DEVINL int bt_next(int batch, const int* __restrict__ order, unsigned* counter, BtShared<T, NT>& sh) {
  __syncthreads();
  if (threadIdx.x == 0) sh.idx = (int)atomicAdd(counter, 1u);
  __syncthreads();
  const int idx = sh.idx;
  if (idx >= batch) return -1;
  return order ? order[idx] : idx;
}

// solve_only: the matrices already hold L\U and ipiv the pivots (a previous
// factor-only launch); only the right-hand sides are solved and written.
template <typename T, int NT, int RPT>
__global__ void __launch_bounds__(NT, bt_min_ctas<T>(NT))
    batched_lu_kernel(int batch, const int* __restrict__ nv, T* const* __restrict__ Av,
                      const int* __restrict__ ldav, int* const* __restrict__ ipivv,
                      const int* __restrict__ nrhsv, T* const* __restrict__ Bv,
                      const int* __restrict__ ldbv, int* __restrict__ infov,
                      const int* __restrict__ order, unsigned* __restrict__ counter, int cap,
                      int solve_only) {
  extern __shared__ double2 bt_smem[];
  T* Ls = reinterpret_cast<T*>(bt_smem);  // [kBtW][cap]
  T* Us = Ls + (size_t)kBtW * cap;        // [cap][bt_ldu]
  __shared__ alignas(16) BtShared<T, NT> sh;
  const int tid = threadIdx.x;
  for (;;) {
    const int sys = bt_next<T, NT>(batch, order, counter, sh);
    if (sys < 0) break;
    const int n = nv[sys];
    const int nrhs = min(nrhsv ? nrhsv[sys] : 0, kBatchMaxRhs);
    T* a = Av[sys];
    const int ld = ldav[sys];
    int* piv = ipivv[sys];
    const bool fits = n <= cap;
    if (!solve_only) {
      int info = 0;
      if (fits) {
        for (int k0 = 0; k0 < n; k0 += kBtW) {
          const int m = n - k0, w = min(kBtW, m), nr = m - w;
          T* P = a + k0 + (size_t)k0 * ld;
          if (RPT == 1 || m <= NT) bt_lu_panel<T, NT, 1>(P, ld, m, w, k0, piv, Ls, cap, sh, info);
          else bt_lu_panel<T, NT, RPT>(P, ld, m, w, k0, piv, Ls, cap, sh, info);
          if (w == kBtW) {
            bt_move_rows<T, NT>(P, ld, k0, nr, Us, sh);
            if (nr > 0) {
              bt_solve_u<T, NT>(P, ld, nr, Ls, cap, Us);
              bt_update<T, NT, false>(P, ld, m, nr, kBtW, Ls, cap, Us);
            }
          } else if (sh.moved) {
            // columns left of a narrow last panel (w rows, all of them top rows)
            for (int c = tid - k0; c < 0; c += NT) {
              T v[kBtW];
#pragma unroll
              for (int r = 0; r < kBtW; ++r) v[r] = r < w ? P[sh.top_src[r] + (ptrdiff_t)c * ld] : (T)0;
#pragma unroll
              for (int r = 0; r < kBtW; ++r)
                if (r < w) P[r + (ptrdiff_t)c * ld] = v[r];
            }
          }
          __syncthreads();
        }
      } else {
        info = bt_lu_in_place<T, NT>(a, ld, n, piv, sh);
      }
      if (tid == 0 && infov) infov[sys] = info;
    }
    if (nrhs <= 0) continue;
    // solve: B <- U^{-1} L^{-1} P B
    T* gB = Bv[sys];
    const int gldb = ldbv[sys];
    __syncthreads();
    T* b = fits ? Us : gB;
    const int ldb = fits ? cap : gldb;
    int* sp = reinterpret_cast<int*>(Us + (size_t)kBatchMaxRhs * cap);
    if (fits) {
      for (int c = 0; c < nrhs; ++c)
        for (int r = tid; r < n; r += NT) b[r + c * ldb] = gB[r + (size_t)c * gldb];
      for (int r = tid; r < n; r += NT) sp[r] = piv[r];
      __syncthreads();
    }
    const int* pp = fits ? sp : piv;
    if (tid < nrhs)
      for (int j = 0; j < n; ++j) {
        const int p = pp[j] - 1;
        if (p > j && p < n) {  // pivots outside j+1 .. n are no interchange
          const T t = b[j + (size_t)tid * ldb];
          b[j + (size_t)tid * ldb] = b[p + (size_t)tid * ldb];
          b[p + (size_t)tid * ldb] = t;
        }
      }
    __syncthreads();
    bt_substitute<T, NT, true, true, false>(a, ld, n, nrhs, b, ldb, Ls);
    bt_substitute<T, NT, false, false, false>(a, ld, n, nrhs, b, ldb, Ls);
    if (fits)
      for (int c = 0; c < nrhs; ++c)
        for (int r = tid; r < n; r += NT) gB[r + (size_t)c * gldb] = b[r + c * ldb];
  }
}

template <typename T, int NT, int RPT>
__global__ void __launch_bounds__(NT, bt_min_ctas<T>(NT))
    batched_chol_kernel(int batch, const int* __restrict__ nv, T* const* __restrict__ Av,
                        const int* __restrict__ ldav, const int* __restrict__ nrhsv,
                        T* const* __restrict__ Bv, const int* __restrict__ ldbv,
                        int* __restrict__ infov, const int* __restrict__ order,
                        unsigned* __restrict__ counter, int cap, int solve_only) {
  extern __shared__ double2 bt_smem[];
  T* Ls = reinterpret_cast<T*>(bt_smem);
  T* Us = Ls + (size_t)kBtW * cap;
  __shared__ alignas(16) BtShared<T, NT> sh;
  const int tid = threadIdx.x;
  for (;;) {
    const int sys = bt_next<T, NT>(batch, order, counter, sh);
    if (sys < 0) break;
    const int n = nv[sys];
    const int nrhs = min(nrhsv ? nrhsv[sys] : 0, kBatchMaxRhs);
    T* a = Av[sys];
    const int ld = ldav[sys];
    const bool fits = n <= cap;
    int info = 0;
    if (!solve_only) {
      if (fits) {
        for (int k0 = 0; k0 < n && info == 0; k0 += kBtW) {
          const int m = n - k0, w = min(kBtW, m), nr = m - w;
          T* P = a + k0 + (size_t)k0 * ld;
          const int wk = (RPT == 1 || m <= NT) ? bt_chol_panel<T, NT, 1>(P, ld, m, w, Ls, cap, sh)
                                                       : bt_chol_panel<T, NT, RPT>(P, ld, m, w, Ls, cap, sh);
          if (wk < w) info = k0 + wk + 1;
          if (nr > 0) bt_update<T, NT, true>(P, ld, m, nr, wk, Ls, cap, nullptr);
          __syncthreads();
        }
      } else {
        info = bt_chol_in_place<T, NT>(a, ld, n, sh);
      }
      if (tid == 0 && infov) infov[sys] = info;
    }
    if (nrhs <= 0 || info != 0) continue;
    // L y = b, then L^t x = y
    T* gB = Bv[sys];
    const int gldb = ldbv[sys];
    __syncthreads();
    T* b = fits ? Us : gB;
    const int ldb = fits ? cap : gldb;
    if (fits) {
      for (int c = 0; c < nrhs; ++c)
        for (int r = tid; r < n; r += NT) b[r + c * ldb] = gB[r + (size_t)c * gldb];
      __syncthreads();
    }
    bt_substitute<T, NT, true, false, false>(a, ld, n, nrhs, b, ldb, Ls);
    bt_substitute<T, NT, false, false, true>(a, ld, n, nrhs, b, ldb, Ls);
    if (fits)
      for (int c = 0; c < nrhs; ++c)
        for (int r = tid; r < n; r += NT) gB[r + (size_t)c * gldb] = b[r + c * ldb];
  }
}

// Launch shape: `cap` (rows the shared memory is sized for), dynamic shared
// memory and the grid, SMs x ctas_per_sm (0: as many CTAs as fit an SM).
template <typename T, int NT, int RPT, typename K>
static cudaError_t bt_shape(K kern, int batch, int max_n, int ctas_per_sm, int* cap, size_t* smem, int* grid) {
  const DeviceProps& dp = device_props();
  constexpr int top = NT * RPT < kBtCap ? NT * RPT : kBtCap;
  int c = max_n < top ? max_n : top;
  // with systems that are eliminated in place, the CTAs the caller asks for per SM
  // are to fit, with panels for what then remains of the shared memory
  if (max_n > kBtCap && ctas_per_sm > 1) {
    const int rows = (int)((dp.smem_optin / ctas_per_sm - 4096) / bt_smem_bytes<T>(1));  // at most 32 CTAs
    if (c > rows) c = rows & ~15;
  }
  if (c < 64) c = 64;  // the solve stages 32 x 32 blocks in the panel's part
  c = (c + 3) & ~3;
  *cap = c;
  *smem = bt_smem_bytes<T>(c);
  cudaError_t e = ensure_dyn_smem(kern, *smem);
  if (e != cudaSuccess) return e;
  if (ctas_per_sm <= 0) {
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ctas_per_sm, kern, NT, *smem);
    if (e != cudaSuccess) return e;
    if (ctas_per_sm < 1) ctas_per_sm = 1;
  }
  *grid = (dp.num_sms > 0 ? dp.num_sms : 1) * ctas_per_sm;
  if (*grid > batch) *grid = batch;
  return cudaSuccess;
}

// Which CTA a batch gets, by the largest order it may hold. FP32 is bound by the
// latency of the column chain, so it takes the smallest CTA that holds the
// panel in registers at two rows per thread and runs more of them per SM (LU,
// orders up to 256: 128 threads 2.28 ms, 256 threads 2.59 ms). FP64 is bound by
// the FP64 pipe and does not care (15.2 / 15.4 ms); 256 threads keep one row
// each, with half the registers. A batch with larger orders, whose elimination in
// place is bound by the loads one CTA has in flight, gets the CTA the caller asks for.
#define GBLA_BT_DISPATCH(RUN)                                        \
  if (max_n <= 128) RUN(128, 1)                                      \
  if (max_n <= 256) {                                                \
    if (sizeof(T) == 4) RUN(128, 2)                                  \
    RUN(256, 1)                                                      \
  }                                                                  \
  if (max_n > kBtCap && threads >= 1024) RUN(1024, 1)                \
  if (max_n > kBtCap && threads >= 512) RUN(512, 1)                  \
  RUN(256, 2)

template <typename T>
cudaError_t launch_lu_batched(int batch, const int* n, T* const* A, const int* lda, int* const* ipiv,
                              const int* nrhs, T* const* B, const int* ldb, int* info,
                              const int* order, int max_n, int threads, int ctas_per_sm, unsigned* counter,
                              bool solve_only, cudaStream_t s) {
  if (batch <= 0) return cudaSuccess;
  cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(unsigned), s);
  if (e != cudaSuccess) return e;
  int cap = 0, grid = 0;
  size_t smem = 0;
#define GBLA_BT_LU(NT, RPT)                                                                        \
  {                                                                                                \
    auto kern = batched_lu_kernel<T, NT, RPT>;                                                     \
    e = bt_shape<T, NT, RPT>(kern, batch, max_n, ctas_per_sm, &cap, &smem, &grid);                 \
    if (e != cudaSuccess) return e;                                                                \
    kern<<<grid, NT, smem, s>>>(batch, n, A, lda, ipiv, nrhs, B, ldb, info, order, counter, cap,   \
                                solve_only ? 1 : 0);                                               \
    count_launch();                                                                                \
    return cudaGetLastError();                                                                     \
  }
  GBLA_BT_DISPATCH(GBLA_BT_LU)
#undef GBLA_BT_LU
}

template <typename T>
cudaError_t launch_chol_batched(int batch, const int* n, T* const* A, const int* lda, const int* nrhs,
                                T* const* B, const int* ldb, int* info, const int* order, int max_n,
                                int threads, int ctas_per_sm, unsigned* counter, bool solve_only, cudaStream_t s) {
  if (batch <= 0) return cudaSuccess;
  cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(unsigned), s);
  if (e != cudaSuccess) return e;
  int cap = 0, grid = 0;
  size_t smem = 0;
#define GBLA_BT_CHOL(NT, RPT)                                                                      \
  {                                                                                                \
    auto kern = batched_chol_kernel<T, NT, RPT>;                                                   \
    e = bt_shape<T, NT, RPT>(kern, batch, max_n, ctas_per_sm, &cap, &smem, &grid);                 \
    if (e != cudaSuccess) return e;                                                                \
    kern<<<grid, NT, smem, s>>>(batch, n, A, lda, nrhs, B, ldb, info, order, counter, cap,         \
                                solve_only ? 1 : 0);                                               \
    count_launch();                                                                                \
    return cudaGetLastError();                                                                     \
  }
  GBLA_BT_DISPATCH(GBLA_BT_CHOL)
#undef GBLA_BT_CHOL
}
#undef GBLA_BT_DISPATCH

#define GBLA_BT_INST(T)                                                                             \
  template cudaError_t launch_lu_batched<T>(int, const int*, T* const*, const int*, int* const*,    \
                                            const int*, T* const*, const int*, int*, const int*,    \
                                            int, int, int, unsigned*, bool, cudaStream_t);          \
  template cudaError_t launch_chol_batched<T>(int, const int*, T* const*, const int*, const int*,   \
                                              T* const*, const int*, int*, const int*, int, int,    \
                                              int, unsigned*, bool, cudaStream_t);
GBLA_BT_INST(double)
GBLA_BT_INST(float)
#undef GBLA_BT_INST

}  // namespace gbla
