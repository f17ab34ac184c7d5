// Cholesky factorisation A = L L^t of an SPD matrix (paper section 2), lower
// triangle, blocked right-looking: outer blocks of nb columns (64 .. 256,
// autotunable), each processed in 64-column steps:
//   potf2   -- the 64 x 64 diagonal block factored by one CTA in shared memory
//              (column by column: d = a_jj, stop with info = j + 1 if d <= 0,
//              l_jj = sqrt(d), l_ij = a_ij * (1 / l_jj), a_ik -= l_ij l_kj);
//   trsm    -- the rows below it: L21 = A21 L11^{-t} (four lanes per row, its
//              values in registers, the triangle in shared memory);
//   update  -- A22 -= L21 L21^t on the lower triangle (the SIMT GEMM with its
//              lower-triangle mask; tiles above the diagonal are skipped):
//              inside the outer block for its remaining columns, then once
//              per outer block (rank nb) for the trailing matrix.
// The strict upper triangle of A is never read or written.
#include "common.cuh"
#include "internal.h"

namespace gbla {

constexpr int kCholNb = 64;

// The kb x kb diagonal block (kb <= 64) in shared memory, FP64: column by column.
// A GPU-wide FP64 rate of
// 2 multiply-adds per clock and SM is half a lane per clock for each of its
// four schedulers: one FP64 instruction of one warp takes 64 clocks however few
// of its lanes are active. So per column the reciprocal root is formed by one
// warp only, which first updates the next diagonal element and then works on
// it while the other seven update the rest of the triangle, each warp with 32
// live elements of it (columns c and m - 1 - c of the triangle are m + 1
// elements together).
// d <= 0 (or NaN) stops; the columns to the right have received the updates of
// the finished ones. An earlier block that failed leaves the rest of the
// factor undefined; the first failure stays in info.
__global__ void __launch_bounds__(256)
    potf2_f64_kernel(int kb, double* __restrict__ A, int lda, int row0, int* __restrict__ info) {
  typedef double T;
  __shared__ T D[kCholNb][kCholNb + 1];
  __shared__ T s_rl;
  __shared__ int s_bad;
  const int tid = threadIdx.x;
  for (int idx = tid; idx < kCholNb * kCholNb; idx += blockDim.x) {
    const int r = idx & 63, c = idx >> 6;
    D[r][c] = (r < kb && c < kb && r >= c) ? A[r + (size_t)c * lda] : (T)0;
  }
  if (tid == 0) s_bad = kCholNb;
  __syncthreads();
  // d = the finished diagonal element of column j (one warp)
  auto root = [&](int j, T d) {
    if (!(d > (T)0)) {
      if (tid == 0) {
        s_bad = j;
        D[j][j] = d;
        atomicCAS(info, 0, row0 + j + 1);
      }
    } else {
      T l, rl;
      sqrt_rcp(d, &l, &rl);
      if (tid == 0) {
        D[j][j] = l;
        s_rl = rl;
      }
    }
  };
  if (tid < 32) root(0, D[0][0]);
  __syncthreads();
  for (int j = 0; j < kb && s_bad > j; ++j) {
    const T rl = s_rl;
    if (tid > j && tid < kb) D[tid][j] *= rl;
    __syncthreads();
    const int m = kb - j - 1;
    if (tid < 32) {
      if (m > 0) root(j + 1, fma(-D[j + 1][j], D[j + 1][j], D[j + 1][j + 1]));
    } else {
      const int half = (m + 1) >> 1;
      for (int e = tid - 32; e < half * (m + 1); e += 224) {
        const int c = e / (m + 1), r = e - c * (m + 1);
        const bool first = r < m - c;
        const int k = first ? c : m - 1 - c, i = first ? c + r : k + r - (m - c);
        if (i + k > 0 && (first || 2 * c != m - 1))  // (0, 0) belongs to the first warp
          D[j + 1 + i][j + 1 + k] = fma(-D[j + 1 + i][j], D[j + 1 + k][j], D[j + 1 + i][j + 1 + k]);
      }
    }
    __syncthreads();
  }
  for (int idx = tid; idx < kCholNb * kCholNb; idx += blockDim.x) {
    const int r = idx & 63, c = idx >> 6;
    if (r < kb && c < kb && r >= c) A[r + (size_t)c * lda] = D[r][c];
  }
}

// FP32: 16 columns at a time. Bound by the chain over the columns (root, scaling,
// update of the next column) and, column by column, by two barriers of the CTA for
// each. Here the 16 x 16 diagonal block is factored by one warp in registers with
// shuffles alone (lane: one row, every second column); four lanes per row then
// solve the rows below it; and all warps apply the rank-16 update. Every element
// receives the operations of the column-by-column elimination in its order.
// Measured per 64 x 64 block 41 -> 18 us. (In FP64, where one warp's chain is 64
// clocks per instruction, 63 us against the 61 of the kernel above.)
__global__ void __launch_bounds__(256)
    potf2_f32_kernel(int kb, float* __restrict__ A, int lda, int row0, int* __restrict__ info) {
  typedef float T;
  constexpr int PB = 16;
  __shared__ T D[kCholNb][kCholNb + 1];
  __shared__ T s_rl[PB];
  __shared__ int s_done;  // columns of the current 16 that were finished
  const int tid = threadIdx.x, lane = tid & 31;
  for (int idx = tid; idx < kCholNb * kCholNb; idx += blockDim.x) {
    const int r = idx & 63, c = idx >> 6;
    D[r][c] = (r < kb && c < kb && r >= c) ? A[r + (size_t)c * lda] : (T)0;
  }
  __syncthreads();
  for (int p0 = 0; p0 < kb; p0 += PB) {
    const int pb = min(PB, kb - p0);
    if (tid < 32) {
      const int i = lane & 15, h = lane >> 4;
      T v[PB / 2];
#pragma unroll
      for (int t = 0; t < PB / 2; ++t) v[t] = D[p0 + i][p0 + 2 * t + h];
      int done = 0;
      bool go = true;
      T myrl = (T)0, cp = (T)0;
#pragma unroll
      for (int j = 0; j < PB; ++j) {
        if (go && j < pb) {
          const T d = __shfl_sync(0xffffffffu, v[j / 2], j + 16 * (j & 1));
          const T a = __shfl_sync(0xffffffffu, v[j / 2], i + 16 * (j & 1));
          T l, rl;
          sqrt_rcp(d, &l, &rl);
          // meanwhile what column j - 1 leaves for the columns after this pair
          if (j > 0) {
#pragma unroll
            for (int t = j / 2 + 1; t < PB / 2; ++t) v[t] = fma(-cp, __shfl_sync(0xffffffffu, cp, 2 * t + h), v[t]);
          }
          go = d > (T)0;
          if (go) {
            done = j + 1;
            cp = a * rl;  // l_ij
            if (i == j) myrl = rl;
            if (h == (j & 1)) v[j / 2] = i == j ? l : (i > j ? cp : v[j / 2]);
            // the next column now (and its neighbour in the register)
            const int t = (j + 1) / 2;
            if (j + 1 < PB) {
              const T lk = __shfl_sync(0xffffffffu, cp, 2 * t + h);
              if (2 * t + h > j) v[t] = fma(-cp, lk, v[t]);
            }
          } else if (lane == 0) {
            atomicCAS(info, 0, row0 + p0 + j + 1);
          }
        }
      }
#pragma unroll
      for (int t = 0; t < PB / 2; ++t)
        if (2 * t + h <= i) D[p0 + i][p0 + 2 * t + h] = v[t];
      if (h == 0) s_rl[i] = myrl;
      if (lane == 0) s_done = done;
    }
    __syncthreads();
    const int done = s_done;
    const int q0 = p0 + PB;
    {  // rows q0 .. kb - 1: four lanes each, lane g with the columns g + 4 t
      const int r = q0 + 8 * (tid >> 5) + (lane & 7), g = lane >> 3;
      if (q0 + 8 * (tid >> 5) < kb) {
        T x[PB / 4];
        const bool in = r < kb;
#pragma unroll
        for (int t = 0; t < PB / 4; ++t) x[t] = in ? D[r][p0 + g + 4 * t] : (T)0;
#pragma unroll
        for (int j = 0; j < PB; ++j) {
          if (j < done) {
            const T xj = __shfl_sync(0xffffffffu, x[j / 4], (lane & 7) + 8 * (j & 3)) * s_rl[j];
            if (g == (j & 3)) x[j / 4] = xj;
#pragma unroll
            for (int t = j / 4; t < PB / 4; ++t)
              if (g + 4 * t > j) x[t] = fma(-xj, D[p0 + g + 4 * t][p0 + j], x[t]);
          }
        }
#pragma unroll
        for (int t = 0; t < PB / 4; ++t)
          if (in) D[r][p0 + g + 4 * t] = x[t];
      }
    }
    __syncthreads();
    // rank-16 update of the lower triangle of rows and columns q0 .. kb - 1 (columns
    // c and m - 1 - c of it are m + 1 elements together)
    const int m = max(kb - q0, 0), half = (m + 1) >> 1;
    for (int e = tid; e < half * (m + 1); e += 256) {
      const int c = e / (m + 1), r = e - c * (m + 1);
      const bool first = r < m - c;
      const int k = first ? c : m - 1 - c, i = first ? c + r : k + r - (m - c);
      if (first || 2 * c != m - 1) {
        T s = D[q0 + i][q0 + k];
        if (done == PB) {
#pragma unroll
          for (int t = 0; t < PB; ++t) s = fma(-D[q0 + i][p0 + t], D[q0 + k][p0 + t], s);
        } else {
          for (int t = 0; t < done; ++t) s = fma(-D[q0 + i][p0 + t], D[q0 + k][p0 + t], s);
        }
        D[q0 + i][q0 + k] = s;
      }
    }
    __syncthreads();
    if (done < pb) break;
  }
  for (int idx = tid; idx < kCholNb * kCholNb; idx += blockDim.x) {
    const int r = idx & 63, c = idx >> 6;
    if (r < kb && c < kb && r >= c) A[r + (size_t)c * lda] = D[r][c];
  }
}

// X L11^t = B for the M rows of B (M x kb, ldb); L11 kb x kb lower (kb <= 64).
// Four lanes share a row, each with the columns g + 4 t of it in registers; per
// column one broadcast and the update of the columns to its right. Bound by the
// FP64 pipe (a warp's instruction takes 64 clocks) and, with few rows, by the
// chain over the columns; one thread per row would leave two thirds of the
// schedulers idle at m = 6000 and take four times as long per row.
constexpr int kCholRows = 32;  // rows per CTA of 128 threads

template <typename T>
__global__ void __launch_bounds__(128)
    chol_trsm_kernel(int M, int kb, const T* __restrict__ L, int lda, T* __restrict__ B, int ldb) {
  __shared__ T Ls[kCholNb][kCholNb + 1];
  __shared__ T rdiag[kCholNb];
  const int tid = threadIdx.x, lane = tid & 31;
  const int row0 = blockIdx.x * kCholRows;
  for (int idx = tid; idx < kCholNb * kCholNb; idx += 128) {
    const int r = idx & 63, c = idx >> 6;
    Ls[r][c] = (r < kb && c < kb && r >= c) ? L[r + (size_t)c * lda] : (r == c ? (T)1 : (T)0);
  }
  const int r = row0 + 8 * (tid >> 5) + (lane & 7), g = lane >> 3;
  T x[kCholNb / 4];
#pragma unroll
  for (int t = 0; t < kCholNb / 4; ++t) x[t] = (r < M && g + 4 * t < kb) ? B[r + (size_t)(g + 4 * t) * ldb] : (T)0;
  __syncthreads();
  if (tid < kCholNb) rdiag[tid] = (T)1 / Ls[tid][tid];
  __syncthreads();
  // What the first 32 columns give the others is summed on its own and subtracted
  // once: half as many roundings at the size of the elements.
  constexpr int kHalf = kCholNb / 8;
  T acc[kHalf] = {};
#pragma unroll
  for (int j = 0; j < kCholNb; ++j) {
    if (j == kCholNb / 2) {
#pragma unroll
      for (int t = 0; t < kHalf; ++t) x[kHalf + t] -= acc[t];
    }
    const T xj = __shfl_sync(0xffffffffu, x[j / 4], (lane & 7) + 8 * (j & 3)) * rdiag[j];
    if (g == (j & 3)) x[j / 4] = xj;
#pragma unroll
    for (int t = j / 4; t < kCholNb / 4; ++t) {
      const int k = g + 4 * t;
      if (j < kCholNb / 2 && t >= kHalf) acc[t - kHalf] = fma(xj, Ls[k][j], acc[t - kHalf]);
      else if (t > j / 4) x[t] = fma(-xj, Ls[k][j], x[t]);
      else if (k > j) x[t] = fma(-xj, Ls[k][j], x[t]);
    }
  }
#pragma unroll
  for (int t = 0; t < kCholNb / 4; ++t)
    if (r < M && g + 4 * t < kb) B[r + (size_t)(g + 4 * t) * ldb] = x[t];
}

// One outer block [o0, o0 + ob) in 64-column steps: diagonal block, the
// rows below it, and the update of the rest of the outer block's columns
// (lower part). Arithmetic in T.
template <typename T>
static cudaError_t chol_outer_block(int n, T* A, int lda, int o0, int ob, int* info, cudaStream_t s) {
  for (int k0 = o0; k0 < o0 + ob; k0 += kCholNb) {
    const int kb = o0 + ob - k0 < kCholNb ? o0 + ob - k0 : kCholNb;
    T* A11 = A + k0 + (size_t)k0 * lda;
    prof_begin(KK_PANEL, s);
    if constexpr (sizeof(T) == 8) potf2_f64_kernel<<<1, 256, 0, s>>>(kb, A11, lda, k0, info);
    else potf2_f32_kernel<<<1, 256, 0, s>>>(kb, A11, lda, k0, info);
    count_launch();
    prof_end(KK_PANEL, s);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int m = n - k0 - kb;
    if (m <= 0) break;
    T* A21 = A11 + kb;
    prof_begin(KK_TRSM, s);
    chol_trsm_kernel<T><<<(m + kCholRows - 1) / kCholRows, 128, 0, s>>>(m, kb, A11, lda, A21, lda);
    count_launch();
    prof_end(KK_TRSM, s);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // the rest of the outer block's columns (lower part): rows k0 + kb .. n,
    // columns k0 + kb .. o0 + ob
    const int nrest = o0 + ob - k0 - kb;
    if (nrest > 0) {
      prof_begin(KK_GEMM_SIMT, s);
      e = launch_gemm_simt<T>(m, nrest, kb, (T)-1, A21, lda, A21, lda, true, (T)1,
                              A21 + (size_t)kb * lda, lda, true, s);
      prof_end(KK_GEMM_SIMT, s);
      if (e != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

// Two-level blocking: outer blocks of nb columns (a multiple of 64, up to
// 256); inside one, 64-column steps; after the outer block, one rank-nb
// update of the trailing lower triangle, on the tensor cores when the caller
// gave scratch for the digits (gemm_f64.cu), by FP64 multiply-adds otherwise.
cudaError_t launch_chol(int n, double* A, int lda, int nb, int* info, const F64Digits& dig,
                        cudaStream_t s) {
  if (nb <= 0) nb = kCholNb;
  if (nb % kCholNb != 0 || nb > 256) return cudaErrorInvalidValue;
  for (int o0 = 0; o0 < n; o0 += nb) {
    const int ob = n - o0 < nb ? n - o0 : nb;
    cudaError_t e = chol_outer_block<double>(n, A, lda, o0, ob, info, s);
    if (e != cudaSuccess) return e;
    // the trailing lower triangle: rank-ob update with the outer block's L21
    const int mt = n - o0 - ob;
    if (mt > 0) {
      double* L21 = A + (o0 + ob) + (size_t)o0 * lda;
      if (dig.a) {
        prof_begin(KK_CONVERT, s);
        e = launch_f64_digits_rows(L21, lda, mt, ob, dig.a, dig.ea, s);
        prof_end(KK_CONVERT, s);
        if (e != cudaSuccess) return e;
        prof_begin(KK_GEMM_TC, s);
        e = launch_gemm_f64tc(mt, mt, ob, dig.a, dig.a, dig.ea, dig.ea, L21 + (size_t)ob * lda, lda, dig.list,
                              info, true, s);
        prof_end(KK_GEMM_TC, s);
        if (e != cudaSuccess) return e;
        prof_begin(KK_GEMM_SIMT, s);
        e = launch_gemm_f64_list(mt, mt, ob, L21, lda, L21, lda, true, L21 + (size_t)ob * lda, lda, true,
                                 dig.list, s);
        prof_end(KK_GEMM_SIMT, s);
        if (e != cudaSuccess) return e;
        continue;
      }
      prof_begin(KK_GEMM_SIMT, s);
      e = launch_gemm_simt<double>(mt, mt, ob, -1.0, L21, lda, L21, lda, true, 1.0,
                                   L21 + (size_t)ob * lda, lda, true, s);
      prof_end(KK_GEMM_SIMT, s);
      if (e != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

// F (n x n FP32, lower triangle) <- its Cholesky factor, the trailing update
// of each outer block in the precision `prec`: FP32 SIMT, or on the tensor
// cores (lower tiles only) from a K-major low-precision copy of L21 with one
// power-of-two scale per row, which serves both operands (split kinds: a
// second copy in the right operand's [hi | lo | hi] pattern). Afterwards the
// strict upper triangle holds L^t (a mirror of the strict lower one), so that
// the backward substitution with L^t reads an upper triangle.
cudaError_t launch_chol_mixed(int n, float* F, int ldf, int nb, int prec, void* Ak, void* Bk, int ldk,
                              int* eA, int* info, cudaStream_t s) {
  if (nb % kCholNb != 0 || nb <= 0 || nb > 256) return cudaErrorInvalidValue;
  const bool tensor = prec_is_tensor(prec);
  for (int o0 = 0; o0 < n; o0 += nb) {
    const int ob = n - o0 < nb ? n - o0 : nb;
    cudaError_t e = chol_outer_block<float>(n, F, ldf, o0, ob, info, s);
    if (e != cudaSuccess) return e;
    const int mt = n - o0 - ob;
    if (mt <= 0) continue;
    float* L21 = F + (o0 + ob) + (size_t)o0 * ldf;
    float* C = L21 + (size_t)ob * ldf;
    if (tensor) {
      prof_begin(KK_CONVERT, s);
      e = launch_convert_rows(L21, ldf, mt, ob, prec, Ak, ldk, eA, false, s);
      if (e == cudaSuccess && prec_is_split(prec))
        e = launch_convert_rows(L21, ldf, mt, ob, prec, Bk, ldk, eA, true, s);
      prof_end(KK_CONVERT, s);
      if (e != cudaSuccess) return e;
      prof_begin(KK_GEMM_TC, s);
      e = launch_gemm_tc(prec_mma_kind(prec), mt, mt, prec_kmult(prec) * ob, Ak, ldk,
                         prec_is_split(prec) ? Bk : Ak, ldk, eA, eA, C, ldf, info, true, s);
      prof_end(KK_GEMM_TC, s);
    } else {
      prof_begin(KK_GEMM_SIMT, s);
      e = launch_gemm_simt<float>(mt, mt, ob, -1.0f, L21, ldf, L21, ldf, true, 1.0f, C, ldf, true, s);
      prof_end(KK_GEMM_SIMT, s);
    }
    if (e != cudaSuccess) return e;
  }
  return launch_mirror_lower(n, F, ldf, s);
}

// Strict upper triangle <- transpose of the strict lower one (32 x 32 tiles
// through shared memory: coalesced on both sides).
__global__ void mirror_lower_kernel(int n, float* __restrict__ F, int ldf) {
  __shared__ float t[32][33];
  const int bi = blockIdx.x, bj = blockIdx.y;  // tile (bi, bj) of the lower triangle, bi >= bj
  if (bi < bj) return;
  const int i0 = bi * 32, j0 = bj * 32;
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int i = i0 + threadIdx.x, j = j0 + r;
    t[r][threadIdx.x] = (i < n && j < n && i > j) ? F[i + (size_t)j * ldf] : 0.0f;
  }
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    // element (j0 + threadIdx.x, i0 + r) of the upper triangle = (i0 + r, j0 + threadIdx.x) of the lower
    const int i = i0 + r, j = j0 + threadIdx.x;
    if (i < n && j < n && i > j) F[j + (size_t)i * ldf] = t[threadIdx.x][r];
  }
}

cudaError_t launch_mirror_lower(int n, float* F, int ldf, cudaStream_t s) {
  if (n <= 1) return cudaSuccess;
  const int T = (n + 31) / 32;
  mirror_lower_kernel<<<dim3(T, T), dim3(32, 8), 0, s>>>(n, F, ldf);
  count_launch();
  return cudaGetLastError();
}

}  // namespace gbla
