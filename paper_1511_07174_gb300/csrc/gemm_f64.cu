// FP64 trailing update C -= A B (paper section 2: the rank-k "delayed update")
// on the 5th-generation tensor cores, as products of 8-bit digits
// (the error-free splitting of Ozaki, Ogita, Oishi and Rump, 2012, with
// integer-aligned slices).
//
// This GPU's FP64 pipe does 2 multiply-adds per clock and SM, so a rank-256
// update on it runs at 1.06 TFLOP/s whatever the kernel; its BF16 tensor rate
// is 1800 times that. Every row of A and column of B is scaled by a power of
// two so that its largest magnitude lies in [64, 128) and written in fixed
// point with 48 fractional bits,
//     x = d_0 + d_1 2^-8 + ... + d_6 2^-48,   -128 <= d_t <= 128 integers,
// each d_t 2^-8t a BF16 number. A digit product is at most 2^14 and the sum of
// K <= 256 of them at most 2^22, so the FP32 accumulator of the tensor cores
// holds the sum of up to four digit pairs exactly, and of five or six unless every
// digit is near 128. The pairs with s + t <= 7 (34 of 49) are multiplied, those with
// the same s + t = g into one accumulator. 6 and 7 share one, whose sums (13 pairs in
// units of 2^-56) need some 26 bits: it rounds, at 2^-55 for typical digits and at
// 2^-48 with every digit near 128. The epilogue rounds the accumulators to 2^-40,
// adds them in 64-bit fixed point, rounds once to FP64 and subtracts from C with one
// FP64 operation per element; what the 15 pairs left out would add is below that
// 2^-40 (typically 2^-46).
//
// Accuracy. With A_i, B_j scaled as above and P = sum_k |a_ik| |b_kj|, the
// representation (2^-49 per element, zero for elements within a factor 4 of
// their row's largest) and the 40 fractional bits of the accumulation leave
// an error of about 2^-41 for K = 256; the chain of 256 rounded FP64
// multiply-adds leaves about 0.4 P 2^-53. For dense rows and columns
// P > 2^16 and the digits are several times more accurate; when P is small
// (rows and columns whose large elements do not meet: graded or sparse
// operands) they could be less so. One more product, of |d_0| with |d_0|,
// gives P; a tile with an element below 1024 sqrt(K), or with a row or column
// that holds an infinity, a NaN or a magnitude outside 2^+-450, is left
// untouched and listed, and the listed tiles are updated by FP64 multiply-adds.
//
// Kernel: persistent, one CTA per SM, 128 x 128 tiles, warp-specialised like
// the mixed-precision update. One tile takes two passes over K, 32 at a time:
//   pass L: digits 0..6 of both operands (14 slices of 128 x 32, 112 KB a
//           stage, two stages), groups 3, 4, 5 and 6+7 in the four 128-column
//           accumulators (28 pairs);
//   pass H: |d_0| and digits 0..2 (8 slices), P and groups 0, 1, 2 (7 pairs).
// A slice is used by up to seven pairs while it is in shared memory, which is
// what keeps the loads (1.4 MB per tile) below the L2 rate; two passes because
// eight accumulators of 128 columns would be twice the tensor memory. L comes
// first so that the FP64 update of C of one tile runs while the long pass of
// the next is multiplied.
//
// Measured (whole factorisation, GB300): LU n = 8192, nb = 256: trailing updates
// 286 -> 11.9 ms, factor + 16 right-hand sides 361 -> 88 ms; n = 3001 34.9 ->
// 21.5 ms; Cholesky n = 6000, nb = 128: 69 -> 4.6 ms of updates.
#include <cuda_bf16.h>
#include <math.h>
#include <string.h>

#include "common.cuh"
#include "internal.h"
#include "tcgen05.cuh"

namespace gbla {

constexpr int kF6Tile = 128;
constexpr int kF6BK = 32;                          // k per stage
constexpr int kF6Slices = 8;                       // |d_0|, d_0 .. d_6
constexpr int kF6SliceBytes = kF6Tile * kF6BK * 2; // 128 rows of 64 bytes
constexpr int kF6StageSlices = 14;
constexpr int kF6Stages = 2;
constexpr int kF6StageBytes = kF6StageSlices * kF6SliceBytes;
// Warp 0 TMA, warp 1 MMA, warps 4-11 epilogue (64 64-bit sums per thread): the first
// warpgroup gives registers to the other two (56 + 2 x 224 = 3 x 168, what the
// block is launched with).
constexpr int kF6Threads = 384;
constexpr int kF6RegsIo = 56, kF6RegsEpi = 224;
constexpr int kF6Smem = kF6Stages * kF6StageBytes + 1024 + 256;
constexpr int kF6RowZero = 1 << 20, kF6RowBad = 1 << 21, kF6ExpBias = 4096;

size_t f64tc_ld(int K) { return (size_t)((K + kF6BK - 1) / kF6BK) * kF6BK * kF6Slices; }
size_t f64tc_list_ints(int M, int N) {
  return (size_t)((M + kF6Tile - 1) / kF6Tile) * ((N + kF6Tile - 1) / kF6Tile) + 1;
}

// ---- digits --------------------------------------------------------------------
// Scale word of a row with largest magnitude bits `mx` (as an integer): the
// exponent e with max 2^e in [64, 128), biased, plus the flags.
GBLA_DEVINL int f6_scale(unsigned long long mx) {
  const int ex = (int)(mx >> 52);
  if (mx == 0) return kF6RowZero + kF6ExpBias;
  if (ex < 1023 - 450 || ex > 1023 + 450) return kF6RowBad + kF6ExpBias;
  return 6 - (ex - 1023) + kF6ExpBias;
}

// Four consecutive elements of a row -> their digits in the eight slices
// (out: the element's place in slice 0 of its 32-block; a slice is 32 elements).
GBLA_DEVINL void f6_store_digits(const double (&v)[4], int scale, __nv_bfloat16* out) {
  const int e = (scale & 0xffff) - kF6ExpBias;
  const bool ok = (scale >> 16) == 0;
  long long Y[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v[i]);
    int ex = (int)((b >> 52) & 0x7ff);
    unsigned long long m = b & 0xfffffffffffffull;
    if (ex) m |= 1ull << 52;
    else ex = 1;
    const int sh = ex - 1075 + e + 48;  // at most 2
    unsigned long long x = 0;
    if (sh >= 0) x = m << sh;
    else if (sh > -55) x = (m + (1ull << (-sh - 1))) >> -sh;
    if (!ok) x = 0;
    const long long X = (b >> 63) ? -(long long)x : (long long)x;
    Y[i] = X + 0x0000808080808080ll;  // every byte below the top digit biased by 128
  }
#pragma unroll
  for (int t = -1; t < 7; ++t) {
    uint32_t h[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      int d;
      if (t <= 0) d = (int)(Y[i] >> 48);
      else d = (int)((unsigned)(Y[i] >> (48 - 8 * t)) & 255u) - 128;
      if (t < 0) d = d < 0 ? -d : d;
      // exact: |d| <= 128 has at most 8 significant bits
      const float f = (float)d * __int_as_float((127 - 8 * (t < 0 ? 0 : t)) << 23);
      h[i] = __float_as_uint(f) >> 16;
    }
    *reinterpret_cast<uint2*>(out + (t + 1) * kF6BK) =
        make_uint2(h[0] | (h[1] << 16), h[2] | (h[3] << 16));
  }
}

// Rows of a column-major M x K matrix (K <= 256): one CTA per 32 rows, staged
// in shared memory once (the row maximum is needed before the first digit).
// Bound by HBM: 8 bytes read and 16 written per element.
__global__ void __launch_bounds__(256)
    f64_digits_rows_kernel(const double* __restrict__ F, int ldf, int M, int K, int Kp,
                           __nv_bfloat16* __restrict__ out, int* __restrict__ scale) {
  extern __shared__ double f6_tile[];  // [Kp][33]
  __shared__ unsigned long long wmax[8][32];
  __shared__ int sc[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int m0 = blockIdx.x * 32, m = m0 + lane;
  unsigned long long mx = 0;
#pragma unroll 8
  for (int k = warp; k < Kp; k += 8) {
    const double v = (m < M && k < K) ? F[m + (size_t)k * ldf] : 0.0;
    f6_tile[k * 33 + lane] = v;
    const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
    mx = b > mx ? b : mx;
  }
  wmax[warp][lane] = mx;
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int q = 1; q < 8; ++q) mx = wmax[q][lane] > mx ? wmax[q][lane] : mx;
    sc[lane] = f6_scale(mx);
    if (m < M) scale[m] = sc[lane];
  }
  __syncthreads();
  const size_t ld = (size_t)Kp * kF6Slices;
  for (int it = threadIdx.x; it < 32 * (Kp / 4); it += 256) {
    const int q = it & 7, r = (it >> 3) & 31, kb = it >> 8;
    if (m0 + r >= M) continue;
    double v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = f6_tile[(kb * kF6BK + q * 4 + i) * 33 + r];
    f6_store_digits(v, sc[r], out + (size_t)(m0 + r) * ld + (size_t)kb * kF6BK * kF6Slices + q * 4);
  }
}

// Columns of a column-major K x N matrix (K <= 256): one warp per column.
__global__ void __launch_bounds__(256)
    f64_digits_cols_kernel(const double* __restrict__ B, int ldb, int N, int K, int Kp,
                           __nv_bfloat16* __restrict__ out, int* __restrict__ scale) {
  const int lane = threadIdx.x & 31;
  const int n = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (n >= N) return;
  const double* b = B + (size_t)n * ldb;
  double v[2][4];
  unsigned long long mx = 0;
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = 4 * (lane + 32 * h) + i;
      v[h][i] = k < K ? b[k] : 0.0;
      const unsigned long long u = (unsigned long long)__double_as_longlong(v[h][i]) & 0x7fffffffffffffffull;
      mx = u > mx ? u : mx;
    }
  mx = warp_max(mx);
  const int sc = f6_scale(mx);
  if (lane == 0) scale[n] = sc;
  const size_t ld = (size_t)Kp * kF6Slices;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int k = 4 * (lane + 32 * h);
    if (k < Kp)
      f6_store_digits(v[h], sc, out + (size_t)n * ld + (size_t)(k / kF6BK) * kF6BK * kF6Slices + k % kF6BK);
  }
}

cudaError_t launch_f64_digits_rows(const double* F, int ldf, int M, int K, void* out, int* scale,
                                   cudaStream_t s) {
  if (M <= 0 || K <= 0) return cudaSuccess;
  if (K > 256) return cudaErrorInvalidValue;
  const int Kp = (K + kF6BK - 1) / kF6BK * kF6BK;
  const size_t smem = (size_t)Kp * 33 * sizeof(double);
  cudaError_t e = ensure_dyn_smem(f64_digits_rows_kernel, smem);
  if (e != cudaSuccess) return e;
  f64_digits_rows_kernel<<<(M + 31) / 32, 256, smem, s>>>(F, ldf, M, K, Kp,
                                                          static_cast<__nv_bfloat16*>(out), scale);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_f64_digits_cols(const double* B, int ldb, int N, int K, void* out, int* scale,
                                   cudaStream_t s) {
  if (N <= 0 || K <= 0) return cudaSuccess;
  if (K > 256) return cudaErrorInvalidValue;
  const int Kp = (K + kF6BK - 1) / kF6BK * kF6BK;
  f64_digits_cols_kernel<<<(N + 7) / 8, 256, 0, s>>>(B, ldb, N, K, Kp, static_cast<__nv_bfloat16*>(out),
                                                     scale);
  count_launch();
  return cudaGetLastError();
}

// ---- the update ------------------------------------------------------------------
struct F6Args {
  int M, N, KBn;  // KBn: 32-wide steps over K
  int tilesM, ntiles, lower;
  double* C;
  int ldc;
  const int* eA;
  const int* eB;
  int* list;  // [0] count, then the tiles left to the FP64 pipe
  float pmin;
  int* info;
  uint64_t wait_ns;
};

// a 2^e as a double, rounded to nearest (ties away), for a 64-bit integer a and
// e such that the result is a normal number.
GBLA_DEVINL double f6_fixed_to_double(long long a, int e) {
  const unsigned long long u = a < 0 ? (unsigned long long)(-a) : (unsigned long long)a;
  if (u == 0) return 0.0;
  int lz = __clzll((long long)u);
  const unsigned long long n = u << lz;
  unsigned long long r = n + 0x400ull;
  if (r < n) {  // rounded up to a power of two
    r = 1ull << 63;
    --lz;
  }
  const unsigned long long ex = (unsigned long long)(1023 + 63 - lz + e);
  unsigned long long bits = (ex << 52) | ((r >> 11) & 0xfffffffffffffull);
  if (a < 0) bits |= 1ull << 63;
  return __longlong_as_double((long long)bits);
}

// 16 columns of one accumulator: acc += round(D 2^MUL) 2^SH
template <int MUL, int SH, bool FIRST>
GBLA_DEVINL void f6_add16(uint32_t taddr, long long* acc) {
  uint32_t v[16];
  tmem_ld16(taddr, v);
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const int d = __float2int_rn(__uint_as_float(v[j]) * __int_as_float((127 + MUL) << 23));
    const long long x = (long long)d << SH;
    acc[j] = FIRST ? x : acc[j] + x;
  }
}

__global__ void __launch_bounds__(kF6Threads, 1)
    gemm_f64tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                      F6Args args) {
  extern __shared__ unsigned char smraw[];
  const uint32_t raw = smem_u32(smraw);
  const uint32_t sbase = (raw + 1023u) & ~1023u;
  unsigned char* sm = smraw + (sbase - raw);
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm + kF6Stages * kF6StageBytes);
  const uint32_t bar_full = smem_u32(bars);        // [2] TMA -> MMA
  const uint32_t bar_empty = bar_full + 16;        // [2] MMA -> TMA
  const uint32_t bar_tfull = bar_full + 32;        // accumulators of a pass complete
  const uint32_t bar_tempty = bar_full + 40;       // [4] accumulator drained
  const uint32_t bar_flag = bar_full + 72;         // every epilogue warp has its verdict in s_bad
  const uint32_t bar_drain = bar_full + 80;        // the MMA issuer's last commit
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bars + 11);
  volatile int* s_fail = reinterpret_cast<volatile int*>(tmem_holder + 1);
  volatile int* s_issued = s_fail + 1;
  volatile int* s_bad = s_fail + 2;  // [2], by tile parity

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar_full + 8 * i, 1);
      mbar_init(bar_empty + 8 * i, 1);
    }
    mbar_init(bar_tfull, 1);
    for (int i = 0; i < 4; ++i) mbar_init(bar_tempty + 8 * i, 8);
    mbar_init(bar_flag, 8);
    mbar_init(bar_drain, 1);
    *s_fail = 0;
    *s_issued = 0;
    s_bad[0] = s_bad[1] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_holder)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_holder;
  constexpr uint32_t kIdesc = make_idesc(1u, kF6Tile, kF6Tile);  // BF16 operands, FP32 accumulator

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kF6RegsIo));
    if (warp == 0) {
      if (lane == 0) {  // TMA producer: stage = slices of A, then of B
        int it = 0;
        bool ok = true;
        for (int t = blockIdx.x; t < args.ntiles && ok; t += gridDim.x) {
          int ti, tj;
          tile_coords(t, args.tilesM, args.lower, ti, tj);
          for (int pass = 0; pass < 2 && ok; ++pass) {
            const int first = pass == 0 ? 1 : 0, ns = pass == 0 ? 7 : 4;
            for (int kb = 0; kb < args.KBn; ++kb, ++it) {
              const int st = it & 1;
              if (*s_fail || !mbar_wait_bounded(bar_empty + 8 * st, ((uint32_t)(it >> 1) & 1u) ^ 1u, args.wait_ns)) {
                *s_fail = 1;
                ok = false;
                break;
              }
              const uint32_t bar = bar_full + 8 * st;
              const uint32_t dst = sbase + st * kF6StageBytes;
              mbar_expect_tx(bar, (uint32_t)(2 * ns * kF6SliceBytes));
              for (int q = 0; q < ns; ++q) {
                const int x = (kb * kF6Slices + first + q) * kF6BK;
                tma_load_2d(dst + q * kF6SliceBytes, &tmA, x, ti * kF6Tile, bar);
                tma_load_2d(dst + (7 + q) * kF6SliceBytes, &tmB, x, tj * kF6Tile, bar);
              }
            }
          }
        }
        *s_issued = it;
      }
    } else if (warp == 1) {
      if (lane == 0) {  // MMA issuer
        int it = 0, pc = 0;
        bool ok = true;
        // one digit pair over the 32 k of a stage: two MMAs
        auto pair = [&](uint32_t stage, int buf, int sa, int sb, bool first) {
#pragma unroll
          for (int kk = 0; kk < 2; ++kk)
            mma_issue<GBLA_PREC_BF16>(tmem + (uint32_t)(buf * kF6Tile),
                                      make_sdesc<64>(stage + sa * kF6SliceBytes + kk * 32),
                                      make_sdesc<64>(stage + (7 + sb) * kF6SliceBytes + kk * 32), kIdesc,
                                      (first && kk == 0) ? 0u : 1u);
        };
        for (int t = blockIdx.x; t < args.ntiles && ok; t += gridDim.x) {
          for (int pass = 0; pass < 2 && ok; ++pass, ++pc) {
            for (int kb = 0; kb < args.KBn && ok; ++kb, ++it) {
              const int st = it & 1;
              if (*s_fail || !mbar_wait_bounded(bar_full + 8 * st, (uint32_t)(it >> 1) & 1u, args.wait_ns)) {
                *s_fail = 1;
                ok = false;
                break;
              }
              asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
              const uint32_t stage = sbase + st * kF6StageBytes;
              for (int b = 0; b < 4; ++b) {
                if (kb == 0) {
                  // the epilogue has read what this accumulator held
                  if (!mbar_wait_bounded(bar_tempty + 8 * b, ((uint32_t)pc & 1u) ^ 1u, args.wait_ns)) {
                    *s_fail = 1;
                    ok = false;
                    break;
                  }
                  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                }
                bool first = kb == 0;
                if (pass == 0) {
                  // slots 0..6 = digits 0..6; accumulators: s + t = 3, 4, 5, 6 and 7
                  const int g_hi = b < 3 ? 3 + b : 7;
                  for (int g = 3 + b; g <= g_hi; ++g)
                    for (int sa = g > 6 ? g - 6 : 0; sa <= (g < 6 ? g : 6); ++sa) {
                      pair(stage, b, sa, g - sa, first);
                      first = false;
                    }
                } else if (b == 0) {
                  pair(stage, 0, 0, 0, first);  // slot 0 = |d_0|
                } else {
                  // slots 1..3 = digits 0..2; accumulators: s + t = 0, 1, 2
                  for (int sa = 0; sa <= b - 1; ++sa) {
                    pair(stage, b, 1 + sa, 1 + (b - 1 - sa), first);
                    first = false;
                  }
                }
              }
              mma_commit(bar_empty + 8 * st);
            }
            if (ok) mma_commit(bar_tfull);
          }
        }
        // every MMA this thread issued has finished before tensor memory is freed
        mma_commit(bar_drain);
        const uint64_t dns = args.wait_ns > kPsDrainFloorNs ? args.wait_ns : kPsDrainFloorNs;
        if (!mbar_wait_bounded(bar_drain, 0u, dns)) *s_fail = 1;
      }
    }
  } else {  // epilogue warps: TMEM lane group warp % 4, column half (warp - 4) / 4
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kF6RegsEpi));
    const int eg = warp & 3;
    const int c_lo = ((warp - 4) >> 2) * (kF6Tile / 2);
    int i = 0;
    for (int t = blockIdx.x; t < args.ntiles; t += gridDim.x, ++i) {
      int ti, tj;
      tile_coords(t, args.tilesM, args.lower, ti, tj);
      const int row = ti * kF6Tile + eg * 32 + lane;
      const int col0 = tj * kF6Tile + c_lo;
      const bool rok = row < args.M;
      const int ra = rok ? args.eA[row] : 0;
      // this lane's two column scales, and the columns that hold zeros only or
      // cannot be represented
      int cb2[2];
      unsigned czero[2], cbad[2], cval[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int col = col0 + 32 * h + lane;
        const bool cok = col < args.N;
        cb2[h] = cok ? args.eB[col] : 0;
        cval[h] = __ballot_sync(0xffffffffu, cok);
        czero[h] = __ballot_sync(0xffffffffu, (cb2[h] & kF6RowZero) != 0);
        cbad[h] = __ballot_sync(0xffffffffu, (cb2[h] & kF6RowBad) != 0);
        if (args.lower) {  // columns above the diagonal are not written
          const int nlow = row - (col0 + 32 * h) + 1;  // columns <= row
          cval[h] &= nlow >= 32 ? 0xffffffffu : (nlow <= 0 ? 0u : (1u << nlow) - 1u);
        }
      }
      const bool rzero = (ra & kF6RowZero) != 0;
      int bad = 0;  // this row of the tile must go to the FP64 pipe
      if (rok) bad = ((ra & kF6RowBad) && (cval[0] | cval[1])) || (cbad[0] & cval[0]) || (cbad[1] & cval[1]);

      long long acc[64];
      bool stop = false;
#pragma unroll 1
      for (int pass = 0; pass < 2; ++pass) {
        int fail = 0;
        if (lane == 0)
          fail = (!mbar_wait_bounded(bar_tfull, (uint32_t)pass, args.wait_ns)) || *s_fail;
        fail = __shfl_sync(0xffffffffu, fail, 0);
        if (fail) {
          *s_fail = 1;
          stop = true;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t tb = tmem + ((uint32_t)(eg * 32) << 16) + (uint32_t)c_lo;
        auto drained = [&](int b) {
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_tempty + 8 * b);
        };
        if (pass == 0) {
#pragma unroll
          for (int q = 0; q < 4; ++q) f6_add16<24, 16, true>(tb + 16 * q, acc + 16 * q);
          drained(0);
#pragma unroll
          for (int q = 0; q < 4; ++q) f6_add16<32, 8, false>(tb + kF6Tile + 16 * q, acc + 16 * q);
          drained(1);
#pragma unroll
          for (int q = 0; q < 4; ++q) f6_add16<40, 0, false>(tb + 2 * kF6Tile + 16 * q, acc + 16 * q);
          drained(2);
#pragma unroll
          for (int q = 0; q < 4; ++q) f6_add16<40, 0, false>(tb + 3 * kF6Tile + 16 * q, acc + 16 * q);
          drained(3);
        } else {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            uint32_t v[16];
            tmem_ld16(tb + 16 * q, v);
            unsigned low = 0;
#pragma unroll
            for (int j = 0; j < 16; ++j) low |= (__uint_as_float(v[j]) < args.pmin ? 1u : 0u) << j;
            const unsigned need = ((cval[q >> 1] & ~czero[q >> 1]) >> (16 * (q & 1))) & 0xffffu;
            if (rok && !rzero && (low & need)) bad = 1;
          }
          drained(0);
#pragma unroll
          for (int q = 0; q < 4; ++q) f6_add16<0, 40, false>(tb + kF6Tile + 16 * q, acc + 16 * q);
          drained(1);
#pragma unroll
          for (int q = 0; q < 4; ++q) f6_add16<8, 32, false>(tb + 2 * kF6Tile + 16 * q, acc + 16 * q);
          drained(2);
#pragma unroll
          for (int q = 0; q < 4; ++q) f6_add16<16, 24, false>(tb + 3 * kF6Tile + 16 * q, acc + 16 * q);
          drained(3);
        }
      }
      if (stop) break;
      // one verdict for the tile
      bad = __any_sync(0xffffffffu, bad);
      if (lane == 0) {
        if (bad) s_bad[i & 1] = 1;
        mbar_arrive(bar_flag);
        bad = 2 * (int)!mbar_wait_bounded(bar_flag, (uint32_t)(i & 1), args.wait_ns);
        bad |= s_bad[i & 1];
      }
      bad = __shfl_sync(0xffffffffu, bad, 0);
      if (bad & 2) {
        *s_fail = 1;
        break;
      }
      if (warp == 4 && lane == 0) {
        s_bad[(i + 1) & 1] = 0;  // last read before this tile's verdict, written after the next one's passes
        if (bad) args.list[1 + atomicAdd(args.list, 1)] = t;
      }
      if (rok && !bad) {
        double* crow = args.C + row + (size_t)col0 * args.ldc;
        const int ea = (ra & 0xffff) - kF6ExpBias;
#pragma unroll
        for (int q = 0; q < 64; q += 8) {
          double cv[8];
          int eb[8];
          const unsigned ok8 = cval[q >> 5] >> (q & 31);
          asm volatile("" ::: "memory");  // one chunk of loads at a time: the sums hold the registers
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            cv[j] = (ok8 >> j) & 1u ? crow[(size_t)(q + j) * args.ldc] : 0.0;
            eb[j] = (ok8 >> j) & 1u ? __ldg(args.eB + col0 + q + j) : 0;
          }
#pragma unroll
          for (int j = 0; j < 8; ++j)
            if ((ok8 >> j) & 1u)
              crow[(size_t)(q + j) * args.ldc] =
                  cv[j] + f6_fixed_to_double(-acc[q + j], -40 - ea - ((eb[j] & 0xffff) - kF6ExpBias));
        }
      }
      __syncwarp();
    }
  }
  __syncthreads();
  if (*s_fail) {
    if (threadIdx.x == 0) {
      gbla_flag_timeout(args.info);
      const int issued = *s_issued;
      const uint64_t dns = args.wait_ns > kPsDrainFloorNs ? args.wait_ns : kPsDrainFloorNs;
      for (int it = (issued > kF6Stages ? issued - kF6Stages : 0); it < issued; ++it)
        mbar_wait_bounded(bar_full + 8 * (it & 1), (uint32_t)((it >> 1) & 1), dns);
    }
    __syncthreads();
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
  }
}

static bool f6_encode(CUtensorMap* map, const void* ptr, int Kp, int rows) {
  EncodeTiledFn enc = get_encode();
  if (!enc) return false;
  const cuuint64_t width = (cuuint64_t)Kp * kF6Slices;
  cuuint64_t gdim[2] = {width, (cuuint64_t)rows};
  cuuint64_t gstride[1] = {width * 2};
  cuuint32_t box[2] = {(cuuint32_t)kF6BK, (cuuint32_t)kF6Tile};
  cuuint32_t estr[2] = {1u, 1u};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), gdim, gstride, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

cudaError_t launch_gemm_f64tc(int M, int N, int K, const void* Ad, const void* Bd, const int* eA,
                              const int* eB, double* C, int ldc, int* list, int* info, bool lower,
                              cudaStream_t s, int grid_cap) {
  if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
  if (K > 256 || (lower && M != N)) return cudaErrorInvalidValue;
  if ((reinterpret_cast<uintptr_t>(Ad) & 15) || (reinterpret_cast<uintptr_t>(Bd) & 15))
    return cudaErrorInvalidValue;
  const int KBn = (K + kF6BK - 1) / kF6BK;
  CUtensorMap ta, tb;
  if (!f6_encode(&ta, Ad, KBn * kF6BK, M) || !f6_encode(&tb, Bd, KBn * kF6BK, N)) return cudaErrorInvalidValue;
  const int tilesM = (M + kF6Tile - 1) / kF6Tile, tilesN = (N + kF6Tile - 1) / kF6Tile;
  const int ntiles = lower ? tilesM * (tilesM + 1) / 2 : tilesM * tilesN;
  cudaError_t e = cudaMemsetAsync(list, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  F6Args a{M,  N,  KBn, tilesM, ntiles, lower ? 1 : 0, C, ldc, eA, eB, list, 1024.0f * sqrtf((float)K),
           info, wait_timeout_ns()};
  const DeviceProps& dp = device_props();
  int grid = dp.num_sms > 0 ? dp.num_sms : 1;
  if (grid_cap > 0 && grid > grid_cap) grid = grid_cap;
  if (grid > ntiles) grid = ntiles;
  e = ensure_dyn_smem(gemm_f64tc_kernel, (size_t)kF6Smem);
  if (e != cudaSuccess) return e;
  gemm_f64tc_kernel<<<grid, kF6Threads, kF6Smem, s>>>(ta, tb, a);
  count_launch();
  return cudaGetLastError();
}

}  // namespace gbla
