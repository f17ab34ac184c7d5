// Shared device helpers for the gbla kernels (sm_103a).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/gbla.h"

#define GBLA_DEVINL __device__ __forceinline__

// Nanosecond wall clock of the GPU; used to bound every inter-CTA wait.
GBLA_DEVINL uint64_t gbla_now_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

GBLA_DEVINL unsigned ld_acquire_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

GBLA_DEVINL void st_release_u32(unsigned* p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

GBLA_DEVINL int ld_acquire_s32(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Record the first device-side failure in the caller's info word: the
// timeout code only replaces a zero (a numerical info already set stays).
GBLA_DEVINL void gbla_flag_timeout(int* info) {
  if (info) atomicCAS(info, 0, GBLA_INFO_TIMEOUT);
}

// Spin until *p >= target or the wait exceeds limit_ns. Returns true on
// success. One thread per CTA calls it.
GBLA_DEVINL bool gbla_wait_geq(const unsigned* p, unsigned target, uint64_t limit_ns) {
  if (ld_acquire_u32(p) >= target) return true;
  uint64_t t0 = gbla_now_ns();
  while (true) {
    if (ld_acquire_u32(p) >= target) return true;
    if (gbla_now_ns() - t0 > limit_ns) return false;
    __nanosleep(32);
  }
}

// FP32 -> FP64 with integer instructions: the conversion instruction occupies the
// FP64 pipe like a multiply-add does (64 clocks a warp). Zeros, subnormals,
// infinities and NaN take it.
GBLA_DEVINL double to_f64(float f) {
  const unsigned b = __float_as_uint(f);
  if ((((b >> 23) + 1u) & 0xffu) <= 1u) return (double)f;
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20))), (int)(b << 29));
}
GBLA_DEVINL double to_f64(double f) { return f; }

template <typename T>
GBLA_DEVINL T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <typename T>
GBLA_DEVINL T warp_max(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    T u = __shfl_xor_sync(0xffffffffu, v, o);
    v = u > v ? u : v;
  }
  return v;
}

// (|value|, index) argmax: larger magnitude wins, ties go to the lower index.
GBLA_DEVINL void argmax_merge(double& bv, int& bi, double v, int i) {
  if (v > bv || (v == bv && i < bi)) {
    bv = v;
    bi = i;
  }
}

GBLA_DEVINL void warp_argmax(double& bv, int& bi) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    double v = __shfl_xor_sync(0xffffffffu, bv, o);
    int i = __shfl_xor_sync(0xffffffffu, bi, o);
    argmax_merge(bv, bi, v, i);
  }
}

// Output tile t -> (row tile, column tile): column-major over the tile grid,
// or, for the lower triangle of tiles, row by row over (i, j), j <= i.
GBLA_DEVINL void tile_coords(int t, int tilesM, int lower, int& ti, int& tj) {
  if (!lower) {
    ti = t % tilesM;
    tj = t / tilesM;
    return;
  }
  int i = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  while ((long long)(i + 1) * (i + 2) / 2 <= t) ++i;
  while ((long long)i * (i + 1) / 2 > t) --i;
  ti = i;
  tj = t - i * (i + 1) / 2;
}

// *l = sqrt(d), *rl = 1 / *l for d > 0.
GBLA_DEVINL void sqrt_rcp(float d, float* l, float* rl) {
  *l = sqrtf(d);
  *rl = 1.0f / *l;
}
// Subnormal or infinite d, out of line: unrolled 16 times in a panel, the square root
// and the division were half of its instructions (2000 Cholesky systems of n = 8, one
// CTA per SM, with the test of a column's rows inside the loop: 281 -> 234 us).
static __device__ __noinline__ double2 sqrt_rcp_rare(double d) {
  const double l = sqrt(d);
  return make_double2(l, 1.0 / l);
}
// FP64: sqrt followed by a division is a chain of some twenty dependent FP64
// operations per column, at the latency this GPU's FP64 pipe has. Instead, d is
// scaled by a power of four to x in [1/2, 2); with the FP32 approximation y of
// 1 / sqrt(x) and e = 1 - x y^2, |e| < 2^-20, one third-order step of the series
//   (1 - e)^-1/2 = 1 + e/2 + 3/8 e^2 + O(e^3)
// takes y to 1 / sqrt(x) and x y to sqrt(x), side by side, the neglected term below
// 2^-61. The root is then corrected by its residual, and the reciprocal by its
// product with the root as rounded: it is the reciprocal of that root, not of
// sqrt(d), so that a column scaled with it leaves the residual that one divided by
// the root leaves (with 1 / sqrt(d) rounded on its own 1.03 to 1.09 times that, rms,
// orders 16 to 64). Its two operations cost the Cholesky of n = 6000 16.2 -> 16.7 ms.
GBLA_DEVINL void sqrt_rcp(double d, double* l, double* rl) {
  const int hi = __double2hiint(d);
  const int ex = hi >> 20;  // d > 0: no sign
  if (ex == 0 || ex >= 0x7ff) {
    const double2 v = sqrt_rcp_rare(d);
    *l = v.x;
    *rl = v.y;
    return;
  }
  const int q = (ex - 1022) >> 1;  // d = x 4^q, exponent of x: 1022 or 1023
  const double x = __hiloint2double(hi - (q << 21), __double2loint(d));
  const double y = (double)rsqrtf((float)x);
  const double g = x * y;
  const double e = fma(-g, y, 1.0);
  const double p = fma(0.375, e, 0.5);
  const double r = fma(y * e, p, y);
  const double h = fma(g * e, p, g);
  const double s = fma(fma(-h, h, x), 0.5 * r, h);
  const double t = fma(r, fma(-s, r, 1.0), r);
  *rl = __hiloint2double(__double2hiint(t) - (q << 20), __double2loint(t));
  *l = __hiloint2double(__double2hiint(s) + (q << 20), __double2loint(s));
}

// Final sources of the rows touched by kb <= 256 sequential interchanges
// (row t <-> row p_t for t = 0 .. kb - 1 in order, p_t >= t, rows relative to
// the block's first row), worked out by the threads t < kb in parallel. With
// pre(t) the value row t holds just before interchange t:
//   pre(t) = pre(i) for the last i < t with p_i = t, else row t's own value;
//   row t ends with pre(t) if p_t = t, else with what row p_t held just
//   before interchange t: pre(i) for the last i < t with p_i = p_t, else p_t's
//   own value;
//   a partner row x >= kb ends with pre(i) for the last interchange i naming it.
// pre follows the chains t -> i (i < t) to a row that kept its own value,
// found by pointer jumping (8 rounds cover chains of 256). Every thread of the
// CTA must call it (it contains barriers); s.p must already hold the p_t.
struct SwapPlanShared {
  int p[256];
  int J[2][256];
};

// Thread t < kb: *src_b = the row whose original value ends in row t; when t
// is the last interchange naming a partner row p_t >= kb, *dst_o = p_t and
// *src_o its source, else *dst_o = -1.
GBLA_DEVINL void swap_plan(SwapPlanShared& s, int kb, int t, int* src_b, int* dst_o, int* src_o) {
  int last_to = -1, prev_same = -1;
  bool later = false;
  const int pt = t < kb ? s.p[t] : -1;
  if (t < kb) {
    for (int i = 0; i < kb; ++i) {
      const int q = s.p[i];
      if (i < t) {
        if (q == t) last_to = i;
        if (q == pt) prev_same = i;
      } else if (i > t && q == pt) {
        later = true;
      }
    }
    s.J[0][t] = last_to < 0 ? t : last_to;
  }
  __syncthreads();
  int cur = 0;
#pragma unroll 1
  for (int r = 0; r < 8; ++r) {
    if (t < kb) s.J[cur ^ 1][t] = s.J[cur][s.J[cur][t]];
    __syncthreads();
    cur ^= 1;
  }
  *dst_o = -1;
  if (t < kb) {
    const int pre_t = s.J[cur][t];
    *src_b = pt == t ? pre_t : (prev_same >= 0 ? s.J[cur][prev_same] : pt);
    if (pt >= kb && !later) {
      *dst_o = pt;
      *src_o = pre_t;
    }
  }
}
