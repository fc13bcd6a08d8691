// pp_zsing.cuh -- the singular mode of a problem without Dirichlet faces (Sec. "Well-posedness"):
// remove the source mean, pin u_0 = 0, solve rows 1..n-1, shift the result to zero mean.
//
// One CTA solves one real slot of the mode: every thread holds a run of rows in registers, takes the
// pinned Thomas recurrences over them twice (from a zero carry, and from the true one), and the carries
// come from block-wide scans of the runs' affine maps; the two means are block-wide sums.  One thread of
// the sweeps took the mode before, in six passes over the line, each row waiting for the one before: 1.1 ms
// for 512 rows, beside 0.3 ms for all the other modes of a 512^3 grid.  Multipliers, the order of the steps
// and what is rounded to the spill type are those of that recurrence (zsing_serial).
#pragma once
#include "pp_internal.h"
#include "pp_range.cuh"
#include "pp_zmul.cuh"

namespace pp {

constexpr int kZsingRows = 16;                          // rows a thread holds
// Up to here one thread does all rows: six block-wide sums and scans take 24 us however few the rows, one thread 13 us for
// 8 rows, 17 for 24, 22 for 40 and 25 for 48 (z stage of 16 x 16 lines).
constexpr int kZsingSerial = 40;
constexpr size_t kZsingSmem = 64 * sizeof(float2);      // warp totals of a scan

__device__ __forceinline__ df zs_ld(const float2* p) { const float2 v = *p; return df{v.x, v.y}; }
__device__ __forceinline__ df zs_ld(const float* p) { return df{*p, 0.0f}; }
__device__ __forceinline__ void zs_st(float2* p, df v) { *p = make_float2(v.hi, v.lo); }
__device__ __forceinline__ void zs_st(float* p, df v) { *p = df_to_f32(v); }

// A value as it reads back from the spill array.
__device__ __forceinline__ df zs_round(const float2*, df v) { return v; }
__device__ __forceinline__ df zs_round(const float*, df v) { return df{df_to_f32(v), 0.0f}; }

__device__ __forceinline__ df zs_shfl(df v, int src) {
  return df{__shfl_sync(0xffffffffu, v.hi, src), __shfl_sync(0xffffffffu, v.lo, src)};
}
// Sum of v over the CTA (every thread, whole warps; sm: 32 entries, free again on return).
__device__ __forceinline__ df block_sum(df v, float2* sm) {
  const int lane = (int)threadIdx.x & 31, nw = (int)blockDim.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = v + zs_shfl(v, lane ^ o);
  if (lane == 0) sm[threadIdx.x >> 5] = make_float2(v.hi, v.lo);
  __syncthreads();
  const float2 t = lane < nw ? sm[lane] : make_float2(0.f, 0.f);
  df s = df{t.x, t.y};
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s = s + zs_shfl(s, lane ^ o);
  __syncthreads();
  return s;
}
// The value that enters this thread's run when every thread's run maps x -> A x + B and 0 enters the
// first run: run 0 (REV: that of the last thread).  sm: 64 entries, free again on return.
template <bool REV> __device__ __forceinline__ df block_carry(df A, df B, float2* sm) {
  const int lane = (int)threadIdx.x & 31, w = (int)threadIdx.x >> 5, nw = (int)blockDim.x >> 5;
  const int pl = REV ? 31 - lane : lane;  // place in the order of the runs
  auto before = [&](df v, int o) { return zs_shfl(v, REV ? (lane + o) & 31 : (lane - o) & 31); };
  // composition of the maps up to this one, within the warp
  auto inclusive = [&](df& a, df& b) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const df a0 = before(a, o), b0 = before(b, o);
      if (pl >= o) {
        b = a * b0 + b;
        a = a * a0;
      }
    }
  };
  inclusive(A, B);
  const df Ap = before(A, 1), Bp = before(B, 1);
  if (pl == 31) {
    sm[w] = make_float2(A.hi, A.lo);
    sm[32 + w] = make_float2(B.hi, B.lo);
  }
  __syncthreads();
  // the warps' totals, in the same order of lanes (REV: warp nw - 1 on lane 31)
  const int j = REV ? lane - (32 - nw) : lane;
  const bool has = j >= 0 && j < nw;
  df WA = has ? df{sm[j].x, sm[j].y} : df{1.f, 0.f}, WB = has ? df{sm[32 + j].x, sm[32 + j].y} : df{0.f, 0.f};
  inclusive(WA, WB);
  const int mine = REV ? w + (32 - nw) : w;                       // this warp's lane
  const bool first = REV ? w == nw - 1 : w == 0;
  df x = zs_shfl(WB, REV ? (mine + 1) & 31 : (mine - 1) & 31);
  if (first) x = df{0.f, 0.f};
  __syncthreads();
  return pl == 0 ? x : Ap * x + Bp;
}

// One thread, any line length (short lines, and lines of more rows than a CTA holds in registers): the pinned Thomas
// recurrence of rows 1..n-1, whose multipliers -k/(k+1) the table stores as 1 + w.
template <class S>
__device__ __noinline__ void zsing_serial(S* base, long long P, int n, df scale, const float2* wt, float& dmax,
                                          float& umax) {
  // The pinned system is consistent only for a zero-mean right-hand side; a remainder c of the mean
  // would add a profile growing like c k^2 / 2.  One double-float pass leaves the rounding of a sum
  // of n values of the source's own mean magnitude (relative 2^-48 per term), so a second pass takes
  // the mean of the residuals, which are of the size of the fluctuations.
  auto wk = [&](int r) { const float2 v = __ldg(wt + r); return df{v.x, v.y}; };
  const df rn = df_rcp(df{(float)n, 0.f});
  df sum = df{0.f, 0.f};
  for (int k = 0; k < n; k++) sum = sum + zs_ld(base + k * P);
  df mean = sum * rn;
  df rsum = df{0.f, 0.f};
  for (int k = 0; k < n; k++) rsum = rsum + (zs_ld(base + k * P) - mean);
  mean = mean + rsum * rn;
  // rows 1..n-1 of the pinned system; multipliers of the sub-system in the table
  df g = df{0.f, 0.f};
  for (int k = 1; k < n; k++) {
    df d = (zs_ld(base + k * P) - mean) * scale;
    track(dmax, d.hi);
    g = zw_mul<true>(d - g, wk(k - 1));  // the pinned table is stored as 1 + w
    zs_st(base + k * P, g);
  }
  df u = df{0.f, 0.f};
  df usum = df{0.f, 0.f};
  for (int k = n - 1; k >= 1; k--) {
    df gk = zs_ld(base + k * P);
    u = (k == n - 1) ? gk : zw_sub<true>(gk, wk(k - 1), u);
    usum = usum + u;
    zs_st(base + k * P, u);
  }
  df umean = usum * rn;
  // the same second pass for the solution's mean (u_0 = 0 is pinned)
  df ursum = -umean;
  for (int k = 1; k < n; k++) ursum = ursum + (zs_ld(base + k * P) - umean);
  umean = umean + ursum * rn;
  zs_st(base, -umean);
  track(umax, umean.hi);
  for (int k = 1; k < n; k++) {
    const df v = zs_ld(base + k * P) - umean;
    track(umax, v.hi);
    zs_st(base + k * P, v);
  }
}

// Real slot `part` of the singular mode (mode (0, 0): slots 0, and 1 for a complex mode), by one CTA
// (every thread calls it; whole warps).  sm: kZsingSmem bytes.
template <class S>
__device__ __noinline__ void zsing_block(const ZArgs& a, int part, float2* sm, float& dmax, float& umax) {
  S* base = reinterpret_cast<S*>(a.data) + part;
  const long long P = a.plane;
  const int n = a.nz;
  const df scale = df{a.scale[0], a.scale[1]};
  const int R = (n + (int)blockDim.x - 1) / (int)blockDim.x;
  if (R > kZsingRows || n <= kZsingSerial) {
    if (threadIdx.x == 0) zsing_serial<S>(base, P, n, scale, a.wtab + a.modes[0].woff, dmax, umax);
    return;
  }
  const df zero = df{0.f, 0.f};
  const int k0 = (int)threadIdx.x * R;
  const int nr = max(0, min(R, n - k0));  // rows of this thread
  const float2* wt = a.wtab + a.modes[0].woff - 1 + k0;  // row k >= 1: entry k - 1, stored as 1 + w
  auto wk = [&](int i) { const float2 x = __ldg(wt + i); return df{x.x, x.y}; };
  df v[kZsingRows];
#pragma unroll
  for (int i = 0; i < kZsingRows; i++) v[i] = i < nr ? zs_ld(base + (long long)(k0 + i) * P) : zero;
  const df rn = df_rcp(df{(float)n, 0.f});
  // the mean, and in a second pass the mean of what the first left (see zsing_serial)
  df t = zero;
#pragma unroll
  for (int i = 0; i < kZsingRows; i++)
    if (i < nr) t = t + v[i];
  df mean = block_sum(t, sm) * rn;
  t = zero;
#pragma unroll
  for (int i = 0; i < kZsingRows; i++)
    if (i < nr) t = t + (v[i] - mean);
  mean = mean + block_sum(t, sm) * rn;
  // forward elimination of rows 1..n-1
  df A = df{1.f, 0.f}, x = zero;
#pragma unroll
  for (int i = 0; i < kZsingRows; i++)
    if (i < nr) {
      v[i] = (v[i] - mean) * scale;
      if (k0 + i > 0) {
        track(dmax, v[i].hi);
        const df w = wk(i);
        x = zw_mul<true>(v[i] - x, w);
        A = zw_neg_mul<true>(A, w);
      }
    }
  df g = block_carry<false>(A, x, sm);
#pragma unroll
  for (int i = 0; i < kZsingRows; i++)
    if (i < nr && k0 + i > 0) {
      g = zw_mul<true>(v[i] - g, wk(i));
      v[i] = zs_round(base, g);
    }
  // back substitution
  x = zero;
#pragma unroll
  for (int i = kZsingRows - 1; i >= 0; i--)
    if (i < nr && k0 + i > 0) x = zw_sub<true>(v[i], wk(i), x);
  df u = block_carry<true>(A, x, sm);
  t = zero;
#pragma unroll
  for (int i = kZsingRows - 1; i >= 0; i--)
    if (i < nr) {
      if (k0 + i > 0) {
        u = zw_sub<true>(v[i], wk(i), u);
        t = t + u;
        v[i] = zs_round(base, u);
      } else {
        v[i] = zero;  // u_0 is pinned
      }
    }
  // zero mean, in two passes like the source's
  mean = block_sum(t, sm) * rn;
  t = zero;
#pragma unroll
  for (int i = 0; i < kZsingRows; i++)
    if (i < nr) t = t + (v[i] - mean);
  mean = mean + block_sum(t, sm) * rn;
#pragma unroll
  for (int i = 0; i < kZsingRows; i++)
    if (i < nr) {
      const df o = v[i] - mean;
      track(umax, o.hi);
      zs_st(base + (long long)(k0 + i) * P, o);
    }
}

}  // namespace pp
