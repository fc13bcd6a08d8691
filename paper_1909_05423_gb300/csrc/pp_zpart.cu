// pp_zpart.cu -- the z tridiagonal solve with every line split into chunks
// (Sec. "Solution of the Resulting Tridiagonal Matrices"; the parallel alternatives to the
// sequential Thomas sweep of Sec. "Cyclic Reduction Technique" / "Parallel Cyclic Reduction").
//
// The Thomas solve of a mode (pp_zsolve.cu) is two first-order linear recurrences over the rows,
// with the plan's precomputed multipliers w_k:
//     forward   g_k = (s d_k - g_{k-1}) w_k = a_k g_{k-1} + w_k s d_k,      a_k = -w_k, g_{-1} = 0,
//     backward  u_k = g_k - w_k u_{k+1}     = a_k u_{k+1} + g_k,            u_n = 0.
// One thread per line runs them in sequence, and reads every value twice: with fewer than about
// 150 k lines the GPU has too few threads for that, and a 256-row chain of double-float steps takes
// 0.3 ms however few lines there are.  Here a line is split into P chunks of M consecutive rows, one
// thread per chunk, whose M values stay in registers from the one load to the one store.  Each
// recurrence runs twice over them:
//   1. from a zero carry, only to get B, the value that leaves the chunk; the value that enters it
//      adds A x_in with A the product of the chunk's a_k;
//   2. from the chunk's true carry, keeping the values.
// A second run of the recurrence costs less than adding (product of a_i up to row k) x carry to the
// kept values of the first (which the products alone make 1.5 times as long), and its rounding is that
// of the plain sweep.
// The carry of chunk c is B_{c-1} + A_{c-1} (B_{c-2} + A_{c-2} (...)).  A decays by the mode's
// multiplier to the power M, so for most modes a few terms reach 2^-56 of the first and every thread
// sums them itself (Horner, at most kZpWindow terms); a CTA that holds a slower mode composes the
// chunk maps by recursive doubling instead, with warp shuffles inside a warp's run of chunks and one
// shared-memory exchange of the warps' totals.
// The multipliers and the order of the per-row operations are those of the Thomas sweeps; unlike
// cyclic reduction applied to the rows of the tridiagonal system, nothing forms the reduced systems'
// diagonals, whose distance from weak diagonal dominance (about the square of the lowest wavenumber)
// double-float coefficients would not keep.
//
// Periodic z is the Sherman-Morrison form of pp_zsolve.cu: the partial sums of y_0 = sum q_k d_k
// travel with the forward carries, the last chunk's thread forms c, and the back substitution starts
// from u_n = c.  The adjoint's transposed system is the same one (the row-scaled matrix is symmetric;
// FP64-class plans run it here).
//
// A CTA takes G adjacent real slots (consecutive threads: consecutive slots, so every row access of a
// warp is a few contiguous segments) x P chunks.  The singular mode's slots are solved by one more CTA
// each (pp_zsing.cuh).
//
// Arithmetic: double-float (pp_arith.cuh) on the plan's spill type, with the steps of the sweeps.  Range report: pp_range.cuh.
#include <algorithm>
#include <atomic>

#include "pp_range.cuh"
#include "pp_zmul.cuh"
#include "pp_zsing.cuh"

namespace pp {

__device__ __forceinline__ df zp_ld(const float2* p) { const float2 v = *p; return df{v.x, v.y}; }
__device__ __forceinline__ df zp_ld(const float* p) { return df{*p, 0.0f}; }
__device__ __forceinline__ void zp_st(float2* p, df v) { *p = make_float2(v.hi, v.lo); }
__device__ __forceinline__ void zp_st(float* p, df v) { *p = df_to_f32(v); }
__device__ __forceinline__ df zp_f2(float2 v) { return df{v.x, v.y}; }
__device__ __forceinline__ df zp_f2(const float* v) { return df{v[0], v[1]}; }

// Chunk maps x -> A x + B and their composition, (X o Y)(x) = X(Y(x)) = (A_X A_Y) x + (A_X B_Y + B_X).  Where a mode
// of the CTA runs the near -1 form (N1), A is kept as 1 - A, like the multipliers: a converged chunk has the same A all
// along the line, and the rounding of an A close to 1, the same in every chunk, would add up to 2^-48 / (1 + w) of
// the solution (3000 x 48 x 48, source of smooth blobs: relative error 6.2e-14 against 2.6e-14).
template <bool N1> __device__ __forceinline__ df zp_apply(df A, df B, df x) {
  if constexpr (N1) return zw_sub<true>(B, A, x);  // (B + x) - (1 - A) x
  else return A * x + B;
}
template <bool N1> __device__ __forceinline__ void zp_compose(df& A, df& B, df Ay, df By) {
  B = zp_apply<N1>(A, B, By);
  if constexpr (N1) A = zw_sub<true>(A, A, Ay);    // 1 - A A_y = a + a_y - a a_y
  else A = A * Ay;
}
__device__ __forceinline__ df zp_shfl(df v, int delta, bool up) {
  return up ? df{__shfl_up_sync(0xffffffffu, v.hi, delta), __shfl_up_sync(0xffffffffu, v.lo, delta)}
            : df{__shfl_down_sync(0xffffffffu, v.hi, delta), __shfl_down_sync(0xffffffffu, v.lo, delta)};
}

// Terms of the carry that a thread sums itself; a mode that needs more takes the doubling.
constexpr int kZpWindow = 8;

// Carry of every chunk from the chunk maps of its line.  dir = +1 (forward recurrence): the value
// that leaves chunk c - 1 (0 for chunk 0); dir = -1 (backward): the one that leaves chunk c + 1 (0 for
// the last).  sA, sB: one entry per thread.  Every thread of the CTA calls it, with the same `wide`;
// threads past the line (c >= P) hold the zero map: the doubling composes it
// before the last chunk of a backward line, whose B already holds what enters there.  `terms`: predecessors
// that matter to the thread's mode (windowed form).  Contains one barrier.
//
// Doubling (wide): a warp holds CW = 32 / G consecutive chunks of each of the CTA's G lines (lane =
// chunk-in-warp x G + line), one segment per line; the segments are scanned with shuffles (log2 CW
// levels: at level o a chunk composes its map with the one o chunks nearer the start), the segment
// totals are exchanged through shared memory, and each chunk composes the totals of the segments
// before its own.  (A near -1 mode always needs more terms than the window has: N1 comes with `wide`.)
template <bool N1>
__device__ __forceinline__ df zp_carry(df A, df B, float2* sA, float2* sB, int c, int P, int col, int G, int lgG,
                                       int dir, bool wide, int terms) {
  const bool fwd = dir > 0;
  if (!wide) {
    sA[threadIdx.x] = make_float2(A.hi, A.lo);
    sB[threadIdx.x] = make_float2(B.hi, B.lo);
    __syncthreads();
    const int have = fwd ? c : P - 1 - c;
    const int nt = min(have, terms);
    df x = df{0.f, 0.f};
    if (nt > 0) {
      int t = (int)threadIdx.x - dir * (nt << lgG);  // farthest chunk that matters
      x = zp_f2(sB[t]);
      for (int j = 1; j < nt; j++) {
        t += dir * G;
        x = zp_apply<N1>(zp_f2(sA[t]), zp_f2(sB[t]), x);
      }
    }
    return x;
  }
  const int lane = (int)threadIdx.x & 31;
  const int cw = 32 >> lgG;          // chunks per warp and line
  const int ci = lane >> lgG;        // chunk within the warp's segment
  const int seg = (int)threadIdx.x >> 5;
  const int nseg = ((int)blockDim.x + 31) >> 5;
  // 1. inclusive scan within the segment
  for (int o = 1; o < cw; o <<= 1) {
    const df An = zp_shfl(A, o * G, fwd), Bn = zp_shfl(B, o * G, fwd);
    if (fwd ? (ci >= o) : (ci + o < cw)) zp_compose<N1>(A, B, An, Bn);
  }
  // the inclusive map of the neighbouring chunk nearer the start (same segment unless at its edge)
  const df An1 = zp_shfl(A, G & 31, fwd), Bn1 = zp_shfl(B, G & 31, fwd);
  // 2. segment totals: the last chunk of a forward segment, the first of a backward one
  if (fwd ? (ci == cw - 1) : (ci == 0)) {
    sA[seg * G + col] = make_float2(A.hi, A.lo);
    sB[seg * G + col] = make_float2(B.hi, B.lo);
  }
  __syncthreads();
  // 3. L: the composition of the segments before this one (forward: segments 0 .. seg-1, applied
  // in that order; backward: the last segment down to seg+1); only its value at 0 is needed
  df Lb = df{0.f, 0.f};
  for (int t = 0; t < (fwd ? seg : nseg - 1 - seg); t++) {
    const int j = fwd ? t : nseg - 1 - t;
    Lb = zp_apply<N1>(zp_f2(sA[j * G + col]), zp_f2(sB[j * G + col]), Lb);
  }
  // the carry: the neighbour's output, its segment map applied to L's output (at the segment's
  // edge, L's output itself)
  const bool edge = fwd ? (ci == 0) : (ci == cw - 1);
  return edge ? Lb : zp_apply<N1>(An1, Bn1, Lb);
}

// The near -1 form out of line, as in the sweeps: few CTAs take it, and the others keep their registers.
__device__ __noinline__ df zp_carry_near1(df A, df B, float2* sA, float2* sB, int c, int P, int col, int G, int lgG,
                                          int dir) {
  return zp_carry<true>(A, B, sA, sB, c, P, col, G, lgG, dir, true, 0);
}

// The multipliers of a line, as stored (pp_zmul.cuh).
struct ZpW {
  const float2* wt;  // prefix, wlen entries
  int wlen;
  bool plus1;        // the table holds w but the thread runs the near -1 form: converts to 1 + w
  df winf, wlast;    // converged, and of the last row
};

// How a warp runs its rows.
//  ZP_FAST: every row of every lane is past the table prefix and not the last one, so w = winf
//           throughout.
//  ZP_TAB:  the multipliers come from the thread's rows of sW in shared memory.  (Taken row after row
//           from the table where they were used, and only by the lanes that needed them, they made the
//           prefix warps of a CTA three times as slow as the others, which waited at the barriers.)
//  ZP_NEAR: the same with the near -1 form of the products (pp_zmul.cuh).
enum { ZP_FAST = 0, ZP_TAB = 1, ZP_NEAR = 2 };

// Steps of the recurrences, in both runs those of the sweeps (pp_zsolve.cu: zr_fwd, zr_bwd): normalised for the
// double-float spill, unnormalised for the FP32 spill.  (Unnormalised first runs and inner steps of the double-float spill
// took 10 % less time, 256^3 0.109 against 0.125 ms, at about two bits of every carry and step.)
template <class S, int V> __device__ __forceinline__ df zp_step_f(df d, df g, df w) {
  if constexpr (V == ZP_NEAR) return zw_mul<true>(d - g, w);
  else if constexpr (sizeof(S) == 4) return mul_u(add_u(d, -g), w);
  else return (d - g) * w;
}
template <class S, int V> __device__ __forceinline__ df zp_step_b(df g, df w, df u) {
  if constexpr (V == ZP_NEAR) return zw_sub<true>(g, w, u);
  else if constexpr (sizeof(S) == 4) return add_u(g, -mul_u(w, u));
  else return g - w * u;
}

struct ZpRows {
  df winf;
  const float2* w;  // multipliers of the thread's rows
  template <int V> __device__ __forceinline__ df mult(int i) const {
    if constexpr (V == ZP_FAST) return winf;
    else return zp_f2(w[i]);
  }
};

// Rows past the line's end (the last chunk) have d = 0 and w = -1, which pass g and u on unchanged.
// scaled right-hand sides d_k in place of the raw values, and the value that leaves the chunk
template <class S, int M, int V>
__device__ __forceinline__ void zp_fwd1(df (&v)[M], df& B, const ZpRows& R, df scale, float& dmax) {
#pragma unroll
  for (int i = 0; i < M; i++) {
    v[i] = (sizeof(S) == 4) ? mul_u(v[i], scale) : v[i] * scale;
    track(dmax, v[i].hi);
    B = zp_step_f<S, V>(v[i], B, R.mult<V>(i));
  }
}
// g_k from the true carry, in place of d_k; rounded for the FP32 spill as the sweeps round it between
// their two passes, so that both give a plan the same results but for rare last-place flips
template <class S, int M, int V>
__device__ __forceinline__ void zp_fwd2(df (&v)[M], df& g, const ZpRows& R) {
#pragma unroll
  for (int i = 0; i < M; i++) {
    g = zp_step_f<S, V>(v[i], g, R.mult<V>(i));
    v[i] = (sizeof(S) == 4) ? df{df_to_f32(g), 0.0f} : g;
  }
}
// back substitution u_k = g_k - w_k u_{k+1}: the value that leaves the chunk
template <class S, int M, int V>
__device__ __forceinline__ void zp_bwd1(const df (&v)[M], df& u, const ZpRows& R) {
#pragma unroll
  for (int i = M - 1; i >= 0; i--) u = zp_step_b<S, V>(v[i], R.mult<V>(i), u);
}
// ... and from the true carry, keeping the values
template <class S, int M, int V>
__device__ __forceinline__ void zp_bwd2(df (&v)[M], df u, const ZpRows& R) {
#pragma unroll
  for (int i = M - 1; i >= 0; i--) {
    u = zp_step_b<S, V>(v[i], R.mult<V>(i), u);
    v[i] = u;
  }
}

#define ZP_DISPATCH(fn, ...)                               \
  do {                                                     \
    if (var == ZP_FAST) fn<S, M, ZP_FAST>(__VA_ARGS__);    \
    else if (var == ZP_TAB) fn<S, M, ZP_TAB>(__VA_ARGS__); \
    else fn<S, M, ZP_NEAR>(__VA_ARGS__);                   \
  } while (0)

// A of a converged chunk, (-w)^M, M a power of two; and 1 - A of one from v = 1 + w, in FP64 (two or three operations
// a doubling, in the few near -1 CTAs): three double-float roundings of a value that every chunk of the line applies
// were worth a third of the whole solve's error on 3000 x 48 x 48.
template <int M> __device__ __forceinline__ df zp_pow(df x) {
#pragma unroll
  for (int m = 1; m < M; m <<= 1) x = x * x;
  return x;
}
template <int M> __device__ __forceinline__ df zp_pow_near1(df v) {
  double x = (double)v.hi + (double)v.lo;
#pragma unroll
  for (int m = 1; m < M; m <<= 1) x = __fma_rn(-x, x, x + x);  // 1 - A^2 = 2 a - a a
  const float hi = (float)x;
  return df{hi, (float)(x - (double)hi)};
}

// CTAs of up to 1024 threads at 64 registers (8 or 16 rows a thread), 512 at 128 (32 rows)
template <int M> struct ZpThreads { static constexpr int v = M <= 16 ? 1024 : 512; };

template <class S, int M, bool PER>
__global__ void __launch_bounds__(ZpThreads<M>::v) k_zpart(const ZArgs a, int G, int lgG, int P) {
  // per-thread chunk maps (A, B) of the forward and the backward carries; periodic z: partial sums
  // of y_0, and c per line
  extern __shared__ float2 zp_sm[];
  float dmax = 0.0f, umax = 0.0f;
  if ((int)blockIdx.x < a.nsing) {
    pdl_wait();
    zsing_block<S>(a, (int)blockIdx.x, zp_sm, dmax, umax);
    range_report(a.rstat, a.dmin, a.umax, gridDim.x, dmax, umax);
    return;
  }
  const int T = (int)blockDim.x;
  float2 *fA = zp_sm, *fB = zp_sm + T, *bA = zp_sm + 2 * T, *bB = zp_sm + 3 * T;
  float2* sW = zp_sm + 4 * T + (int)threadIdx.x * (M + 1);  // M entries a thread (odd stride: no bank conflicts)
  float2* sQ = zp_sm + (5 + M) * T;  // T entries
  float2* sC = sQ + T;               // G entries
  const int tid = (int)threadIdx.x;
  const int col = tid & (G - 1);
  const int c = tid >> lgG;
  const long long s = (long long)((int)blockIdx.x - a.nsing) * G + col;
  const int n = a.nz;
  const long long PL = a.plane;

  // the slot's mode; padding slots, the singular mode and the threads that round the CTA up to
  // whole warps (c >= P) do no work but join every barrier
  const bool inb = c < P;
  bool live = inb && s < a.nreal;
  const ZMode* m = nullptr;
  if (live) {
    const unsigned row = a.fd_row.div((unsigned)s);
    const int cr = (int)(s - (long long)row * a.row_reals);
    live = cr < a.row_valid;
    if (live) {
      m = a.modes + ((long long)row * a.row_modes + (a.cplx ? (cr >> 1) : cr));
      live = !(m->flags & ZF_SINGULAR);
    }
  }
  const int k0 = c * M;
  ZpW W;
  W.wt = a.wtab;
  W.wlen = 0;
  W.winf = df{0.f, 0.f};
  W.wlast = df{0.f, 0.f};
  bool mine = false;
  int qlen = 0;
  if (live) {
    const int4 off = __ldg(reinterpret_cast<const int4*>(m));          // woff, wlen, qoff, qlen
    const float4 ww = __ldg(reinterpret_cast<const float4*>(m) + 1);   // winf, wlast
    W.winf = df{ww.x, ww.y};
    W.wlast = df{ww.z, ww.w};
    W.wlen = off.y;
    W.wt = a.wtab + off.x;
    mine = (m->flags & ZF_NEAR1) != 0;
    if (PER) qlen = off.w;
  }
  pdl_wait();
  const int nr = max(0, min(M, n - k0));  // rows of the chunk (below M only at the line's end)
  S* base = reinterpret_cast<S*>(a.data) + s + (long long)k0 * PL;
  df v[M];
  if (live && nr == M) {
#pragma unroll
    for (int i = 0; i < M; i++) v[i] = zp_ld(base + (long long)i * PL);
  } else {
#pragma unroll
    for (int i = 0; i < M; i++) v[i] = (live && i < nr) ? zp_ld(base + (long long)i * PL) : df{0.f, 0.f};
  }
  // a warp runs the near -1 form when any of its modes needs it (the others convert their w); every
  // warp holds all G lines, so all warps of the CTA agree
  const bool n1 = __any_sync(0xffffffffu, mine);
  W.plus1 = n1 && !mine;
  if (W.plus1) {
    W.winf = W.winf + df{1.f, 0.f};
    W.wlast = W.wlast + df{1.f, 0.f};
  }
  const df scale = df{a.scale[0], a.scale[1]};

  // A of a converged chunk and how many chunks back it reaches
  df A = n1 ? zp_pow_near1<M>(W.winf) : zp_pow<M>(-W.winf);
  const float reach = n1 ? 1.0f - A.hi : A.hi;
  const int terms = reach < 0x1p-56f ? 1 : (int)__fdividef(-56.0f, __log2f(fminf(reach, 0.999f))) + 1;
  const bool wide = n1 || __any_sync(0xffffffffu, live && terms > kZpWindow);
  const bool lanes_fast = __all_sync(0xffffffffu, k0 >= W.wlen && k0 + M < n);
  const int var = n1 ? ZP_NEAR : (lanes_fast ? ZP_FAST : ZP_TAB);
  ZpRows R;
  R.winf = W.winf;
  R.w = sW;
  if (var != ZP_FAST) {
    // the chunk's multipliers, read back by this thread only: asynchronous copies of the table's part
#pragma unroll
    for (int i = 0; i < M; i++) {
      const int k = k0 + i;
      if (k < W.wlen && k < n - 1) {
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((unsigned)__cvta_generic_to_shared(sW + i)),
                     "l"(__cvta_generic_to_global(W.wt + k)) : "memory");
      } else {
        const df w = k < n - 1 ? W.winf : (k == n - 1 ? W.wlast : df{n1 ? 0.f : -1.f, 0.f});
        sW[i] = make_float2(w.hi, w.lo);
      }
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    if (W.plus1)
      for (int i = 0; i < M && k0 + i < min(W.wlen, n - 1); i++) {
        const df w = zp_f2(sW[i]) + df{1.f, 0.f};
        sW[i] = make_float2(w.hi, w.lo);
      }
    // A of a chunk in the prefix (nothing passes through the first chunk, or through the last)
    if (k0 < W.wlen && c > 0 && c < P - 1) {
      A = df{n1 ? 0.f : 1.f, 0.f};
#pragma unroll
      for (int i = 0; i < M; i++) {
        const df w = zp_f2(sW[i]);
        A = n1 ? zw_sub<true>(w, w, A) : zw_neg_mul<false>(A, w);  // N1: 1 - A (1 - v) = v + a - v a
      }
    }
  }

  // forward recurrence
  df B = df{0.f, 0.f};
  ZP_DISPATCH(zp_fwd1, v, B, R, scale, dmax);
  if (PER) {
    df y0 = df{0.f, 0.f};
    if (k0 < qlen) {
#pragma unroll
      for (int i = 0; i < M; i++)
        if (k0 + i < qlen) y0 = y0 + zp_f2(__ldg(a.qtab + m->qoff + k0 + i)) * v[i];
    }
    sQ[tid] = make_float2(y0.hi, y0.lo);
  }
  df x = n1 ? zp_carry_near1(A, B, fA, fB, c, P, col, G, lgG, +1)
            : zp_carry<false>(A, B, fA, fB, c, P, col, G, lgG, +1, wide, terms);
  ZP_DISPATCH(zp_fwd2, v, x, R);

  // back substitution; periodic z starts it from c = (y_0 + y_{n-1} / gamma) / (1 + z_0 + z_{n-1} / gamma)
  df top = df{0.f, 0.f};
  if (PER && live && c == P - 1) {
    df y0 = df{0.f, 0.f};
    for (int j = 0; j * M < qlen; j++) y0 = y0 + zp_f2(sQ[(j << lgG) + col]);
    top = (y0 + x * zp_f2(m->igam)) * zp_f2(m->dsm);  // x == y_{n-1}
    sC[col] = make_float2(top.hi, top.lo);
  }
  if (nr < M) {
#pragma unroll
    for (int i = 0; i < M; i++)
      if (i >= nr) v[i] = df{0.f, 0.f};
  }
  B = top;
  ZP_DISPATCH(zp_bwd1, v, B, R);
  x = n1 ? zp_carry_near1(A, B, bA, bB, c, P, col, G, lgG, -1)
         : zp_carry<false>(A, B, bA, bB, c, P, col, G, lgG, -1, wide, terms);
  if (c == P - 1) x = top;
  pdl_start();
  ZP_DISPATCH(zp_bwd2, v, x, R);
  if (live) {
    if (PER && k0 < qlen) {
      const df cg = zp_f2(sC[col]) * zp_f2(m->gam);
#pragma unroll
      for (int i = 0; i < M; i++)
        if (k0 + i < qlen) v[i] = v[i] - cg * zp_f2(__ldg(a.qtab + m->qoff + k0 + i));
    }
    if (nr == M) {
#pragma unroll
      for (int i = 0; i < M; i++) {
        track(umax, v[i].hi);
        zp_st(base + (long long)i * PL, v[i]);
      }
    } else {
#pragma unroll
      for (int i = 0; i < M; i++)
        if (i < nr) {
          track(umax, v[i].hi);
          zp_st(base + (long long)i * PL, v[i]);
        }
    }
  }
  range_report(a.rstat, a.dmin, a.umax, gridDim.x, dmax, umax);
}
#undef ZP_DISPATCH

// Chunk count P = ceil(nz / M) and slots per CTA G (a power of two up to 16; the CTA is G P threads
// rounded up to whole warps); false when a line needs more than 512 chunks.  CTAs of up to 512
// threads, two or more of which share an SM (one loads while another computes), as long as a row's
// segment keeps 64 bytes; larger ones down to whole 32-byte sectors where the line is longer.
bool zpart_shape(int nz, int M, int elem, int* G, int* lgG, int* P) {
  const int p = (nz + M - 1) / M;
  if (p > 512) return false;
  const int tmax = M <= 16 ? 1024 : 512;
  int g = 16, lg = 4;
  while (g * elem > 64 && g * p > 512) { g >>= 1; lg--; }
  while (g > 1 && g * p > tmax) { g >>= 1; lg--; }
  *G = g; *lgG = lg; *P = p;
  return true;
}

template <class S, int M, bool PER>
static cudaError_t launch_zpart_t(const ZArgs& a, cudaStream_t st) {
  int G, lgG, P;
  if (!zpart_shape(a.nz, M, (int)sizeof(S), &G, &lgG, &P)) return cudaErrorInvalidConfiguration;
  const long long grid = (a.nreal + G - 1) / G + a.nsing;
  if (grid > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  const int threads = (G * P + 31) / 32 * 32;  // whole warps (the scans and the range report shuffle)
  const size_t sm = std::max(sizeof(float2) * ((5 + M + (PER ? 1 : 0)) * (size_t)threads + (PER ? G : 0)), kZsingSmem);
  // dynamic shared memory above 48 KB must be opted into, per device (one bit per device ordinal below
  // 64; higher ordinals set the attribute on every launch)
  static std::atomic<unsigned long long> attr_done{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = (dev >= 0 && dev < 64) ? (1ull << dev) : 0ull;
  if (!bit || !(attr_done.load(std::memory_order_acquire) & bit)) {
    e = cudaFuncSetAttribute(k_zpart<S, M, PER>, cudaFuncAttributeMaxDynamicSharedMemorySize, 208 * 1024);
    if (e != cudaSuccess) return e;
    attr_done.fetch_or(bit, std::memory_order_release);
  }
  return launch_pdl(a.pdl, k_zpart<S, M, PER>, (unsigned)grid, (unsigned)threads, sm, st, a, G, lgG, P);
}

template <class S, bool PER>
static cudaError_t launch_zpart_m(const ZArgs& a, int M, cudaStream_t st) {
  switch (M) {
    case 8: return launch_zpart_t<S, 8, PER>(a, st);
    case 16: return launch_zpart_t<S, 16, PER>(a, st);
    case 32: return launch_zpart_t<S, 32, PER>(a, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_zpart_impl(const ZArgs& a, bool df_spill, bool zper, int M, cudaStream_t st) {
  if (df_spill) return zper ? launch_zpart_m<float2, true>(a, M, st) : launch_zpart_m<float2, false>(a, M, st);
  return zper ? launch_zpart_m<float, true>(a, M, st) : launch_zpart_m<float, false>(a, M, st);
}

}  // namespace pp
