// pp_hlines.cuh -- FP64-class line transforms of power-of-two lengths in block-scaled arithmetic.
//
// The transforms, their recipes and their layouts are those of pp_lines.cuh; the arithmetic is that of
// pp_hx.cuh.  A thread holds 16 complex values: two radix-8 butterflies, or as many of the last stage's.
//  * Forward real kinds and C2C read the inputs of their first butterflies from global memory straight
//    into registers (the pair of butterflies j and MC/8-1-j holds whole quads u[4k..4k+3] of the Makhoul
//    order), find the line's scale there, and write the first stage's output to shared memory.
//  * Inverse kinds read Hermitian items (k, MC-k) instead, and write the FFT input.
//  * The last stage's output of the inverse kinds, the type-IV kinds and C2C leaves from registers; the
//    Hermitian split of the forward kinds reads it back from shared memory.
// So a line makes three trips through shared memory, where pp_lines.cuh takes four or five.
//  * A CTA prefetches a later tile into L2 while it waits for its own.
//  * The post-processing of DCT-II forms W_k = A + B and W_{M-k} = conj(A - B) exp(-i pi/4), A = 2 E_k w,
//    B = 2 O_k w w_N^k, w = exp(-i pi k/2N): two products and a rotation per item instead of three
//    products, since exp(-i pi (M-k)/2N) = exp(-i pi/4) conj(w).  DCT-III reverses it.
//
// x lines (OY false): a line's MC/16 threads are consecutive lanes, shared memory holds lines with one
// padding slot in 32.  y lines: lanes run over the tile's lines first, [element][line], so every global
// access is a run of adjacent columns and every shared-memory access of a warp is contiguous.
//
// What bounds them: load latency and issue slots together.  The 512-point kernels issue 125 to 145
// instructions a point (double-float pairs: 195 to 230) at 55 to 62 % of the issue slots, load stalls
// leading, with 16 to 24 warps an SM (registers).  1024^3 (ms; double-float kernels at their autotuned shapes /
// these): x-forward 7.8 / 5.7, y-forward 7.6 / 5.8, y-inverse 8.0 / 5.8, x-inverse 7.8 / 6.3; 512-point C2C
// columns at 512^3 1.17 / 0.53.  The four transforms alone, forward and back, differ from FP64 by 1.0e-14 to
// 2.0e-14 (double-float pairs: 3.4e-14 to 5.5e-14).
#pragma once
#include "pp_hx.cuh"
#include "pp_lines.cuh"

namespace pp {

enum { HG_FWD = 0, HG_INV = 1, HG_IV = 2, HG_C2CF = 3, HG_C2CI = 4 };  // kind groups

// read-only loads of twiddles
__device__ __forceinline__ htwa hld(const htwa* p) {
  const int4 v = __ldg(reinterpret_cast<const int4*>(p));
  return htwa{v.x, v.y, __int_as_float(v.z), __int_as_float(v.w)};
}
__device__ __forceinline__ htwb hld(const htwb* p) {
  const float2 v = __ldg(reinterpret_cast<const float2*>(p));
  return htwb{v.x, v.y};
}

// Streamed inputs bypass L1, which then keeps the twiddle tables (28 KB beside three CTAs' shared memory).  They are
// the kernel before's output, or (z lines) this kernel's own: coherent loads, volatile and with a memory clobber so
// that the compiler keeps them behind pdl_wait().
__device__ __forceinline__ df hld1(const double* p) {
  double a;
  asm volatile("ld.global.L1::no_allocate.f64 %0, [%1];\n" : "=d"(a) : "l"(__cvta_generic_to_global(p)) : "memory");
  return df_from_double(a);
}
__device__ __forceinline__ df hld1(const float2* p) {
  float a, b;
  asm volatile("ld.global.L1::no_allocate.v2.f32 {%0, %1}, [%2];\n" : "=f"(a), "=f"(b) : "l"(__cvta_generic_to_global(p)) : "memory");
  return df{a, b};
}
__device__ __forceinline__ void hld2(const double* p, df* t) {
  double a, b;
  asm volatile("ld.global.L1::no_allocate.v2.f64 {%0, %1}, [%2];\n" : "=d"(a), "=d"(b) : "l"(__cvta_generic_to_global(p)) : "memory");
  t[0] = df_from_double(a);
  t[1] = df_from_double(b);
}
__device__ __forceinline__ void hld2(const float2* p, df* t) {
  asm volatile("ld.global.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];\n"
      : "=f"(t[0].hi), "=f"(t[0].lo), "=f"(t[1].hi), "=f"(t[1].lo) : "l"(__cvta_generic_to_global(p)) : "memory");
}
// four adjacent reals of an x line (32-byte aligned FP64, or spill pairs)
__device__ __forceinline__ void hld4(const double* p, df* t) {
  double a, b, c, d;
  asm volatile("ld.global.L1::no_allocate.v4.f64 {%0, %1, %2, %3}, [%4];\n" : "=d"(a), "=d"(b), "=d"(c), "=d"(d) : "l"(__cvta_generic_to_global(p)) : "memory");
  t[0] = df_from_double(a);
  t[1] = df_from_double(b);
  t[2] = df_from_double(c);
  t[3] = df_from_double(d);
}
__device__ __forceinline__ void hld4(const float2* p, df* t) {
  hld2(p, t);
  hld2(p + 2, t + 2);
}

template <bool OY, int MC> struct HShape {
  static constexpr int TPL = MC / 16;                                  // threads of a line
  static constexpr int T = MC >= 1024 ? (OY ? 512 : 128) : MC == 512 ? 256 : 128;
  static constexpr int NL = T / TPL;                                   // lines of a CTA
  static constexpr int LDM = MC + (MC >= 256 ? MC / 32 : 8) + 1;       // x: stride of a line
  static constexpr int BUF = OY ? NL * MC : NL * LDM;                  // complex values
  static constexpr int W = T / 32;
  // only the integer twiddles are in shared memory (their remainders come through L1): three CTAs of eight
  // 512-point lines fit an SM
  static constexpr size_t smem = (size_t)BUF * 16 + (size_t)MC * 16 + (OY || TPL > 32 ? (size_t)W * NL * 8 : 0);
};

template <bool OY, int MC> struct HLine {
  using H = HShape<OY, MC>;
  hcx* buf;           // x: the line's values; y: the tile's, offset by the line
  const htwa* ta;
  const htwb* tb;
  int lt;
  // elements i + off (off a compile-time multiple that keeps the padding of i, see pp_fft.cuh)
  __device__ __forceinline__ hcx* at(int i) const { return buf + (OY ? i * H::NL : pad(i)); }
  static constexpr __device__ int step(int off) { return OY ? off * H::NL : off + (off >> 5); }
  __device__ __forceinline__ void sync() const {
    if constexpr (!OY && H::TPL <= 32) __syncwarp();
    else __syncthreads();
  }
  // butterfly j of the stage (stride S, radix RAD): DFT, twiddles, store
  template <int RAD, bool INV, int S, int TWOFF> __device__ __forceinline__ void finish(hcx* a, int j) const {
    hdft<RAD, INV>(a);
    const int p = j / S, q = j % S;
    // x: the first stage's output 8p + t goes to (MC/8 + 1) t + p, where the second stage reads it: both
    // sides then touch distinct banks (8p + t with one slot in 32 is a four-way conflict of 16-byte stores)
    constexpr bool TR = !OY && S == 1;
    hcx* y = TR ? buf + p : at(q + S * RAD * p);
    auto pos = [](int t) constexpr { return TR ? (MC / 8 + 1) * t : step(S * t); };
    if constexpr (S * RAD == MC) {
#pragma unroll
      for (int t = 0; t < RAD; t++) y[pos(t)] = a[t];
    } else {
      constexpr int PS = MC / (S * RAD);  // twiddles per t
      const htwa* wa = ta + TWOFF + p;
      const htwb* wb = tb + TWOFF + p;
      y[0] = hquarter(a[0]);
#pragma unroll
      for (int t = 1; t < RAD; t++) y[pos(t)] = hmul<INV>(a[t], wa[(t - 1) * PS], hld(wb + (t - 1) * PS));
    }
  }
};

// Stages from stride S on, values in shared memory.  KEEP: the last stage's results stay in a (butterfly i
// of NB: j = lt + TPL i, and its mirror MC/RAD - 1 - j at i + NB/2); otherwise they are stored.
template <bool OY, int MC, bool INV, int S, int TWOFF, bool KEEP>
__device__ __forceinline__ void h_stages(const HLine<OY, MC>& L, hcx (&a)[16]) {
  if constexpr (S < MC) {
    using H = HShape<OY, MC>;
    constexpr int RAD = CtRadix<MC / S>::v, NBL = MC / RAD, NB = 16 / RAD;
    constexpr bool last = S * RAD == MC;
    auto jof = [&](int i) {
      return (!KEEP || !last || i < NB / 2) ? L.lt + H::TPL * i : NBL - 1 - (L.lt + H::TPL * (i - NB / 2));
    };
#pragma unroll
    for (int i = 0; i < NB; i++) {
      const int j = jof(i);
      constexpr bool TR = !OY && S == 8;  // as the first stage left it (HLine::finish)
      const hcx* x = TR ? L.buf + (MC / 8 + 1) * (j & 7) + (j >> 3) : L.at(j);
#pragma unroll
      for (int u = 0; u < RAD; u++) a[i * RAD + u] = x[TR ? u * (NBL / 8) : HLine<OY, MC>::step(u * NBL)];
    }
    if constexpr (last && KEEP) {
#pragma unroll
      for (int i = 0; i < NB; i++) hdft<RAD, INV>(a + i * RAD);
    } else {
      L.sync();
#pragma unroll
      for (int i = 0; i < NB; i++) L.template finish<RAD, INV, S, TWOFF>(a + i * RAD, jof(i));
      L.sync();
      constexpr int NEXT = (S * RAD < MC) ? TWOFF + (MC / (S * RAD)) * (RAD - 1) : TWOFF;
      h_stages<OY, MC, INV, S * RAD, NEXT, KEEP>(L, a);
    }
  }
}

// Sum and maximum over the threads of a line (fixed order).  red: W x NL pairs; y and lines of more than a
// warp: one barrier.
template <bool OY, int MC>
__device__ __forceinline__ void h_line_stats(float& mx, float& l1, float2* red, int L) {
  using H = HShape<OY, MC>;
  constexpr int lo = OY ? H::NL : 1, hi = OY ? 32 : (H::TPL < 32 ? H::TPL : 32);
#pragma unroll
  for (int o = lo; o < hi; o <<= 1) {
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    l1 += __shfl_xor_sync(0xffffffffu, l1, o);
  }
  if constexpr (OY || H::TPL > 32) {
    constexpr int W = OY ? H::W : H::TPL / 32;
    const int w = OY ? (int)threadIdx.x >> 5 : ((int)threadIdx.x >> 5) % W;
    if (OY ? ((int)threadIdx.x & 31) < H::NL : ((int)threadIdx.x & 31) == 0) red[w * H::NL + L] = make_float2(mx, l1);
    __syncthreads();
    mx = l1 = 0.0f;
#pragma unroll
    for (int i = 0; i < W; i++) {
      const float2 v = red[i * H::NL + L];
      mx = fmaxf(mx, v.x);
      l1 += v.y;
    }
  }
}

// Registers a thread may take (the launch bound is the CTAs that leaves).  The 16 values of a thread are 64
// registers; with more to spare the compiler loads twiddles early, and two CTAs of 256 threads beat three
// (1024^3: y 6.6 -> 6.0 ms, C2C of 512 points 0.66 -> 0.51), except in the forward x kernels, which wait for
// their loads first and want the warps (5.9 against 7.0 ms).
template <int HG, bool OY, int MC> struct HRegs {
  static constexpr int v = (!OY && HG == HG_FWD) ? (MC == 512 ? 80 : 96) : 112;
};

template <int HG, class SI, class SO, bool OY, int MC>
__global__ void __launch_bounds__((HShape<OY, MC>::T), (65536 / HRegs<HG, OY, MC>::v / HShape<OY, MC>::T)) k_hlines(const __grid_constant__ LineArgs a) {
  using H = HShape<OY, MC>;
  constexpr int M = MC, TPL = H::TPL, NL = H::NL;
  constexpr bool C2C = HG == HG_C2CF || HG == HG_C2CI;
  constexpr bool INV = HG == HG_INV || HG == HG_C2CI;
  const int N = a.N, kind = a.kind;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  hcx* buf = reinterpret_cast<hcx*>(smem_raw);
  htwa* sta = reinterpret_cast<htwa*>(buf + H::BUF);
  float2* red = reinterpret_cast<float2*>(sta + MC);
  const htwa* gta = reinterpret_cast<const htwa*>(a.htab);
  const htwb* gtb = reinterpret_cast<const htwb*>(gta + MC);
  const htwa* x1a = reinterpret_cast<const htwa*>(a.haux);   // pre/post twiddles: two tables
  const htwb* x1b = reinterpret_cast<const htwb*>(x1a + (M + 2));
  const htwa* x2a = reinterpret_cast<const htwa*>(x1b + (M + 2));
  const htwb* x2b = reinterpret_cast<const htwb*>(x2a + (M + 2));
  for (int i = threadIdx.x; i < MC; i += H::T)
    cp_async_cx(reinterpret_cast<cx<df>*>(sta) + i, reinterpret_cast<const cx<df>*>(gta) + i);
  cp_async_commit();

  HLine<OY, MC> ln;
  const int tid = (int)threadIdx.x;
  const int L = OY ? tid % NL : tid / TPL;
  ln.lt = OY ? tid / NL : tid % TPL;
  ln.ta = sta;
  ln.tb = gtb;
  ln.buf = buf + (OY ? L : L * H::LDM);
  const int lt = ln.lt;
  int line0, nl;
  if (!OY) {
    line0 = (int)blockIdx.x * NL;
    nl = min(NL, a.nlines - line0);
  } else {
    const int plane = (int)a.fd_nblk.div(blockIdx.x);
    const int c0 = ((int)blockIdx.x - plane * a.nblk) * a.tx;
    line0 = plane * a.lines_per_plane + c0 * a.parts;
    nl = min(a.tx, a.ncols - c0) * a.parts;
  }
  const bool act = L < nl;
  const unsigned g = (unsigned)(line0 + (act ? L : 0));
  const SI* in = reinterpret_cast<const SI*>(a.in) + line_base(a, g, false);
  const long long ip = a.in_pos, op = a.out_pos;
  auto rd = [&](int j) -> df { return act ? hld1(in + (long long)j * ip) : df{0.f, 0.f}; };
  // complex value k (spill arrays: 16-byte aligned pairs)
  auto rdc = [&](int k, df& re, df& im) {
    if constexpr (std::is_same<SI, float2>::value) {
      if (act) {
        df t[2];
        hld2(in + (long long)k * ip, t);
        re = t[0];
        im = t[1];
        return;
      }
    }
    re = im = df{0.f, 0.f};
  };
  pdl_wait();
  prefetch_tile<SI, OY>(a, blockIdx.x + a.ahead, kind == LK_C2R ? M + 1 : N);
  float mx = 0.0f, l1 = 0.0f;
  // Spill pairs come unnormalised, and a line of cancelled values may hold them in the low parts alone: the
  // leading part becomes the nearest FP32 value of the pair, for the line's scale and the split at it.
  auto stat = [&](df& v) {
    if constexpr (std::is_same<SI, float2>::value) {
      const float t = __fadd_rn(v.hi, v.lo);
      v.lo = __fsub_rn(v.lo, __fsub_rn(t, v.hi));
      v.hi = t;
    }
    hx_stat(mx, l1, v.hi);
  };
  hcx v[16];
  float S;
  if constexpr (HG != HG_INV) {
    // ---- inputs of butterflies lt and M/8-1-lt: element j + (M/8) u at v[u], v[8 + u]
    constexpr int NBL = M / 8;
    const int j0 = lt, j1 = NBL - 1 - lt;
    df r[16][2];
    auto quads = [&](auto&& fn) {
      // fn(k, &z_k, &z_{M-1-k}), k < M/2
#pragma unroll
      for (int u = 0; u < 4; u++) {
        fn(j0 + NBL * u, r[u], r[8 + 7 - u]);
        fn(j1 + NBL * u, r[8 + u], r[7 - u]);
      }
    };
    if constexpr (C2C) {
#pragma unroll
      for (int u = 0; u < 8; u++) {
        rdc(j0 + NBL * u, r[u][0], r[u][1]);
        rdc(j1 + NBL * u, r[8 + u][0], r[8 + u][1]);
      }
    } else if (HG == HG_FWD && kind == LK_R2C) {
#pragma unroll
      for (int u = 0; u < 16; u++) {
        const int k = (u < 8 ? j0 : j1) + NBL * (u & 7);
        if constexpr (!OY) {
          if (a.vec_ok) {
            if (act) hld2(in + 2 * k, r[u]);
            else r[u][0] = r[u][1] = df{0.f, 0.f};
            continue;
          }
        }
        r[u][0] = rd(2 * k);
        r[u][1] = rd(2 * k + 1);
      }
    } else if constexpr (HG == HG_FWD) {
      // DCT-II / DST-II: z_k = (u_4k, u_4k+2), z_{M-1-k} = +-(u_4k+3, u_4k+1)
      quads([&](int k, df* z0, df* z1) {
        if constexpr (!OY) {
          if (a.vec_ok) {
            if (act) {
              df t[4];
              hld4(in + 4 * k, t);
              z0[0] = t[0];
              z1[1] = t[1];
              z0[1] = t[2];
              z1[0] = t[3];
            } else {
              z0[0] = z0[1] = z1[0] = z1[1] = df{0.f, 0.f};
            }
            return;
          }
        }
        z0[0] = rd(4 * k);
        z0[1] = rd(4 * k + 2);
        z1[0] = rd(4 * k + 3);
        z1[1] = rd(4 * k + 1);
      });
    } else {
      // DCT-IV / DST-IV: (u_2n, u_{N-1-2n}) or the other way round
      quads([&](int n, df* z0, df* z1) {
        df lo[2], hi[2];  // u_2n, u_2n+1; u_{N-2-2n}, u_{N-1-2n}
        bool done = false;
        if constexpr (!OY) {
          if (a.vec_ok) {
            if (act) {
              hld2(in + 2 * n, lo);
              hld2(in + (N - 2 - 2 * n), hi);
            } else {
              lo[0] = lo[1] = hi[0] = hi[1] = df{0.f, 0.f};
            }
            done = true;
          }
        }
        if (!done) {
          lo[0] = rd(2 * n);
          lo[1] = rd(2 * n + 1);
          hi[0] = rd(N - 2 - 2 * n);
          hi[1] = rd(N - 1 - 2 * n);
        }
        const bool c4 = kind == LK_DCT4;
        z0[0] = c4 ? lo[0] : hi[1];
        z0[1] = c4 ? hi[1] : lo[0];
        z1[0] = c4 ? hi[0] : lo[1];
        z1[1] = c4 ? lo[1] : hi[0];
      });
    }
#pragma unroll
    for (int u = 0; u < 16; u++) {
      stat(r[u][0]);
      stat(r[u][1]);
    }
    h_line_stats<OY, MC>(mx, l1, red, L);
    pdl_start();
    S = hx_scale(a.hs, mx, l1);
#pragma unroll
    for (int u = 0; u < 16; u++) v[u] = hcx{hx_from(r[u][0], S), hx_from(r[u][1], S)};
    if (HG == HG_FWD && kind == LK_DST2) {
      // samples of odd index change sign: the halves of the Makhoul order from M/2 on (u < 4: k < M/2)
#pragma unroll
      for (int u = 4; u < 8; u++) {
        v[u] = hcx{-v[u].re, -v[u].im};
        v[8 + u] = hcx{-v[8 + u].re, -v[8 + u].im};
      }
    }
    if constexpr (HG == HG_IV) {
#pragma unroll
      for (int u = 0; u < 16; u++) {
        const int k = (u < 8 ? j0 : j1) + NBL * (u & 7);
        v[u] = hmul<false>(v[u], hld(x1a + k), hld(x1b + k));
      }
    }
    cp_async_wait_all();
    __syncthreads();
    ln.template finish<8, INV, 1, 0>(v, j0);
    ln.template finish<8, INV, 1, 0>(v + 8, j1);
    ln.sync();
    h_stages<OY, MC, INV, 8, (M / 8) * 7, HG != HG_FWD>(ln, v);
  } else {
    // ---- Hermitian items k = lt + TPL i and the middle one (thread 0 of the line)
    df r[8][4], rm[2];
    const bool c2r = kind == LK_C2R, c3 = kind == LK_DCT3;
    auto item = [&](int k, df* y) {
      if (c2r) {
        rdc(k, y[0], y[1]);
        rdc(M - k, y[2], y[3]);
        if (k == 0) y[1] = y[3] = df{0.f, 0.f};
      } else {
        auto row = [&](int j) { return c3 ? j : N - 1 - j; };
        y[0] = rd(row(k));
        y[1] = k > 0 ? rd(row(N - k)) : df{0.f, 0.f};
        y[2] = rd(row(M - k));
        y[3] = rd(row(M + k));
      }
    };
#pragma unroll
    for (int i = 0; i < 8; i++) item(lt + TPL * i, r[i]);
    rm[0] = rm[1] = df{0.f, 0.f};
    if (lt == 0) {
      if (c2r) rdc(M / 2, rm[0], rm[1]);
      else {
        rm[0] = rd(c3 ? M / 2 : N - 1 - M / 2);
        rm[1] = rd(c3 ? N - M / 2 : M / 2 - 1);
      }
    }
#pragma unroll
    for (int i = 0; i < 8; i++)
#pragma unroll
      for (int c = 0; c < 4; c++) stat(r[i][c]);
    // (the middle item takes its two values as both of its pairs: they count twice)
#pragma unroll
    for (int c = 0; c < 2; c++) {
      stat(rm[c]);
      hx_stat(mx, l1, rm[c].hi);
    }
    h_line_stats<OY, MC>(mx, l1, red, L);
    pdl_start();
    S = hx_scale(a.hs, mx, l1);
    // E = X_k + conj X_{M-k}, O = (X_k - conj X_{M-k}) conj(w_N^k), both / 4; Z_k = E + i O, Z_{M-k} its
    // partner.  DCT-III / DST-III: X_k = A c, conj X_{M-k} = B c with A = Y_k - i Y_{N-k},
    // B = (Y_{M-k} + i Y_{M+k}) exp(-i pi/4), c = conj(exp(-i pi k/2N)).
    auto pre = [&](int k, const hx* y, bool mid) {
      const hcx A = c2r ? hcx{y[0], y[1]} : hcx{y[0], -y[1]};
      const hcx B = c2r ? hcx{y[2], -y[3]} : hrot8<false>(hcx{y[2], y[3]});
      const hcx E = c2r ? hquarter(A + B) : hmul<true>(A + B, hld(x1a + k), hld(x1b + k));
      const hcx O = hmul<true>(A - B, c2r ? hld(x1a + k) : hld(x2a + k), c2r ? hld(x1b + k) : hld(x2b + k));
      *ln.at(k) = hcx{E.re - O.im, E.im + O.re};
      if (!mid && k > 0) *ln.at(M - k) = hcx{E.re + O.im, O.re - E.im};
    };
#pragma unroll
    for (int i = 0; i < 8; i++) {
      const hx y[4] = {hx_from(r[i][0], S), hx_from(r[i][1], S), hx_from(r[i][2], S), hx_from(r[i][3], S)};
      pre(lt + TPL * i, y, false);
    }
    if (lt == 0) {
      const hx y0 = hx_from(rm[0], S), y1 = hx_from(rm[1], S);
      const hx y[4] = {y0, y1, y0, y1};
      pre(M / 2, y, true);
    }
    cp_async_wait_all();
    __syncthreads();
    h_stages<OY, MC, true, 1, 0, true>(ln, v);
  }

  // ---- output
  const float f = hx_unscale(a.hs, S);
  SO* out = reinterpret_cast<SO*>(a.out) + line_base(a, g, true);
  constexpr bool F64 = std::is_same<SO, double>::value;
  const int E = (int)(__float_as_uint(f) >> 23) - 127;  // f = 2^E
  const bool bad = !(S == S);
  auto cv = [&](hx x) {
    if constexpr (F64) return bad ? __longlong_as_double(0x7ff8000000000000ll) : hx_to_double(x, E);
    else return hx_to(x, f);
  };
  auto wr = [&](int j, hx x) {
    if (!act) return;
    if constexpr (F64) {
      out[(long long)j * op] = cv(x);
    } else {
      const df t = cv(x);
      out[(long long)j * op] = make_float2(t.hi, t.lo);
    }
  };
  auto wrc = [&](int k, hcx z) {
    if constexpr (std::is_same<SO, float2>::value) {
      const df re = hx_to(z.re, f), im = hx_to(z.im, f);
      if (act) *reinterpret_cast<float4*>(out + (long long)k * op) = make_float4(re.hi, re.lo, im.hi, im.lo);
    }
  };
  auto wr2 = [&](int j, hx x0, hx x1) {  // x lines: two adjacent reals
    if (!act) return;
    if constexpr (F64) {
      *reinterpret_cast<double2*>(out + j) = make_double2(cv(x0), cv(x1));
    } else {
      const df t[2] = {cv(x0), cv(x1)};
      *reinterpret_cast<float4*>(out + j) = make_float4(t[0].hi, t[0].lo, t[1].hi, t[1].lo);
    }
  };
  auto wr4 = [&](int j, const hx* x) {  // four adjacent reals
    if (!act) return;
    if constexpr (F64) {
      const double t[4] = {cv(x[0]), cv(x[1]), cv(x[2]), cv(x[3])};
      asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};\n" ::"l"(__cvta_generic_to_global(out + j)), "d"(t[0]), "d"(t[1]),
                   "d"(t[2]), "d"(t[3]) : "memory");
    } else {
      wr2(j, x[0], x[1]);
      wr2(j + 2, x[2], x[3]);
    }
  };
  if constexpr (HG == HG_FWD) {
    const bool r2c = kind == LK_R2C, dst = kind == LK_DST2;
    auto post = [&](int k, bool mid) {
      const hcx Zk = *ln.at(k), Zc = hconj(*ln.at(k == 0 ? 0 : M - k));
      const hcx E = Zk + Zc, d = Zk - Zc;  // 2 E_k, 2i O_k
      const hcx O{d.im, -d.re};
      if (r2c) {
        const hcx P = hmul<false>(O, hld(x1a + k), hld(x1b + k)), Eq = hquarter(E);
        wrc(k, Eq + P);
        if (!mid) wrc(M - k, hconj(Eq - P));
        return;
      }
      const hcx A = hmul<false>(E, hld(x1a + k), hld(x1b + k)), B = hmul<false>(O, hld(x2a + k), hld(x2b + k));
      const hcx W0 = A + B;
      wr(dst ? N - 1 - k : k, W0.re);
      if (k > 0) wr(dst ? k - 1 : N - k, -W0.im);
      if (!mid) {
        const hcx W1 = hrot8<false>(hconj(A - B));
        wr(dst ? N - 1 - (M - k) : M - k, W1.re);
        if (k > 0) wr(dst ? M - k - 1 : M + k, -W1.im);
      }
    };
#pragma unroll 4
    for (int i = 0; i < 8; i++) post(lt + TPL * i, false);
    if (lt == 0) post(M / 2, true);
  } else {
    constexpr int RAD = [] {
      int m = MC;
      while (m > 8) m /= 8;
      return m;
    }();  // last radix: 8, 4 or 2 (powers of two from 64)
    constexpr int NBL = M / RAD, NB = 16 / RAD;
#pragma unroll
    for (int i = 0; i < NB / 2; i++)
#pragma unroll
      for (int t = 0; t < RAD; t++) {
        const int k = lt + TPL * i + NBL * t;          // < M/2 for t < RAD/2
        const hcx e = v[i * RAD + t], m = v[(i + NB / 2) * RAD + RAD - 1 - t];  // z_k, z_{M-1-k}
        if constexpr (C2C) {
          wrc(k, e);
          wrc(M - 1 - k, m);
        } else {
          const int kk = t < RAD / 2 ? k : M - 1 - k;
          hcx z0 = t < RAD / 2 ? e : m, z1 = t < RAD / 2 ? m : e;  // z_kk, z_{M-1-kk}
          if (HG == HG_IV) {
            const bool c4 = kind == LK_DCT4;
            z0 = hmul<false>(z0, hld(x2a + kk), hld(x2b + kk));
            z1 = hmul<false>(z1, hld(x2a + (M - 1 - kk)), hld(x2b + (M - 1 - kk)));
            const hx i0 = c4 ? -z0.im : z0.im, i1 = c4 ? -z1.im : z1.im;
            bool done = false;
            if constexpr (!OY) {
              if (a.vec_ok) {
                wr2(2 * kk, z0.re, i1);
                wr2(N - 2 - 2 * kk, z1.re, i0);
                done = true;
              }
            }
            if (!done) {
              wr(2 * kk, z0.re);
              wr(2 * kk + 1, i1);
              wr(N - 2 - 2 * kk, z1.re);
              wr(N - 1 - 2 * kk, i0);
            }
          } else if (kind == LK_C2R) {
            bool done = false;
            if constexpr (!OY) {
              if (a.vec_ok) {
                wr2(2 * kk, z0.re, z0.im);
                wr2(2 * (M - 1 - kk), z1.re, z1.im);
                done = true;
              }
            }
            if (!done) {
              wr(2 * kk, z0.re);
              wr(2 * kk + 1, z0.im);
              wr(2 * (M - 1 - kk), z1.re);
              wr(2 * (M - 1 - kk) + 1, z1.im);
            }
          } else {
            // u[4k..4k+3] = (z_k.re, s z_{M-1-k}.im, z_k.im, s z_{M-1-k}.re), s = -1 for DST-III
            if (kind == LK_DST3) z1 = hcx{-z1.re, -z1.im};
            bool done = false;
            if constexpr (!OY) {
              if (a.vec_ok) {
                const hx q[4] = {z0.re, z1.im, z0.im, z1.re};
                wr4(4 * kk, q);
                done = true;
              }
            }
            if (!done) {
              wr(4 * kk, z0.re);
              wr(4 * kk + 1, z1.im);
              wr(4 * kk + 2, z0.im);
              wr(4 * kk + 3, z1.re);
            }
          }
        }
      }
  }
}

template <int HG, class SI, class SO, bool OY, int MC>
cudaError_t launch_hlines_k(const LineArgs& a, cudaStream_t st) {
  using H = HShape<OY, MC>;
  auto k = k_hlines<HG, SI, SO, OY, MC>;
  static std::atomic<unsigned long long> attr_done{0};  // as launch_lines_k
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = (dev >= 0 && dev < 64) ? (1ull << dev) : 0ull;
  if (!bit || !(attr_done.load(std::memory_order_acquire) & bit)) {
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)H::smem);
    if (e != cudaSuccess) return e;
    attr_done.fetch_or(bit, std::memory_order_release);
  }
  return launch_pdl(a.pdl, k, (unsigned)a.ntiles, (unsigned)H::T, H::smem, st, a);
}

// One translation unit per length (compiled in parallel).
template <int MC> cudaError_t dispatch_hlines(const LineArgs& a, int oy, cudaStream_t st) {
  const int k = a.kind;
  const bool fwd = k == LK_R2C || k == LK_DCT2 || k == LK_DST2, iv = k == LK_DCT4 || k == LK_DST4;
  if (oy) {
    if (k == LK_C2C_F) return launch_hlines_k<HG_C2CF, float2, float2, true, MC>(a, st);
    if (k == LK_C2C_I) return launch_hlines_k<HG_C2CI, float2, float2, true, MC>(a, st);
    if (iv) return launch_hlines_k<HG_IV, float2, float2, true, MC>(a, st);
    if (fwd) return launch_hlines_k<HG_FWD, float2, float2, true, MC>(a, st);
    return launch_hlines_k<HG_INV, float2, float2, true, MC>(a, st);
  }
  if (fwd) return launch_hlines_k<HG_FWD, double, float2, false, MC>(a, st);
  if (iv) return a.hdir ? launch_hlines_k<HG_IV, float2, double, false, MC>(a, st)
                        : launch_hlines_k<HG_IV, double, float2, false, MC>(a, st);
  return launch_hlines_k<HG_INV, float2, double, false, MC>(a, st);
}

// lines and threads per CTA of length MC (also the host's launch shapes)
template <int MC> void hlines_shape(int oy, int* lpc, int* threads) {
  *lpc = oy ? HShape<true, MC>::NL : HShape<false, MC>::NL;
  *threads = oy ? HShape<true, MC>::T : HShape<false, MC>::T;
}

}  // namespace pp
