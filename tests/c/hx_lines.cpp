// The block-scaled line transforms (csrc/pp_hx.cuh) on the host: the arithmetic, bounds and tables of the library's own
// header around the recipes of csrc/pp_hlines.cuh, one line at a time, against direct sums in long double.
//   hx_lines <family> <M>   prints, per kind, its name, M, the number of lines and the largest relative error.
// Built with the compiler's check of signed overflow, which prints a line to stderr for a sum that leaves 32 bits.
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <string>
#include <vector>

#include "pp_hx.cuh"
using namespace pp;

enum Kind { R2C, C2R, C2CF, C2CI, DCT2, DCT3, DST2, DST3, DCT4, DST4, NKINDS };
static const char* kNames[] = {"r2c", "c2r", "c2c_f", "c2c_i", "dct2", "dct3", "dst2", "dst3", "dct4", "dst4"};
typedef std::vector<double> Vec;
static const long double PI = 3.14159265358979323846264338327950288L;

struct Tw { htwa a; htwb b; };
static Tw tw(long long num, long long den) {  // exp(-2 pi i num / den)
  const long double t = 2.0L * PI * (num % den) / den;
  Tw w;
  hx_twiddle((double)cosl(t), -(double)sinl(t), w.a, w.b);
  return w;
}
struct Tables {
  std::vector<Tw> w, a1, a2;  // w_M^j; pre/post tables
};
static Tables tables(int kind, int N, int M) {
  Tables t;
  for (int j = 0; j < M; j++) t.w.push_back(tw(j, M));
  for (int k = 0; k <= M; k++) {
    if (kind == R2C || kind == C2R) t.a1.push_back(tw(k, N));
    else if (kind >= DCT2 && kind <= DST3) { t.a1.push_back(tw(k, 4LL * N)); t.a2.push_back(tw(5LL * k, 4LL * N)); }
    else if (kind >= DCT4) { t.a1.push_back(tw(4LL * k + 1, 8LL * N)); t.a2.push_back(tw(k, 2LL * N)); }
  }
  return t;
}

template <int RAD, bool INV> static void stage(std::vector<hcx>& x, int S, const Tables& t) {
  const int M = (int)x.size(), NB = M / RAD;
  std::vector<hcx> y(M);
  for (int j = 0; j < NB; j++) {
    hcx a[RAD];
    for (int u = 0; u < RAD; u++) a[u] = x[j + u * NB];
    hdft<RAD, INV>(a);
    const int p = j / S, q = j % S;
    for (int u = 0; u < RAD; u++) {
      hcx v = a[u];
      if (S * RAD < M) {
        const Tw& w = t.w[(size_t)p * S * u % M];
        v = u ? hmul<INV>(v, w.a, w.b) : hquarter(v);
      }
      y[q + S * RAD * p + S * u] = v;
    }
  }
  x = y;
}
static std::vector<int> radices(int M) {
  std::vector<int> r;
  while (M > 1) { r.push_back(M >= 8 ? 8 : M); M /= r.back(); }
  return r;
}
template <bool INV> static void fft(std::vector<hcx>& x, const Tables& t) {
  int S = 1;
  for (int r : radices((int)x.size())) {
    if (r == 8) stage<8, INV>(x, S, t);
    else if (r == 4) stage<4, INV>(x, S, t);
    else stage<2, INV>(x, S, t);
    S *= r;
  }
}
template <bool C> static hcx mul(hcx x, const Tw& w) { return hmul<C>(x, w.a, w.b); }

struct Stats { float mx = 0.0f, l1 = 0.0f; };
static df stat(Stats& s, double v) {
  const df r = df_from_double(v);
  hx_stat(s.mx, s.l1, r.hi);
  return r;
}

// One line; complex values are (re, im) pairs.
static Vec transform(int kind, int N, const Vec& in, const Tables& t) {
  const bool c2c = kind == C2CF || kind == C2CI, inv = kind == C2R || kind == DCT3 || kind == DST3, iv = kind >= DCT4;
  const int M = c2c ? N : N / 2;
  const std::vector<int> rad = radices(M);
  const HScale hs = hx_bounds(iv, inv, c2c, rad.data(), (int)rad.size());
  Stats st;
  std::vector<hcx> z(M);
  auto cv = [&](df v, float S) { return hx_from(v, S); };
  float S;
  Vec out;
  auto done = [&](hx v) { return hx_to_double(v, (int)(__float_as_uint(hx_unscale(hs, S)) >> 23) - 127); };
  if (!inv) {
    std::vector<df> r(2 * M);
    for (int k = 0; k < M; k++) {
      int i0 = 2 * k, i1 = 2 * k + 1;
      if (kind == DCT2 || kind == DST2) {  // Makhoul order
        i0 = k < M / 2 ? 4 * k : 4 * (M - 1 - k) + 3;
        i1 = k < M / 2 ? 4 * k + 2 : 4 * (M - 1 - k) + 1;
      } else if (iv) {
        i0 = kind == DCT4 ? 2 * k : N - 1 - 2 * k;
        i1 = kind == DCT4 ? N - 1 - 2 * k : 2 * k;
      }
      r[2 * k] = stat(st, in[i0]);
      r[2 * k + 1] = stat(st, in[i1]);
    }
    S = hx_scale(hs, st.mx, st.l1);
    for (int k = 0; k < M; k++) {
      z[k] = hcx{cv(r[2 * k], S), cv(r[2 * k + 1], S)};
      if (kind == DST2 && k >= M / 2) z[k] = hcx{-z[k].re, -z[k].im};
      if (iv) z[k] = mul<false>(z[k], t.a1[k]);
    }
  } else {
    struct Item { df y[4]; };
    std::vector<Item> it(M / 2 + 1);
    for (int k = 0; k <= M / 2; k++) {
      double y[4];
      if (kind == C2R) {
        y[0] = in[2 * k];
        y[1] = k ? in[2 * k + 1] : 0.0;
        y[2] = in[2 * (M - k)];  // (k = M/2: the same two values once more)
        y[3] = k ? in[2 * (M - k) + 1] : 0.0;
      } else {
        auto row = [&](int j) { return in[kind == DCT3 ? j : N - 1 - j]; };
        y[0] = row(k);
        y[1] = k ? row(N - k) : 0.0;
        y[2] = row(M - k);
        y[3] = row(M + k);
      }
      for (int c = 0; c < 4; c++) {
        it[k].y[c] = stat(st, y[c]);
      }
    }
    S = hx_scale(hs, st.mx, st.l1);
    for (int k = 0; k <= M / 2; k++) {
      hx y[4];
      for (int c = 0; c < 4; c++) y[c] = cv(it[k].y[c], S);
      const bool c2r = kind == C2R;
      const hcx A = c2r ? hcx{y[0], y[1]} : hcx{y[0], -y[1]};
      const hcx B = c2r ? hcx{y[2], -y[3]} : hrot8<false>(hcx{y[2], y[3]});
      const hcx E = c2r ? hquarter(A + B) : mul<true>(A + B, t.a1[k]);
      const hcx O = mul<true>(A - B, c2r ? t.a1[k] : t.a2[k]);
      z[k] = hcx{E.re - O.im, E.im + O.re};
      if (k != M / 2 && k > 0) z[M - k] = hcx{E.re + O.im, O.re - E.im};
    }
  }
  if (inv || kind == C2CI) fft<true>(z, t);
  else fft<false>(z, t);
  if (c2c) {
    for (const hcx& v : z) { out.push_back(done(v.re)); out.push_back(done(v.im)); }
  } else if (inv) {
    out.resize(N);
    for (int k = 0; k < M; k++) {
      if (kind == C2R) {
        out[2 * k] = done(z[k].re);
        out[2 * k + 1] = done(z[k].im);
      } else if (k < M / 2) {
        hcx z1 = z[M - 1 - k];
        if (kind == DST3) z1 = hcx{-z1.re, -z1.im};
        out[4 * k] = done(z[k].re);
        out[4 * k + 1] = done(z1.im);
        out[4 * k + 2] = done(z[k].im);
        out[4 * k + 3] = done(z1.re);
      }
    }
  } else if (iv) {
    out.resize(N);
    for (int k = 0; k < M; k++) {
      const hcx v = mul<false>(z[k], t.a2[k]);
      out[2 * k] = done(v.re);
      out[N - 1 - 2 * k] = kind == DCT4 ? done(-v.im) : done(v.im);
    }
  } else {
    out.resize(kind == R2C ? N + 2 : N);
    const bool dst = kind == DST2;
    for (int k = 0; k <= M / 2; k++) {
      const bool mid = k == M / 2;
      const hcx Zk = z[k], Zc = hconj(z[k == 0 ? 0 : M - k]);
      const hcx E = Zk + Zc, d = Zk - Zc;
      const hcx O{d.im, -d.re};
      if (kind == R2C) {
        const hcx P = mul<false>(O, t.a1[k]), Eq = hquarter(E);
        const hcx a = Eq + P, b = hconj(Eq - P);
        out[2 * k] = done(a.re);
        out[2 * k + 1] = done(a.im);
        if (!mid) { out[2 * (M - k)] = done(b.re); out[2 * (M - k) + 1] = done(b.im); }
        continue;
      }
      const hcx A = mul<false>(E, t.a1[k]), B = mul<false>(O, t.a2[k]);
      const hcx W0 = A + B;
      out[dst ? N - 1 - k : k] = done(W0.re);
      if (k > 0) out[dst ? k - 1 : N - k] = done(-W0.im);
      if (!mid) {
        const hcx W1 = hrot8<false>(hconj(A - B));
        out[dst ? N - 1 - (M - k) : M - k] = done(W1.re);
        if (k > 0) out[dst ? M - k - 1 : M + k] = done(-W1.im);
      }
    }
  }
  return out;
}

// The same transform as direct sums.
static std::vector<long double> direct(int kind, int N, const Vec& in) {
  static std::vector<long double> ct;
  static int cn = 0;
  if (cn != 4 * N) {  // cos(2 pi j / 4N)
    cn = 4 * N;
    ct.resize(cn);
    for (int j = 0; j < cn; j++) ct[j] = cosl(2.0L * PI * j / cn);
  }
  auto C = [&](long long j) { return ct[(size_t)(((j % cn) + cn) % cn)]; };  // cos(pi j / 2N)
  auto Sn = [&](long long j) { return C(j - N); };                           // sin
  std::vector<int> nz;
  const int len = kind == C2R ? N / 2 + 1 : N;
  const bool cin = kind == C2R || kind == C2CF || kind == C2CI;
  for (int n = 0; n < len; n++)
    if (cin ? (in[2 * n] != 0.0 || in[2 * n + 1] != 0.0) : in[n] != 0.0) nz.push_back(n);
  std::vector<long double> out;
  if (kind == R2C || kind == C2CF || kind == C2CI) {
    const int sg = kind == C2CI ? 1 : -1;
    for (int k = 0; k < (kind == R2C ? N / 2 + 1 : N); k++) {
      long double re = 0, im = 0;
      for (int n : nz) {
        const long double c = C(4LL * n * k), s = sg * Sn(4LL * n * k);
        const long double x = kind == R2C ? in[n] : in[2 * n], y = kind == R2C ? 0.0 : in[2 * n + 1];
        re += x * c - y * s;
        im += x * s + y * c;
      }
      out.push_back(re);
      out.push_back(im);
    }
    return out;
  }
  for (int n = 0; n < N; n++) {
    long double v = 0;
    for (int k : nz) {
      switch (kind) {
        case C2R:
          if (k == 0 || k == N / 2) v += in[2 * k] * C(4LL * n * k);
          else v += 2.0L * (in[2 * k] * C(4LL * n * k) - in[2 * k + 1] * Sn(4LL * n * k));
          break;
        case DCT2: v += in[k] * C((long long)n * (2 * k + 1)); break;
        case DCT3: v += (k ? 2.0L : 1.0L) * in[k] * C((long long)k * (2 * n + 1)); break;
        case DST2: v += in[k] * Sn((long long)(n + 1) * (2 * k + 1)); break;
        case DST3: v += k == N - 1 ? (n % 2 ? -1.0L : 1.0L) * in[k] : 2.0L * in[k] * Sn((long long)(k + 1) * (2 * n + 1)); break;
        case DCT4: v += in[k] * cosl(PI * (2 * n + 1) * (2 * k + 1) / (4.0L * N)); break;
        default: v += in[k] * sinl(PI * (2 * n + 1) * (2 * k + 1) / (4.0L * N)); break;
      }
    }
    out.push_back(v);
  }
  return out;
}

// The inputs of the first stage in double (what transform() does before it).
typedef std::complex<double> cd;
static std::vector<cd> before(int kind, int N, const Vec& in) {
  const bool c2c = kind == C2CF || kind == C2CI;
  const int M = c2c ? N : N / 2;
  auto e = [](double num, double den) { return std::polar(1.0, -2.0 * (double)PI * num / den); };
  std::vector<cd> z(M);
  for (int k = 0; k < M; k++) {
    if (c2c || kind == R2C) z[k] = cd(in[2 * k], in[2 * k + 1]);
    else if (kind == DCT2 || kind == DST2)
      z[k] = (kind == DST2 && k >= M / 2 ? -1.0 : 1.0) *
             (k < M / 2 ? cd(in[4 * k], in[4 * k + 2]) : cd(in[4 * (M - 1 - k) + 3], in[4 * (M - 1 - k) + 1]));
    else if (kind == DCT4) z[k] = cd(in[2 * k], in[N - 1 - 2 * k]) * e(4 * k + 1, 8 * N);
    else if (kind == DST4) z[k] = cd(in[N - 1 - 2 * k], in[2 * k]) * e(4 * k + 1, 8 * N);
  }
  if (kind != C2R && kind != DCT3 && kind != DST3) return z;
  for (int k = 0; k <= M / 2; k++) {
    cd A, B, wE = 1.0, wO;
    if (kind == C2R) {
      A = cd(in[2 * k], in[2 * k + 1]);
      B = cd(in[2 * (M - k)], -in[2 * (M - k) + 1]);
      wO = std::conj(e(k, N));
    } else {
      auto row = [&](int j) { return in[kind == DCT3 ? j : N - 1 - j]; };
      A = cd(row(k), k ? -row(N - k) : 0.0);
      B = cd(row(M - k), row(M + k)) * e(1, 8);
      wE = std::conj(e(k, 4 * N));
      wO = std::conj(e(5 * k, 4 * N));
    }
    const cd E = (A + B) * wE, O = (A - B) * wO, I(0.0, 1.0);
    z[k] = E + I * O;
    if (k > 0 && k < M / 2) z[M - k] = std::conj(E - I * O);
  }
  return z;
}

// Values whose square root of one half a radix-8 butterfly takes: re + im or re - im of the odd half's second and
// fourth results, as functions of a line.
struct Probe { int stage, j, o, sign; };
static void probes(int kind, int N, const Vec& in, const std::vector<Probe>& ps, std::vector<double>& val) {
  std::vector<cd> x = before(kind, N, in), y(x.size());
  const int M = (int)x.size();
  const double sg = (kind == C2CI || kind == C2R || kind == DCT3 || kind == DST3) ? 1.0 : -1.0;
  const cd I(0.0, sg);
  std::vector<cd> w(M);
  for (int j = 0; j < M; j++) w[j] = std::polar(1.0, sg * 2.0 * (double)PI * j / M);
  int S = 1, st = 0;
  for (int R : radices(M)) {
    const int NB = M / R;
    for (size_t i = 0; i < ps.size(); i++)
      if (ps[i].stage == st) {
        const cd* b = &x[ps[i].j];
        const cd u = b[NB] - b[5 * NB], v = b[3 * NB] - b[7 * NB];
        const cd o = ps[i].o == 1 ? u + I * v : u - I * v;
        val[i] = o.real() + ps[i].sign * o.imag();
      }
    bool more = false;
    for (const Probe& p : ps) more |= p.stage > st;
    if (!more) return;
    for (int j = 0; j < NB; j++) {
      const int p = j / S, q = j % S;
      for (int t = 0; t < R; t++) {
        cd a = 0.0;
        for (int u = 0; u < R; u++) a += x[j + u * NB] * w[(M / R) * (u * t % R)];
        y[q + S * R * p + S * t] = a * w[(long long)p * S * t % M];
      }
    }
    x.swap(y);
    S *= R;
    st++;
  }
}

static double error(const Vec& a, const std::vector<long double>& b) {
  long double d = 0, r = 0;
  for (size_t i = 0; i < b.size(); i++) { d += (a[i] - b[i]) * (a[i] - b[i]); r += b[i] * b[i]; }
  const double e = (double)sqrtl(d / (r > 0 ? r : 1));
  return e == e ? e : HUGE_VAL;
}

int main(int argc, char** argv) {
  const std::string fam = argc > 1 ? argv[1] : "random";
  std::mt19937_64 rng(7);
  std::uniform_real_distribution<double> un(-1.0, 1.0);
  const int M = argc > 2 ? atoi(argv[2]) : 64;
  for (int kind = 0; kind < NKINDS; kind++) {
    const bool c2c = kind == C2CF || kind == C2CI;
    const int N = c2c ? M : 2 * M, reals = c2c ? 2 * N : kind == C2R ? N + 2 : N;
    const Tables t = tables(kind, N, M);
    double worst = 0.0;
    int lines = 0;
    auto check = [&](const Vec& v) {
      const double e = error(transform(kind, N, v, t), direct(kind, N, v));
      worst = e > worst ? e : worst;
      lines++;
    };
    Vec v(reals, 0.0);
    auto zero = [&] { std::fill(v.begin(), v.end(), 0.0); };
    auto tidy = [&] { if (kind == C2R) v[1] = v[N + 1] = 0.0; };  // imaginary parts that a real line does not have
    const double mags[] = {1.0, 1.13, 1.27, 1.4, 1.55, 1.7, 1.8, 1.9, 1.99};
    if (fam == "random") {
      for (int r = 0; r < (M > 256 ? 2 : 4); r++) {
        for (double& x : v) x = un(rng);
        tidy();
        check(v);
      }
    } else if (fam == "fours") {
      // four equal cells, +-, on one butterfly of the first stage (complex points j + u M/8)
      for (int r = 0; r < (M > 256 ? 24 : 200); r++) {
        zero();
        const int j = (int)(rng() % (M / 8));
        const double m = mags[rng() % 9];
        for (int c = 0; c < 4; c++) {
          const int k = j + (M / 8) * (int)(rng() % 8);
          const int i = kind >= DCT4 ? ((rng() & 1) ? 2 * k : N - 1 - 2 * k) : 2 * k + (int)(rng() & 1);
          v[i] = (rng() & 1) ? m : -m;
        }
        tidy();
        check(v);
      }
      // and the one found first: u[5N/8-1], u[5N/8], u[7N/8-1], u[7N/8]
      if (!c2c && kind != C2R)
        for (double m : mags) {
          zero();
          v[5 * N / 8 - 1] = v[5 * N / 8] = v[7 * N / 8 - 1] = v[7 * N / 8] = m;
          check(v);
        }
    } else if (fam == "few") {
      // 1 to 96 cells of like magnitude anywhere
      for (int r = 0; r < (M > 256 ? 24 : 120); r++) {
        zero();
        const double m = mags[rng() % 9];
        const int cells = 1 + (int)(rng() % 96);
        for (int c = 0; c < cells; c++) v[rng() % reals] = (rng() & 1) ? m : -m;
        tidy();
        check(v);
      }
    } else if (fam == "aligned") {
      // lines of k cells that add up in one such value: the k that weigh most in it, of equal magnitude and with
      // their signs, in proportion to their weights, or with the larger of every complex value's two parts at m
      std::vector<Probe> ps;
      int st = 0;
      for (int R : radices(M)) {
        if (R == 8)
          for (int r = 0; r < (M > 128 ? 1 : 4); r++)
            for (int o : {1, 3}) ps.push_back(Probe{st, (int)(rng() % (M / 8)), o, (rng() & 1) ? 1 : -1});
        st++;
      }
      std::vector<std::vector<double>> w(ps.size(), std::vector<double>(reals));
      std::vector<double> val(ps.size());
      for (int i = 0; i < reals; i++) {
        zero();
        v[i] = 1.0;
        tidy();
        probes(kind, N, v, ps, val);
        for (size_t p = 0; p < ps.size(); p++) w[p][i] = val[p];
      }
      for (size_t p = 0; p < ps.size(); p++) {
        std::vector<int> by(reals);
        for (int i = 0; i < reals; i++) by[i] = i;
        std::sort(by.begin(), by.end(), [&](int a, int b) { return std::fabs(w[p][a]) > std::fabs(w[p][b]); });
        for (int k : {4, 6, 8, 16, 24, 32, 48, 64, 90}) {
          if (k > reals || (M > 256 && k > 64)) continue;
          for (double m : {1.2, 1.35, 1.5, 1.6, 1.7, 1.8, 1.9}) {
            if (M > 256 && m != 1.35 && m != 1.8) continue;
            zero();
            for (int c = 0; c < k; c++) v[by[c]] = w[p][by[c]] < 0 ? -m : m;
            tidy();
            check(v);
            for (int c = 0; c < k; c++) v[by[c]] = m * w[p][by[c]];
            tidy();
            check(v);
            for (int c = 0; c < k; c++) {
              const int i = by[c], q = kind >= DCT4 ? N - 1 - i : kind == DCT3 || kind == DST3 ? (N - i) % N : kind >= DCT2 ? i ^ 2 : i ^ 1;
              const double h = std::max(std::fabs(w[p][i]), std::fabs(w[p][q]));
              if (h < 1e-9) continue;
              v[i] = m * w[p][i] / h;
              v[q] = m * w[p][q] / h;
            }
            tidy();
            check(v);
          }
        }
      }
    } else if (fam == "modes") {
      // one coefficient (a source of a single wave), or two, at the ends and in the middle
      for (int i : {0, 1, 2, 3, M / 4, M / 2 - 1, M / 2, M / 2 + 1, M - 2, M - 1, M, M + 1, 3 * M / 2 - 1, 3 * M / 2, N - 2, N - 1, reals - 2, reals - 1})
        for (double m : mags) {
          if (i < 0 || i >= reals) continue;
          zero();
          v[i] = m;
          tidy();
          check(v);
          if (i + 1 < reals) {
            v[i + 1] = -m;
            tidy();
            check(v);
          }
        }
    } else if (fam == "huge") {
      // magnitudes whose sum leaves FP32's range while the transform does not
      for (int r = 0; r < 2; r++) {
        for (double& x : v) x = (2.5e39 / reals) * un(rng);
        tidy();
        check(v);
      }
    } else {
      return 2;
    }
    printf("%s %d %d %.3g\n", kNames[kind], M, lines, worst);
  }
  return 0;
}
