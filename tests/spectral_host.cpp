// Host driver of the spectral transform core (csrc/spectral.cuh) for the
// tests: the line transform, and the five lattice passes of the
// preconditioner with the same tile indexing, pairing of real lines into
// complex lines, Hartley split and symbol scaling as the device solver, run
// tile by tile.
#include <cmath>
#include <vector>

#include "spectral.cuh"
using namespace lbeh_spectral;

template <typename T> static std::vector<C2<T>> roots(int n) {
  std::vector<C2<T>> w(n);
  for (int t = 0; t < n; ++t) {
    const double a = -2.0 * M_PI * t / n;
    w[t] = C2<T>{T(std::cos(a)), T(std::sin(a))};
  }
  return w;
}
template <typename T> static std::vector<T> symb(int n) {
  std::vector<T> c(n);
  for (int k = 0; k < n; ++k) c[k] = T(2.0 * (1.0 - std::cos(2.0 * M_PI * k / n)));
  return c;
}

// the Stockham stages of a line plan (the device solver's transform)
template <typename T>
static C2<T> *fft_plan(C2<T> *b0, C2<T> *b1, const LinePlan &P, const std::vector<unsigned> &code,
                       const std::vector<C2<T>> &tw) {
  C2<T> *in = b0, *out = b1;
  for (int s = 0; s < P.nst; ++s) {
    for (int j = 0; j < P.nb[s]; ++j) plan_bfly(P, s, code.data(), tw.data(), in, out, j);
    C2<T> *t = in;
    in = out;
    out = t;
  }
  return in;
}

template <typename T>
static void pass_host(T *u, const Grid3 &g, int A, int W, const std::vector<C2<T>> &, bool fuse, T inv_n,
                      const T *sx, const T *sy, const T *sz, bool wide = true) {
  const int N = line_len(g, A);
  LinePlan P;
  std::vector<unsigned> code;
  std::vector<C2<double>> twd;
  build_plan(N, P, code, twd, wide);
  std::vector<C2<T>> tw(twd.size());
  for (size_t k = 0; k < twd.size(); ++k) tw[k] = C2<T>{T(twd[k].x), T(twd[k].y)};
  const int pairs = W / 2;
  std::vector<C2<T>> b0(N), b1(N), Z((size_t)pairs * N);
  const int nt = tile_count(g, A, W);
  for (int t = 0; t < nt; ++t) {
    for (int m = 0; m < pairs; ++m) {
      for (int p = 0; p < N; ++p) {
        bool oa, ob;
        const long long ia = tile_index(g, A, W, t, 2 * m, p, oa);
        const long long ib = tile_index(g, A, W, t, 2 * m + 1, p, ob);
        b0[p] = C2<T>{oa ? u[ia] : T(0), ob ? u[ib] : T(0)};
      }
      C2<T> *r = fft_plan(b0.data(), b1.data(), P, code, tw);
      if (fuse) {
        int kxa, kxb, ky;
        zline_k(g, W, t, 2 * m, kxa, ky);
        zline_k(g, W, t, 2 * m + 1, kxb, ky);
        std::vector<C2<T>> zz(N);
        for (int k = 0; k <= N / 2; ++k) {
          const Split<T> s = pair_split(r, N, k);
          const int kn = k == 0 ? 0 : N - k;
          const T sa = kxa < g.nx ? inv_symbol(kxa, ky, k, sx, sy, sz, inv_n) : T(0);
          const T sb = kxb < g.nx ? inv_symbol(kxb, ky, k, sx, sy, sz, inv_n) : T(0);
          const T sa2 = kxa < g.nx ? inv_symbol(kxa, ky, kn, sx, sy, sz, inv_n) : T(0);
          const T sb2 = kxb < g.nx ? inv_symbol(kxb, ky, kn, sx, sy, sz, inv_n) : T(0);
          zz[k] = C2<T>{s.ak * sa, s.bk * sb};
          zz[kn] = C2<T>{s.an * sa2, s.bn * sb2};
        }
        C2<T> *o = r == b0.data() ? b1.data() : b0.data();
        for (int k = 0; k < N; ++k) o[k] = zz[k];
        r = fft_plan(o, r, P, code, tw);
      }
      for (int p = 0; p < N; ++p) Z[(size_t)m * N + p] = r[p];
    }
    for (int m = 0; m < pairs; ++m)
      for (int p = 0; p < N; ++p) {
        const Split<T> s = pair_split(&Z[(size_t)m * N], N, p);
        bool oa, ob;
        const long long ia = tile_index(g, A, W, t, 2 * m, p, oa);
        const long long ib = tile_index(g, A, W, t, 2 * m + 1, p, ob);
        if (oa) u[ia] = s.ak;
        if (ob) u[ib] = s.bk;
      }
  }
}

template <typename T> static int precond(T *u, int nx, int ny, int nz, double eps_ref, int W, bool wide = true) {
  int r[kMaxStages];
  if (!factorize(nx, r) || !factorize(ny, r) || !factorize(nz, r)) return -1;
  Grid3 g{nx, ny, nz};
  auto wx = roots<T>(nx), wy = roots<T>(ny), wz = roots<T>(nz);
  auto cx = symb<T>(nx), cy = symb<T>(ny), cz = symb<T>(nz);
  const T inv = T(1.0 / (eps_ref * double(nx) * ny * nz));
  pass_host<T>(u, g, 0, W, wx, false, T(0), nullptr, nullptr, nullptr, wide);
  pass_host<T>(u, g, 1, W, wy, false, T(0), nullptr, nullptr, nullptr, wide);
  pass_host<T>(u, g, 2, W, wz, true, inv, cx.data(), cy.data(), cz.data(), wide);
  pass_host<T>(u, g, 1, W, wy, false, T(0), nullptr, nullptr, nullptr, wide);
  pass_host<T>(u, g, 0, W, wx, false, T(0), nullptr, nullptr, nullptr, wide);
  return 0;
}

extern "C" int precond_host(float *u, int nx, int ny, int nz, double eps_ref, int W) {
  return precond<float>(u, nx, ny, nz, eps_ref, W);
}
extern "C" int precond_host_f64(double *u, int nx, int ny, int nz, double eps_ref, int W) {
  return precond<double>(u, nx, ny, nz, eps_ref, W);
}

// the same with the plan kind given: the wide plans (FP64, boxes of many cells) or the narrow ones
extern "C" int precond_plan(void *u, int f64, int nx, int ny, int nz, double eps_ref, int W, int wide) {
  return f64 ? precond<double>((double *)u, nx, ny, nz, eps_ref, W, wide)
             : precond<float>((float *)u, nx, ny, nz, eps_ref, W, wide);
}

// stages of a line plan; the radices in order
extern "C" int plan_stages(int N, int wide, int *rad) { return plan_radices(N, rad, wide); }

extern "C" int box_form(int nx, int ny, int nz) { return large_form(nx, ny, nz); }

// one complex line through its plan (interleaved parts)
template <typename T> static int line(const T *in, T *out, int N, bool wide) {
  LinePlan P;
  std::vector<unsigned> code;
  std::vector<C2<double>> twd;
  if (!build_plan(N, P, code, twd, wide)) return -1;
  std::vector<C2<T>> tw(twd.size()), b0(N), b1(N);
  for (size_t k = 0; k < twd.size(); ++k) tw[k] = C2<T>{T(twd[k].x), T(twd[k].y)};
  for (int i = 0; i < N; ++i) b0[i] = C2<T>{in[2 * i], in[2 * i + 1]};
  const C2<T> *Z = fft_plan(b0.data(), b1.data(), P, code, tw);
  for (int i = 0; i < N; ++i) {
    out[2 * i] = Z[i].x;
    out[2 * i + 1] = Z[i].y;
  }
  return 0;
}
extern "C" int plan_line(const double *in, double *out, int N, int wide) { return line<double>(in, out, N, wide); }
extern "C" int plan_line_f32(const float *in, float *out, int N, int wide) { return line<float>(in, out, N, wide); }

// the register DFT of R points (plan butterflies; K points of a line of 32 K)
template <typename T, int R> static int dft(const T *in, T *out) {
  C2<T> v[R];
  for (int i = 0; i < R; ++i) v[i] = C2<T>{in[2 * i], in[2 * i + 1]};
  Dft<T, R>::run(v);
  for (int i = 0; i < R; ++i) {
    out[2 * i] = v[i].x;
    out[2 * i + 1] = v[i].y;
  }
  return 0;
}
template <typename T> static int dft_of(const T *in, T *out, int R) {
  switch (R) {
    case 2: return dft<T, 2>(in, out);
    case 3: return dft<T, 3>(in, out);
    case 4: return dft<T, 4>(in, out);
    case 5: return dft<T, 5>(in, out);
    case 6: return dft<T, 6>(in, out);
    case 7: return dft<T, 7>(in, out);
    case 8: return dft<T, 8>(in, out);
    case 9: return dft<T, 9>(in, out);
    case 10: return dft<T, 10>(in, out);
    case 12: return dft<T, 12>(in, out);
    case 14: return dft<T, 14>(in, out);
    case 15: return dft<T, 15>(in, out);
    case 16: return dft<T, 16>(in, out);
    default: return -1;
  }
}
extern "C" int small_dft(const double *in, double *out, int R) { return dft_of<double>(in, out, R); }
extern "C" int small_dft_f32(const float *in, float *out, int R) { return dft_of<float>(in, out, R); }

extern "C" int dht_line(const float *x, float *h, int N) {
  int rad[kMaxStages];
  if (!factorize(N, rad)) return -1;
  std::vector<cf> w = roots<float>(N), b0(N), b1(N);
  dht_host(x, h, N, w.data(), b0.data(), b1.data());
  return 0;
}

// Hartley transforms of two real lines from one complex transform
extern "C" int dht_pair(const double *a, const double *b, double *ha, double *hb, int N) {
  int rad[kMaxStages];
  if (!factorize(N, rad)) return -1;
  std::vector<C2<double>> w = roots<double>(N), b0(N), b1(N);
  for (int i = 0; i < N; ++i) b0[i] = C2<double>{a[i], b[i]};
  const C2<double> *Z = fft_host(b0.data(), b1.data(), N, w.data());
  for (int k = 0; k < N; ++k) {
    const Split<double> s = pair_split(Z, N, k);
    ha[k] = s.ak;
    hb[k] = s.bk;
  }
  return 0;
}
