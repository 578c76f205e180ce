// Constant-coefficient inverse z = (eps_ref L)^-1 r of the periodic seven-point
// Laplacian L by separable discrete Hartley transforms.  Sec. II.D solves the
// Poisson equation with a Fourier spectral method; at variable permittivity
// this library uses that constant-coefficient inverse as the preconditioner
// of a conjugate-gradient solve of the flux-form equation (eps_ref is a
// reference permittivity of the box, not the vacuum permittivity of
// Sec. II.B).  The discrete Hartley transform H[k] = Re F[k] - Im F[k] of a
// real line is real and is its own inverse up to 1/N; applied along x, y and z
// it diagonalises L with the eigenvalues
// Lambda(k) = -sum_a 2 (1 - cos(2 pi k_a / n_a)).
//
// Line transforms: mixed-radix Stockham FFT (radices 2 to 16, butterflies with
// compile-time roots) of a complex line that packs two real lines
// (z = a + i b); the Hartley transforms of a and b follow from Z[k] and
// Z[N-k]:  H_a[k] = (P[k] + M[N-k]) / 2,  H_b[k] = (M[k] - P[N-k]) / 2 with
// P = Re Z - Im Z and M = Re Z + Im Z.
//
// Lattice passes: a tile of W lines of the pass axis is staged in shared
// memory (W consecutive rows for x; W consecutive x at fixed (z) or (y) for
// the y and z passes, so global accesses are coalesced along x), each warp
// transforms its pairs of lines, and the tile is written back in place.  The
// z pass can apply the symbol and transform again (forward, scale, inverse).
//
// The line and tile functions are __host__ __device__: the tests run them on
// the host with the same index arithmetic as the device solver.
#pragma once
#include <cmath>
#ifndef LBEH_SPEC_HD
#ifdef __CUDACC__
#define LBEH_SPEC_HD __host__ __device__ __forceinline__
#else
#define LBEH_SPEC_HD inline
#endif
#endif

namespace lbeh_spectral {

template <typename T> struct C2 {
  T x, y;
};
template <typename T> LBEH_SPEC_HD C2<T> cadd(C2<T> a, C2<T> b) { return C2<T>{a.x + b.x, a.y + b.y}; }
template <typename T> LBEH_SPEC_HD C2<T> csub(C2<T> a, C2<T> b) { return C2<T>{a.x - b.x, a.y - b.y}; }
template <typename T> LBEH_SPEC_HD C2<T> cmul(C2<T> a, C2<T> b) {
  return C2<T>{a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
template <typename T> LBEH_SPEC_HD C2<T> mul_mi(C2<T> a) { return C2<T>{a.y, -a.x}; }  // a * (-i)
using cf = C2<float>;

constexpr int kMaxStages = 12;
constexpr int kMaxN = 512;

// radices of N (from {8, 4, 2, 3, 5, 7}); returns the count, 0 if N has
// another prime factor or exceeds kMaxN
LBEH_SPEC_HD int factorize(int N, int *rad) {
  if (N < 1 || N > kMaxN) return 0;
  int m = 0, n = N;
  const int order[6] = {8, 4, 2, 3, 5, 7};
  for (int t = 0; t < 6; ++t)
    while (n % order[t] == 0 && m < kMaxStages) {
      rad[m++] = order[t];
      n /= order[t];
    }
  return n == 1 ? m : 0;
}

// cos and sin of 2 pi n / d as constants: the angle's rational remainder past
// the nearest quarter turn (at most pi/4) in a power series
constexpr double series_cs(double x, bool sine) {
  double t = sine ? x : 1.0, sum = t;
  for (int k = 1; k < 12; ++k) {
    t *= -x * x / double(sine ? (2 * k) * (2 * k + 1) : (2 * k - 1) * (2 * k));
    sum += t;
  }
  return sum;
}
constexpr double cos_frac(int n, int d) {
  const int q = (8 * n + d) / (2 * d);  // nearest quarter turn
  const double x = 2.0 * 3.14159265358979323846 * double(4 * n - q * d) / double(4 * d);
  return (q & 3) == 0 ? series_cs(x, false) : (q & 3) == 1 ? -series_cs(x, true)
       : (q & 3) == 2 ? -series_cs(x, false) : series_cs(x, true);
}
constexpr double sin_frac(int n, int d) {
  const int q = (8 * n + d) / (2 * d);
  const double x = 2.0 * 3.14159265358979323846 * double(4 * n - q * d) / double(4 * d);
  return (q & 3) == 0 ? series_cs(x, true) : (q & 3) == 1 ? series_cs(x, false)
       : (q & 3) == 2 ? -series_cs(x, true) : -series_cs(x, false);
}

// Small DFTs in registers (forward, exp(-2 pi i / R) convention).  Odd primes:
// the sums and differences of the mirrored samples times the constant cosines
// and sines.
template <typename T, int R, int J, int K>
LBEH_SPEC_HD void odd_terms(C2<T> &a, C2<T> &b, const C2<T> *t, const C2<T> *d) {
  constexpr T c = T(cos_frac((J * K) % R, R)), s = T(sin_frac((J * K) % R, R));
  a = C2<T>{a.x + c * t[K].x, a.y + c * t[K].y};
  b = C2<T>{b.x + s * d[K].x, b.y + s * d[K].y};
  if constexpr (K < (R - 1) / 2) odd_terms<T, R, J, K + 1>(a, b, t, d);
}
template <typename T, int R, int J> LBEH_SPEC_HD void odd_rows(C2<T> *v, C2<T> v0, const C2<T> *t, const C2<T> *d) {
  C2<T> a = v0, b{T(0), T(0)};
  odd_terms<T, R, J, 1>(a, b, t, d);
  v[J] = cadd(a, mul_mi(b));
  v[R - J] = csub(a, mul_mi(b));
  if constexpr (J < (R - 1) / 2) odd_rows<T, R, J + 1>(v, v0, t, d);
}
template <typename T, int R> struct Dft {
  static_assert(R == 3 || R == 5 || R == 7, "odd primes");
  LBEH_SPEC_HD static void run(C2<T> *v) {
    C2<T> t[(R + 1) / 2], d[(R + 1) / 2];
    const C2<T> v0 = v[0];
#pragma unroll
    for (int k = 1; k <= (R - 1) / 2; ++k) {
      t[k] = cadd(v[k], v[R - k]);
      d[k] = csub(v[k], v[R - k]);
      v[0] = cadd(v[0], t[k]);
    }
    odd_rows<T, R, 1>(v, v0, t, d);
  }
};
template <typename T> struct Dft<T, 2> {
  LBEH_SPEC_HD static void run(C2<T> *v) {
    const C2<T> a = v[0], b = v[1];
    v[0] = cadd(a, b);
    v[1] = csub(a, b);
  }
};
template <typename T> struct Dft<T, 4> {
  LBEH_SPEC_HD static void run(C2<T> *v) {
    const C2<T> s02 = cadd(v[0], v[2]), d02 = csub(v[0], v[2]);
    const C2<T> s13 = cadd(v[1], v[3]), d13 = mul_mi(csub(v[1], v[3]));
    v[0] = cadd(s02, s13);
    v[2] = csub(s02, s13);
    v[1] = cadd(d02, d13);
    v[3] = csub(d02, d13);
  }
};
template <typename T> struct Dft<T, 8> {
  LBEH_SPEC_HD static void run(C2<T> *v) {
    // two radix-4 DFTs of the even and odd samples joined by the eighth roots
    C2<T> e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
    Dft<T, 4>::run(e);
    Dft<T, 4>::run(o);
    const T h = T(0.70710678118654752440);
    const C2<T> t1{h * (o[1].x + o[1].y), h * (o[1].y - o[1].x)};  // o1 * exp(-i pi/4)
    const C2<T> t2 = mul_mi(o[2]);                                 // o2 * exp(-i pi/2)
    const C2<T> t3{h * (o[3].y - o[3].x), -h * (o[3].x + o[3].y)};  // o3 * exp(-3 i pi/4)
    const C2<T> t[4] = {o[0], t1, t2, t3};
    for (int k = 0; k < 4; ++k) {
      v[k] = cadd(e[k], t[k]);
      v[k + 4] = csub(e[k], t[k]);
    }
  }
};

// R = A B: A-point DFTs of the samples B apart, the constant twiddles W_R^(b k), B-point DFTs across them
template <typename T, int A, int B, int I> LBEH_SPEC_HD void const_twiddles(C2<T> (&y)[B][A]) {
  constexpr int b = I / A, k = I % A;
  if constexpr (b * k != 0) {
    constexpr T c = T(cos_frac(b * k, A * B)), s = T(sin_frac(b * k, A * B));
    y[b][k] = cmul(y[b][k], C2<T>{c, -s});
  }
  if constexpr (I + 1 < A * B) const_twiddles<T, A, B, I + 1>(y);
}
template <typename T, int A, int B> struct DftAB {
  LBEH_SPEC_HD static void run(C2<T> *v) {
    C2<T> y[B][A];
#pragma unroll
    for (int b = 0; b < B; ++b) {
#pragma unroll
      for (int a = 0; a < A; ++a) y[b][a] = v[B * a + b];
      Dft<T, A>::run(y[b]);
    }
    const_twiddles<T, A, B, 0>(y);
#pragma unroll
    for (int k = 0; k < A; ++k) {
      C2<T> t[B];
#pragma unroll
      for (int b = 0; b < B; ++b) t[b] = y[b][k];
      Dft<T, B>::run(t);
#pragma unroll
      for (int j = 0; j < B; ++j) v[k + A * j] = t[j];
    }
  }
};
template <typename T> struct Dft<T, 6> : DftAB<T, 2, 3> {};
template <typename T> struct Dft<T, 9> : DftAB<T, 3, 3> {};
template <typename T> struct Dft<T, 10> : DftAB<T, 2, 5> {};
template <typename T> struct Dft<T, 12> : DftAB<T, 4, 3> {};
template <typename T> struct Dft<T, 14> : DftAB<T, 2, 7> {};
template <typename T> struct Dft<T, 15> : DftAB<T, 3, 5> {};
template <typename T> struct Dft<T, 16> : DftAB<T, 4, 4> {};

// the odd primes from a table of their roots (the narrow plans below)
template <typename T, int R> struct DftTable {
  LBEH_SPEC_HD static void run(C2<T> *v, const C2<T> *w) {
    C2<T> o[R];
    for (int a = 0; a < R; ++a) {
      C2<T> s = v[0];
      for (int b = 1; b < R; ++b) s = cadd(s, cmul(v[b], w[(a * b) % R]));
      o[a] = s;
    }
    for (int a = 0; a < R; ++a) v[a] = o[a];
  }
};

// one butterfly j (0 <= j < N/R) of the Stockham stage with radix R after
// sub-transforms of size Ns; w[t] = exp(-2 pi i t / N)
template <typename T, int R>
LBEH_SPEC_HD void stage_bfly_r(const C2<T> *in, C2<T> *out, const C2<T> *w, int N, int Ns, int j) {
  C2<T> v[R];
  const int stride = N / R;
  const int jn = j % Ns;
  const int tstep = N / (Ns * R);  // twiddle index unit of this stage
  v[0] = in[j];
  for (int r = 1; r < R; ++r) v[r] = cmul(in[j + r * stride], w[(jn * r * tstep) % N]);
  Dft<T, R>::run(v);
  const int idx = (j / Ns) * Ns * R + jn;
  for (int a = 0; a < R; ++a) out[idx + a * Ns] = v[a];
}
template <typename T>
LBEH_SPEC_HD void stage_bfly(const C2<T> *in, C2<T> *out, const C2<T> *w, int N, int R, int Ns, int j) {
  switch (R) {
    case 2: stage_bfly_r<T, 2>(in, out, w, N, Ns, j); break;
    case 3: stage_bfly_r<T, 3>(in, out, w, N, Ns, j); break;
    case 4: stage_bfly_r<T, 4>(in, out, w, N, Ns, j); break;
    case 5: stage_bfly_r<T, 5>(in, out, w, N, Ns, j); break;
    case 7: stage_bfly_r<T, 7>(in, out, w, N, Ns, j); break;
    default: stage_bfly_r<T, 8>(in, out, w, N, Ns, j); break;
  }
}

// ---------------------------------------------------------------- line plans
// Precomputed Stockham stages of one line length, so that a butterfly needs
// no integer division: for stage s with radix R after sub-transforms of size
// Ns, butterfly j (0 <= j < N/R) reads in[j + r N/R] and writes
// out[base_j + a Ns]; code[j] packs base_j (low 16 bits) and the offset of its
// R - 1 twiddles in the stage's twiddle table (high 16 bits).  A stage is a
// pass of the line through shared memory, which is what bounds the transform,
// so a wide plan takes as few stages as radices up to 16 allow (two up to
// N = 225 or so), of equal size where there is a choice.  The first stage
// stores R apart: the radix with the fewest bank conflicts goes first.  A
// narrow plan (small boxes, whose results keep their rounding) has radices 8
// while at least 32 butterflies remain per stage, then 4, 2, 3, 5, 7; after
// the twiddles of its stages of radix 3, 5 and 7 come the R roots of unity.
struct LinePlan {
  int n, nst, ncode, ntw;
  int R[kMaxStages], Ns[kMaxStages], nb[kMaxStages], code_off[kMaxStages], tw_off[kMaxStages];
  unsigned inv[kMaxStages];  // 2^32 / nb rounded up (0: nb = 1): line of butterfly e is e inv / 2^32
  unsigned inv_half;         // the same for N/2 + 1
  bool wide;
};

inline bool split_radices(int n, int left, int most, int *rad) {
  if (left == 0) return n == 1;
  for (int r = most; r >= 2; --r) {
    if (r == 11 || r == 13 || n % r) continue;
    rad[left - 1] = r;
    if (split_radices(n / r, left - 1, r, rad)) return true;
  }
  return false;
}
inline int plan_radices(int N, int *rad, bool wide = true) {
  if (N < 2 || N > kMaxN) return 0;
  if (!wide) {
    int m = 0, n = N;
    while (n % 8 == 0 && N / 8 >= 32 && m < kMaxStages) {
      rad[m++] = 8;
      n /= 8;
    }
    const int order[5] = {4, 2, 3, 5, 7};
    for (int t = 0; t < 5; ++t)
      while (n % order[t] == 0 && m < kMaxStages) {
        rad[m++] = order[t];
        n /= order[t];
      }
    return n == 1 ? m : 0;
  }
  for (int m = 1; m <= kMaxStages; ++m)
    for (int most = 2; most <= 16; ++most) {  // the smallest largest radix of m stages
      if (!split_radices(N, m, most, rad)) continue;
      auto conflicts = [](int r) { return r % 16 == 0 ? 16 : r % 8 == 0 ? 8 : r % 4 == 0 ? 4 : r % 2 == 0 ? 2 : 1; };
      int f = 0;
      for (int k = 1; k < m; ++k)
        if (conflicts(rad[k]) < conflicts(rad[f]) || (conflicts(rad[k]) == conflicts(rad[f]) && rad[k] > rad[f])) f = k;
      const int t = rad[f];
      rad[f] = rad[0];
      rad[0] = t;
      return m;
    }
  return 0;
}

// K of a line of N = 32 K points that one warp transforms in registers (0: by
// its plan's stages).  FP64 lines of 96 take their plan of 8 and 12: steps of
// 64 x 64 x 96 2991 us against 3286 with K = 3 in registers, 96^3 4218 / 4970.
inline int reg_fft_k(int N, bool big, bool fp64 = false) {
  const int K = N % 32 == 0 ? N / 32 : 0;
  if (K == 1 || K == 2 || K == 4 || K == 8) return K;
  if (fp64 && K == 3) return 0;
  return big && (K <= 7 || K == 10 || K == 12) ? K : 0;
}

// The form of an FP32 solve.  The large form has wide plans, register lines of
// every K and passes on 16-byte words of cells; the small form has narrow plans
// and K = 1, 2, 4, 8, and fewer registers in its kernel.
//
// Below 2^20 cells, small: solves of such boxes wait for latency and barriers.
// Steps of 48^3 take 248 us in the small form against 267 in the large one, of
// 81^3 413 / 436, of 128 x 128 x 48 417 / 461, of 32 x 32 x 512 364 / 408; 64^3
// 264 / 261 and 84^3 419 / 418 are equal.  Lines of 96 would gain (96^3 473 /
// 417), but the gradients of runs in such boxes, sums of cancelling FP32 terms,
// move by some 1e-5 with any rounding of the solve, and keep theirs.
//
// From there on, large where it has something to offer: only lines of K = 1, 2,
// 4, 8 (the words: 128^3 657 us against 681), a further K (128 x 128 x 384 1908 /
// 1993), three stages saved over all axes (144^3 1141 / 1261), or one of a long
// line (128 x 432 x 128 2227 / 2346; not where rows along x are no whole words).
// Elsewhere its kernel's register passes lose more than the plans save: 128 x
// 128 x 512 takes 2783 us in the large form against 2510 in the small one, 125 x
// 128 x 128 885 / 794, 175^3 2732 / 2620.
constexpr long long kLargeCells = 1LL << 20;
inline bool large_form(int nx, int ny, int nz) {
  if ((long long)nx * ny * nz < kLargeCells) return false;
  int saved = 0, rad[kMaxStages];
  bool plans = false, more = false;
  for (int n : {nx, ny, nz}) {
    if (reg_fft_k(n, false)) continue;
    plans = true;
    if (reg_fft_k(n, true)) {
      more = true;
      continue;
    }
    const int s = plan_radices(n, rad, false) - plan_radices(n, rad, true);
    saved += s;
    more |= s > 0 && n > 343 && nx % 4 == 0;
  }
  return !plans || more || saved >= 3;
}

// host: the plan and its tables in FP64 (converted to the compute type by the caller)
template <class CodeVec, class TwVec> inline bool build_plan(int N, LinePlan &P, CodeVec &code, TwVec &tw, bool wide = true) {
  int rad[kMaxStages];
  const int m = plan_radices(N, rad, wide);
  if (!m) return false;
  P.wide = wide;
  P.n = N;
  P.nst = m;
  code.clear();
  tw.clear();
  auto inverse = [](int n) { return n > 1 ? unsigned((1ull << 32) / unsigned(n)) + 1u : 0u; };
  P.inv_half = inverse(N / 2 + 1);
  const double two_pi = 6.283185307179586476925286766559;
  int Ns = 1;
  for (int s = 0; s < m; ++s) {
    const int R = rad[s], nb = N / R;
    P.R[s] = R;
    P.Ns[s] = Ns;
    P.nb[s] = nb;
    P.inv[s] = inverse(nb);
    P.code_off[s] = (int)code.size();
    P.tw_off[s] = (int)tw.size();
    for (int jn = 0; jn < Ns; ++jn)
      for (int r = 1; r < R; ++r) {
        const double a = -two_pi * double(jn * r) / double(Ns * R);
        tw.push_back({std::cos(a), std::sin(a)});
      }
    if (!wide && (R == 3 || R == 5 || R == 7))
      for (int t = 0; t < R; ++t) {
        const double a = -two_pi * double(t) / double(R);
        tw.push_back({std::cos(a), std::sin(a)});
      }
    for (int j = 0; j < nb; ++j) {
      const int jn = j % Ns;
      const unsigned base = unsigned((j / Ns) * Ns * R + jn);
      code.push_back(base | (unsigned(jn * (R - 1)) << 16));
    }
    Ns *= R;
  }
  P.ncode = (int)code.size();
  P.ntw = (int)tw.size();
  return true;
}

// butterfly j of stage s (tables of this stage: code + code_off, tw + tw_off)
template <typename T, int R, bool TABLE = false>
LBEH_SPEC_HD void plan_bfly_r(const C2<T> *in, C2<T> *out, const C2<T> *tw, int Ns, int nb, int j, unsigned code) {
  C2<T> v[R];
  const unsigned base = code & 0xFFFFu, tb = code >> 16;
#pragma unroll
  for (int r = 0; r < R; ++r) v[r] = in[j + r * nb];
  if (Ns > 1) {
#pragma unroll
    for (int r = 1; r < R; ++r) v[r] = cmul(v[r], tw[tb + r - 1]);
  }
  if constexpr (TABLE) DftTable<T, R>::run(v, tw + Ns * (R - 1));
  else Dft<T, R>::run(v);
#pragma unroll
  for (int a = 0; a < R; ++a) out[base + a * Ns] = v[a];
}
template <bool WIDE, typename T>
LBEH_SPEC_HD void plan_bfly_of(const LinePlan &P, int s, const unsigned *code, const C2<T> *tw, const C2<T> *in,
                               C2<T> *out, int j) {
  const int Ns = P.Ns[s], nb = P.nb[s];
  const unsigned c = code[P.code_off[s] + j];
  const C2<T> *t = tw + P.tw_off[s];
  if constexpr (WIDE) {
    switch (P.R[s]) {
      case 2: plan_bfly_r<T, 2>(in, out, t, Ns, nb, j, c); break;
      case 3: plan_bfly_r<T, 3>(in, out, t, Ns, nb, j, c); break;
      case 4: plan_bfly_r<T, 4>(in, out, t, Ns, nb, j, c); break;
      case 5: plan_bfly_r<T, 5>(in, out, t, Ns, nb, j, c); break;
      case 6: plan_bfly_r<T, 6>(in, out, t, Ns, nb, j, c); break;
      case 7: plan_bfly_r<T, 7>(in, out, t, Ns, nb, j, c); break;
      case 8: plan_bfly_r<T, 8>(in, out, t, Ns, nb, j, c); break;
      case 9: plan_bfly_r<T, 9>(in, out, t, Ns, nb, j, c); break;
      case 10: plan_bfly_r<T, 10>(in, out, t, Ns, nb, j, c); break;
      case 12: plan_bfly_r<T, 12>(in, out, t, Ns, nb, j, c); break;
      case 14: plan_bfly_r<T, 14>(in, out, t, Ns, nb, j, c); break;
      case 15: plan_bfly_r<T, 15>(in, out, t, Ns, nb, j, c); break;
      default: plan_bfly_r<T, 16>(in, out, t, Ns, nb, j, c); break;
    }
  } else {
    switch (P.R[s]) {
      case 2: plan_bfly_r<T, 2>(in, out, t, Ns, nb, j, c); break;
      case 3: plan_bfly_r<T, 3, true>(in, out, t, Ns, nb, j, c); break;
      case 4: plan_bfly_r<T, 4>(in, out, t, Ns, nb, j, c); break;
      case 5: plan_bfly_r<T, 5, true>(in, out, t, Ns, nb, j, c); break;
      case 7: plan_bfly_r<T, 7, true>(in, out, t, Ns, nb, j, c); break;
      default: plan_bfly_r<T, 8>(in, out, t, Ns, nb, j, c); break;
    }
  }
}
template <typename T>
LBEH_SPEC_HD void plan_bfly(const LinePlan &P, int s, const unsigned *code, const C2<T> *tw, const C2<T> *in,
                            C2<T> *out, int j) {
  if (P.wide) plan_bfly_of<true>(P, s, code, tw, in, out, j);
  else plan_bfly_of<false>(P, s, code, tw, in, out, j);
}

// Hartley values at positions k and N-k of the two real lines packed in the
// transformed complex line Z: (H_a[k], H_b[k], H_a[N-k], H_b[N-k])
template <typename T> struct Split {
  T ak, bk, an, bn;
};
template <typename T> LBEH_SPEC_HD Split<T> pair_split(const C2<T> *Z, int N, int k) {
  const int kn = k == 0 ? 0 : N - k;
  const C2<T> zk = Z[k], zn = Z[kn];
  const T Pk = zk.x - zk.y, Mk = zk.x + zk.y, Pn = zn.x - zn.y, Mn = zn.x + zn.y;
  return Split<T>{T(0.5) * (Pk + Mn), T(0.5) * (Mk - Pn), T(0.5) * (Pn + Mk), T(0.5) * (Mn - Pk)};
}

// whole transform of one complex line on the host (reference driver of the
// same stages); returns the buffer holding the result
template <typename T> inline C2<T> *fft_host(C2<T> *b0, C2<T> *b1, int N, const C2<T> *w) {
  int rad[kMaxStages];
  const int m = factorize(N, rad);
  C2<T> *in = b0, *out = b1;
  int Ns = 1;
  for (int s = 0; s < m; ++s) {
    for (int j = 0; j < N / rad[s]; ++j) stage_bfly(in, out, w, N, rad[s], Ns, j);
    Ns *= rad[s];
    C2<T> *t = in;
    in = out;
    out = t;
  }
  return in;
}

// Hartley transform of one real line on the host (imaginary part zero)
inline void dht_host(const float *x, float *h, int N, const cf *w, cf *b0, cf *b1) {
  for (int i = 0; i < N; ++i) b0[i] = cf{x[i], 0.f};
  const cf *Z = fft_host(b0, b1, N, w);
  for (int k = 0; k < N; ++k) h[k] = Z[k].x - Z[k].y;
}

// ---------------------------------------------------------------- tiles
struct Grid3 {
  int nx, ny, nz;
};

// Tiles of W lines along axis A.  A = 0: lines are the rows (y, z), tile t
// holds rows t*W .. t*W+W-1.  A = 1 / 2: lines are the columns at fixed z (A =
// 1) or fixed y (A = 2), tile t holds x = xb*W .. xb*W+W-1 with xb = t % xt.
LBEH_SPEC_HD int line_len(const Grid3 &g, int A) { return A == 0 ? g.nx : (A == 1 ? g.ny : g.nz); }
LBEH_SPEC_HD int tile_count(const Grid3 &g, int A, int W) {
  if (A == 0) return (g.ny * g.nz + W - 1) / W;
  const int xt = (g.nx + W - 1) / W;
  return xt * (A == 1 ? g.nz : g.ny);
}
// global index of element (line l, position p) of tile t; ok = line exists
LBEH_SPEC_HD long long tile_index(const Grid3 &g, int A, int W, int t, int l, int p, bool &ok) {
  if (A == 0) {
    const long long line = (long long)t * W + l;
    ok = line < (long long)g.ny * g.nz;
    return line * g.nx + p;
  }
  const int xt = (g.nx + W - 1) / W;
  const int x = (t % xt) * W + l;
  const int o = t / xt;  // z for A = 1, y for A = 2
  ok = x < g.nx;
  if (A == 1) return ((long long)o * g.ny + p) * g.nx + x;
  return ((long long)p * g.ny + o) * g.nx + x;
}
// wavenumbers (kx, ky) of line l of a z-pass tile (after the x and y passes)
LBEH_SPEC_HD void zline_k(const Grid3 &g, int W, int t, int l, int &kx, int &ky) {
  const int xt = (g.nx + W - 1) / W;
  kx = (t % xt) * W + l;
  ky = t / xt;
}

// scale of the symbol step: 1 / (eps_ref Lambda(k) N_sites), zero mode 0;
// s_a[k] = 2 (1 - cos(2 pi k / n_a))
template <typename T>
LBEH_SPEC_HD T inv_symbol(int kx, int ky, int kz, const T *sx, const T *sy, const T *sz, T inv_eref_n) {
  if (kx == 0 && ky == 0 && kz == 0) return T(0);
  return -inv_eref_n / (sx[kx] + sy[ky] + sz[kz]);
}

}  // namespace lbeh_spectral
