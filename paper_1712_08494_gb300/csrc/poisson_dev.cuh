// Device side of the variable-permittivity Poisson solve (Sec. II.B eq.
// electric_potential, II.D): multigrid level descriptors, double-float
// arithmetic, red-black smoothing, transfer operators, the single-block tail
// cycle and the whole defect-correction solve of one system by one team of
// blocks.  Shared by the single-system solver and the batched step.
#pragma once

#include <cmath>
#include <type_traits>

#include "internal.h"
#include "dfloat.cuh"
#include "team_part.h"

namespace lbeh {

// Cells of the largest level of the tail.  A 16^3 level (4096) swept by one
// block is slower than by the whole grid with its barriers, in FP32 too: the
// solve of the 256^3 suspension 3.15 -> 3.55 ms, of the coated 128^3 drop 700
// -> 793 us.
constexpr long long kTailCells = 512;
constexpr size_t kTailSmem = 200 * 1024;
constexpr int kMaxLevels = 16;
constexpr int kNu = 2;  // pre- and post-smoothing sweeps

template <typename T> struct Level {
  int nx = 0, ny = 0, nz = 0;
  long long N = 0;
  int cf[3] = {0, 0, 0};  // coarsened along x, y, z relative to the finer level
  // face coefficients over H_a^2 (powers of four, folded in exactly); zero
  // along an axis coarsened to a single cell
  T *k[3] = {nullptr, nullptr, nullptr};
  T *x = nullptr, *x2 = nullptr, *b = nullptr;
  T *d = nullptr;          // split levels that hold k: 1 / (sum of the six faces)
  const T *eps = nullptr;  // set (finest split level, FP32): faces (eps_i + eps_{i+a})/2 formed from eps, k unused
  bool rb = false;         // red-black colourable: every extent even or one
  bool split = false;      // arrays stored colour by colour (below)
  bool far = false;        // permittivities so large or small that products of faces leave the type's range
  __host__ __device__ Dims dims() const { return Dims{nx, ny, nz, N}; }
};

// Colour-split storage of the levels above the tail: the red cells (x + y + z
// even) of the level in row-major order, then the black ones.  Cells pair up
// along the first axis that is not a single cell (its extent is even), so a
// cell's place is half its row-major index.  A half sweep, which updates one
// colour from the other, then reads and writes whole 16-byte words of
// consecutive cells and only the colours it needs: at 256^3 (FP32) it moves
// 167 MB instead of the 268 MB of interleaved colours, with 14 loads per four
// cells instead of 60: 61 -> 33 us (75% of the copy rate); at 128^3, in the
// L2, 6.6 -> 3.8 us.
template <typename T> __device__ __forceinline__ unsigned cell_at(const Level<T> &L, unsigned i, int color) {
  return L.split ? (color ? unsigned(L.N >> 1) : 0u) + (i >> 1) : i;
}

// face coefficients k_a(i) (p: +a face) and k_a(i-a) (m) of a cell, row-major levels
template <typename T> struct Faces {
  T xp, xm, yp, ym, zp, zm;
};
template <typename T, typename I>
__device__ __forceinline__ Faces<T> faces(const Level<T> &L, I i, I ixm, I iym, I izm) {
  return Faces<T>{L.k[0][i], L.k[0][ixm], L.k[1][i], L.k[1][iym], L.k[2][i], L.k[2][izm]};
}

template <typename T> struct Tail {
  int n = 0;
  Level<T> L[kMaxLevels];
};

__host__ __device__ inline DF df_split(double v) {
  const float h = float(v);
  return DF{h, float(v - double(h))};
}

// Relative residual sqrt(r2 / b2); zero for a vanishing right-hand side and
// NaN when either sum is not finite (a non-finite input must not pass as a
// vanishing right-hand side).
__host__ __device__ inline double rel_res(double r2, double b2) {
  if (!isfinite(r2) || !isfinite(b2)) return r2 + b2 + NAN;
  return b2 > 0.0 ? sqrt(r2 / b2) : 0.0;
}

// Device-side solver state.
struct PDev {
  double mean_q, mean_phi, bnorm2, rnorm2, relres, tol;
  DF mean_q_df, mean_phi_df;
  int iters, max_iter, cond, notconv;
  long long total_iters;
  int have_prev;  // phi_prev holds the solution of the previous step
  int zero;       // right-hand side vanishes: phi = 0
};


// ---------------------------------------------------------------- level operations
template <typename T>
__device__ __forceinline__ void stencil(const Dims &d, const Level<T> &L, long long i, int x, int y, int z,
                                        const T *__restrict__ xv, T &off, T &diag) {
  const long long ixp = site(d, wrapp(x, d.nx), y, z), ixm = site(d, wrapm(x, d.nx), y, z);
  const long long iyp = site(d, x, wrapp(y, d.ny), z), iym = site(d, x, wrapm(y, d.ny), z);
  const long long izp = site(d, x, y, wrapp(z, d.nz)), izm = site(d, x, y, wrapm(z, d.nz));
  const Faces<T> f = faces(L, i, ixm, iym, izm);
  off = (f.xp * xv[ixp] + f.xm * xv[ixm]) + (f.yp * xv[iyp] + f.ym * xv[iym]) + (f.zp * xv[izp] + f.zm * xv[izm]);
  diag = (f.xp + f.xm) + (f.yp + f.ym) + (f.zp + f.zm);
}

// 32-bit cell walks.  Levels hold fewer than 2^31 cells.  A thread visits the
// cells t0, t0 + dt, ... of a row-major range of rows of width w (w = nx for
// every cell of a level, nx/2 for one colour of a red-black level with nx
// even); its position (u, y, z) advances by the stride decomposed once, with
// no per-cell division, and the walk ends when z reaches nz.
struct Walk {
  int u, y, z, du, dy, dz, w, ny;
  __device__ __forceinline__ Walk(long long t0, long long dt, int w_, int ny_) : w(w_), ny(ny_) {
    const unsigned uw = unsigned(w_), uny = unsigned(ny_);
    unsigned r = unsigned(t0) / uw;
    u = int(unsigned(t0) - r * uw);
    y = int(r % uny);
    z = int(r / uny);
    r = unsigned(dt) / uw;
    du = int(unsigned(dt) - r * uw);
    dy = int(r % uny);
    dz = int(r / uny);
  }
  __device__ __forceinline__ void next() {
    u += du;
    int c = u >= w;
    if (c) u -= w;
    y += dy + c;
    c = y >= ny;
    if (c) y -= ny;
    z += dz + c;
  }
};

__device__ __forceinline__ unsigned site32(const Dims &d, int x, int y, int z) {
  return (unsigned(z) * unsigned(d.ny) + unsigned(y)) * unsigned(d.nx) + unsigned(x);
}

// cell (x, y, z) and its six periodic neighbours as 32-bit indices
struct Nbr {
  unsigned i, xp, xm, yp, ym, zp, zm;
};
__device__ __forceinline__ Nbr nbr(const Dims &d, int x, int y, int z) {
  const unsigned nx = unsigned(d.nx), sz = nx * unsigned(d.ny), n = unsigned(d.N);
  Nbr c;
  c.i = site32(d, x, y, z);
  c.xp = x + 1 == d.nx ? c.i - (nx - 1) : c.i + 1;
  c.xm = x == 0 ? c.i + (nx - 1) : c.i - 1;
  c.yp = y + 1 == d.ny ? c.i - (sz - nx) : c.i + nx;
  c.ym = y == 0 ? c.i + (sz - nx) : c.i - nx;
  c.zp = z + 1 == d.nz ? c.i - (n - sz) : c.i + sz;
  c.zm = z == 0 ? c.i + (n - sz) : c.i - sz;
  return c;
}

// the level stencil at a cell given by its neighbour indices: the same
// arithmetic as stencil()
template <typename T>
__device__ __forceinline__ void stencil_n(const Level<T> &L, const Nbr &c, const T *__restrict__ xv, T &off,
                                          T &diag) {
  const Faces<T> f = faces(L, c.i, c.xm, c.ym, c.zm);
  off = (f.xp * xv[c.xp] + f.xm * xv[c.xm]) + (f.yp * xv[c.yp] + f.ym * xv[c.ym]) +
        (f.zp * xv[c.zp] + f.zm * xv[c.zm]);
  diag = (f.xp + f.xm) + (f.yp + f.ym) + (f.zp + f.zm);
}

// Coarse face coefficient along axis AX of coarse cell (X, Y, Z).  Along a
// coarsened axis the flux between the centres of coarse cells X and X + 1
// crosses three fine faces in series: half of the face inside X (fine 2X |
// 2X+1), the shared face (2X+1 | 2X+2) and half of the face inside X + 1
// (2X+2 | 2X+3); their series conductance over the two fine spacings is
// 2 / (1/(2 k_in) + 1/k_shared + 1/(2 k_next)) -- the harmonic weighting that
// keeps a jump of the permittivity inside a coarse cell from passing as the
// arithmetic mean (fewer cycles on the colloid boxes) -- and the doubled
// spacing divides it by four.  Across the face the fine paths are averaged.
// Along an axis that is not coarsened the coarse face is the fine face.  Axis
// indices are compile-time constants, so the small coordinate arrays stay in
// registers.  The series form takes one division instead of four: what bounds
// the coarsening in FP64 is the division (the FP64 rate of the target is two
// operations per cycle and SM), in FP32 its instruction count.  It multiplies
// faces before it divides; boxes whose permittivities are beyond kFarScale
// (`far`) take the sum of reciprocals.
template <typename T> constexpr double kFarScale = 0x1p24;  // FP32: products of two faces of the coarsest level stay normal
template <> constexpr double kFarScale<double> = 0x1p400;
template <typename T> __device__ __forceinline__ T series(T k_in, T k_sh, T k_nx, bool far = false) {
  if (far) return T(0.5) / (T(0.5) / k_in + T(1) / k_sh + T(0.5) / k_nx);
  const T bc = k_sh * k_nx, den = bc + k_in * (T(2) * k_nx + k_sh);
  return den > T(0) ? k_in * (bc / den) : T(0);  // 1/4 of 2 / (1/(2 k_in) + 1/k_sh + 1/(2 k_nx))
}
template <int AX, typename T>
__device__ __forceinline__ T coarse_coef(const Level<T> &F, const Level<T> &C, int X, int Y, int Z) {
  constexpr int B1 = (AX + 1) % 3, B2 = (AX + 2) % 3;
  const Dims f = F.dims();
  const int fn[3] = {f.nx, f.ny, f.nz}, cn[3] = {C.nx, C.ny, C.nz};
  if (cn[AX] == 1) return T(0);  // a single cell carries no coupling
  const int p[3] = {C.cf[0] ? 2 * X : X, C.cf[1] ? 2 * Y : Y, C.cf[2] ? 2 * Z : Z};
  // fine face coefficient along AX at fine cell q (face q | q + AX)
  auto at = [&](const int (&q)[3]) -> unsigned {
    return cell_at(F, site32(f, q[0], q[1], q[2]), (q[0] + q[1] + q[2]) & 1);
  };
  auto kf = [&](const int (&q)[3]) -> T {
    if (F.eps) {
      int r[3] = {q[0], q[1], q[2]};
      r[AX] = r[AX] + 1 == fn[AX] ? 0 : r[AX] + 1;
      return T(0.5) * (F.eps[at(q)] + F.eps[at(r)]);
    }
    return F.k[AX][at(q)];
  };
  T acc = T(0);
  int cnt = 0;
  for (int t1 = 0; t1 <= C.cf[B1]; ++t1)
    for (int t2 = 0; t2 <= C.cf[B2]; ++t2) {
      int q[3] = {p[0], p[1], p[2]};
      q[B1] += t1;
      q[B2] += t2;
      if (C.cf[AX]) {
        const int x0 = q[AX];
        const T k_in = kf(q);
        q[AX] = x0 + 1;
        const T k_sh = kf(q);
        q[AX] = x0 + 2 == fn[AX] ? 0 : x0 + 2;
        const T k_nx = kf(q);
        acc += series(k_in, k_sh, k_nx, F.far);
      } else {
        acc += kf(q);
      }
      ++cnt;
    }
  return cnt == 4 ? acc * T(0.25) : cnt == 2 ? acc * T(0.5) : acc;
}

// The three coarse faces of coarse cell (X, Y, Z) from the row-major eps of a
// finest level coarsened along every axis: the eight cells inside and the two
// planes past them along each axis are 16 loads of two cells (the general form
// takes 72 of one); bound by its instructions (12 series of three faces).
template <typename T>
__device__ __forceinline__ void coarse_faces_from_eps(const T *__restrict__ eps, const Dims &f, int X, int Y, int Z,
                                                      T (&k)[3]) {
  using P = typename std::conditional<sizeof(T) == 4, float2, double2>::type;
  const unsigned nx = unsigned(f.nx), ny = unsigned(f.ny);
  const unsigned x0 = 2u * unsigned(X), x2 = x0 + 2u == nx ? 0u : x0 + 2u;
  unsigned y[4], z[4];
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    y[t] = 2u * unsigned(Y) + unsigned(t);
    if (y[t] >= ny) y[t] -= ny;
    z[t] = 2u * unsigned(Z) + unsigned(t);
    if (z[t] >= unsigned(f.nz)) z[t] -= unsigned(f.nz);
  }
  auto two = [&](unsigned x, unsigned yy, unsigned zz) -> P {
    return *reinterpret_cast<const P *>(eps + (zz * ny + yy) * nx + x);
  };
  auto path = [](T e0, T e1, T e2, T e3) -> T {
    return series(T(0.5) * (e0 + e1), T(0.5) * (e1 + e2), T(0.5) * (e2 + e3));
  };
  P e[2][2];  // [z][y]
  T acc = T(0);
#pragma unroll
  for (int ty = 0; ty < 2; ++ty)
#pragma unroll
    for (int tz = 0; tz < 2; ++tz) {
      e[tz][ty] = two(x0, y[ty], z[tz]);
      const P n = two(x2, y[ty], z[tz]);
      acc += path(e[tz][ty].x, e[tz][ty].y, n.x, n.y);
    }
  k[0] = acc * T(0.25);
  acc = T(0);
#pragma unroll
  for (int tz = 0; tz < 2; ++tz) {
    const P a2 = two(x0, y[2], z[tz]), a3 = two(x0, y[3], z[tz]);
    acc += path(e[tz][0].x, e[tz][1].x, a2.x, a3.x);
    acc += path(e[tz][0].y, e[tz][1].y, a2.y, a3.y);
  }
  k[1] = acc * T(0.25);
  acc = T(0);
  P b2[2], b3[2];
#pragma unroll
  for (int ty = 0; ty < 2; ++ty) {
    b2[ty] = two(x0, y[ty], z[2]);
    b3[ty] = two(x0, y[ty], z[3]);
  }
  // the paths added in this order, as in the first form of the pass: the
  // coated-drop run, whose contacts close or not by rounding, was checked on it
#pragma unroll
  for (int ty = 0; ty < 2; ++ty) acc += path(e[0][ty].x, e[1][ty].x, b2[ty].x, b3[ty].x);
#pragma unroll
  for (int ty = 0; ty < 2; ++ty) acc += path(e[0][ty].y, e[1][ty].y, b2[ty].y, b3[ty].y);
  k[2] = acc * T(0.25);
}

// Cell t (< N/2) of one colour, colour = (x + y + z) & 1.  Red-black levels
// have every extent even or equal to one; cells pair up along the first axis
// of even extent.
__device__ __forceinline__ long long rb_cell(const Dims &d, int color, long long t, int &x, int &y, int &z) {
  if ((d.nx & 1) == 0) {
    const unsigned hx = unsigned(d.nx / 2);
    const unsigned r = unsigned(t) / hx;
    const int xh = int(unsigned(t) - r * hx);
    z = int(r / unsigned(d.ny));
    y = int(r - unsigned(z) * unsigned(d.ny));
    x = 2 * xh + ((y + z + color) & 1);
  } else if ((d.ny & 1) == 0) {  // nx == 1
    const unsigned hy = unsigned(d.ny / 2);
    const unsigned r = unsigned(t) / hy;
    x = 0;
    z = int(r);
    y = 2 * int(unsigned(t) - r * hy) + ((z + color) & 1);
  } else {  // nx == ny == 1
    x = 0;
    y = 0;
    z = 2 * int(t) + (color & 1);
  }
  return site(d, x, y, z);
}

// one colour of a red-black sweep over the thread range t0, t0+dt, ... < N/2 (row-major levels)
template <typename T>
__device__ __forceinline__ void rb_range(const Level<T> &L, int color, long long t0, long long dt) {
  const Dims d = L.dims();
  for (long long t = t0; t < d.N / 2; t += dt) {
    int x, y, z;
    const long long i = rb_cell(d, color, t, x, y, z);
    T off, diag;
    stencil(d, L, i, x, y, z, L.x, off, diag);
    L.x[i] = (off - L.b[i]) / diag;
  }
}

template <typename T>
__device__ __forceinline__ void jacobi_range(const Level<T> &L, T w, long long t0, long long dt) {
  const Dims d = L.dims();
  for (long long i = t0; i < d.N; i += dt) {
    int x, y, z;
    coords(d, i, x, y, z);
    T off, diag;
    stencil(d, L, i, x, y, z, L.x, off, diag);
    L.x2[i] = L.x[i] + w * ((off - L.b[i]) / diag - L.x[i]);
  }
}

// coarse b(I) = mean over children of the fine residual (b - A x), row-major
// levels.  After a red-black sweep that ended with the black colour the
// residual vanishes on black cells (each was just solved exactly for its
// equation), so only the red children are evaluated.
template <typename T>
__device__ __forceinline__ void restrict_range(const Level<T> &F, const Level<T> &C, long long t0, long long dt) {
  const Dims f = F.dims(), c = C.dims();
  for (Walk w(t0, dt, c.nx, c.ny); w.z < c.nz; w.next()) {
    const int X = w.u, Y = w.y, Z = w.z;
    T acc = T(0);
    int cnt = 0;
    for (int tz = 0; tz <= C.cf[2]; ++tz)
      for (int ty = 0; ty <= C.cf[1]; ++ty)
        for (int tx = 0; tx <= C.cf[0]; ++tx) {
          const int x = C.cf[0] ? 2 * X + tx : X, y = C.cf[1] ? 2 * Y + ty : Y, z = C.cf[2] ? 2 * Z + tz : Z;
          ++cnt;
          if (F.rb && ((x + y + z) & 1)) continue;
          const Nbr n = nbr(f, x, y, z);
          T off, diag;
          stencil_n(F, n, F.x, off, diag);
          acc += F.b[n.i] - (off - diag * F.x[n.i]);
        }
    C.b[site32(c, X, Y, Z)] = acc / T(cnt);
  }
}

// trilinear (cell-centred) prolongation and correction x_f += P x_c.  BLACK:
// only the black cells of a red-black level: the sweep that follows starts
// with the red colour, which it forms from the black one alone, so the red
// cells' prolonged values would be overwritten unread.
template <bool BLACK, typename T>
__device__ __forceinline__ void prolong_range(const Level<T> &F, const Level<T> &C, long long t0, long long dt) {
  const Dims f = F.dims(), c = C.dims();
  const int cd[3] = {c.nx, c.ny, c.nz};
  const long long n = BLACK ? f.N / 2 : f.N;
  for (long long t = t0; t < n; t += dt) {
    int x, y, z;
    long long i = t;
    if (BLACK) i = rb_cell(f, 1, t, x, y, z);
    else coords(f, i, x, y, z);
    const int p[3] = {x, y, z};
    int I0[3], I1[3];
    T w0[3], w1[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if (C.cf[a]) {
        const int I = p[a] >> 1;
        I0[a] = I;
        I1[a] = (p[a] & 1) ? (I + 1 == cd[a] ? 0 : I + 1) : (I == 0 ? cd[a] - 1 : I - 1);
        w0[a] = T(0.75);
        w1[a] = T(0.25);
      } else {
        I0[a] = I1[a] = p[a];
        w0[a] = T(1);
        w1[a] = T(0);
      }
    }
    auto xc = [&](int tx, int ty, int tz) -> T {
      const int X = tx ? I1[0] : I0[0], Y = ty ? I1[1] : I0[1], Z = tz ? I1[2] : I0[2];
      return C.x[cell_at(C, site32(c, X, Y, Z), (X + Y + Z) & 1)];
    };
    T &xf = F.x[cell_at(F, unsigned(i), (x + y + z) & 1)];
    if (C.cf[0] && C.cf[1] && C.cf[2]) {  // weights 27/64, 9/64, 3/64, 1/64; one by one, as the general form adds them
      T acc = T(0.421875) * xc(0, 0, 0);
      acc += T(0.140625) * xc(1, 0, 0);
      acc += T(0.140625) * xc(0, 1, 0);
      acc += T(0.046875) * xc(1, 1, 0);
      acc += T(0.140625) * xc(0, 0, 1);
      acc += T(0.046875) * xc(1, 0, 1);
      acc += T(0.046875) * xc(0, 1, 1);
      acc += T(0.015625) * xc(1, 1, 1);
      xf += acc;
      continue;
    }
    T acc = T(0);
#pragma unroll
    for (int tz = 0; tz < 2; ++tz)
#pragma unroll
      for (int ty = 0; ty < 2; ++ty)
#pragma unroll
        for (int tx = 0; tx < 2; ++tx) {
          const T w = (tx ? w1[0] : w0[0]) * (ty ? w1[1] : w0[1]) * (tz ? w1[2] : w0[2]);
          if (w == T(0)) continue;
          acc += w * xc(tx, ty, tz);
        }
    xf += acc;
  }
}

// ---------------------------------------------------------------- single-block tail
// Sweeps of one tail level held in shared memory.  A red-black level of at
// most 512 cells has one cell of each colour per thread: the thread keeps
// both cells' neighbour indices and 1/diag, so a half sweep is its loads and
// seven multiply-adds, and a level of at most 64 cells is one warp's work
// (the others wait at the closing barrier).  `zero`: the sweeps start from
// x = 0, the first red half sweep reads no neighbour.
template <typename T> __device__ void tail_smooth(const Level<T> &L, int sweeps, bool zero) {
  const Dims d = L.dims();
  const int half = int(d.N / 2);
  if (L.rb && half <= int(blockDim.x)) {
    const bool one_warp = half <= 32;
    const int t = threadIdx.x;
    if (!one_warp || t < 32) {
      const bool on = t < half;
      Nbr n[2] = {};
      T g[2] = {T(0), T(0)}, rhs[2] = {T(0), T(0)};
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        if (!on) continue;
        int x, y, z;
        rb_cell(d, c, t, x, y, z);
        n[c] = nbr(d, x, y, z);
        g[c] = L.d[n[c].i];
        rhs[c] = L.b[n[c].i];
      }
      for (int s = 0; s < sweeps; ++s)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          if (on) {
            const Nbr &m = n[c];
            T off = T(0);
            if (!(zero && s == 0 && c == 0))
              off = (L.k[0][m.i] * L.x[m.xp] + L.k[0][m.xm] * L.x[m.xm]) +
                    (L.k[1][m.i] * L.x[m.yp] + L.k[1][m.ym] * L.x[m.ym]) +
                    (L.k[2][m.i] * L.x[m.zp] + L.k[2][m.zm] * L.x[m.zm]);
            L.x[m.i] = (off - rhs[c]) * g[c];
            // along an axis of one cell a cell is its own neighbour, with a
            // zero coefficient: it must hold a number before it is read
            if (zero && s == 0 && c == 0) L.x[n[1].i] = T(0);
          }
          if (one_warp) __syncwarp();
          else __syncthreads();
        }
    }
    if (one_warp) __syncthreads();
    return;
  }
  if (zero) {
    for (long long i = threadIdx.x; i < d.N; i += blockDim.x) L.x[i] = T(0);
    __syncthreads();
  }
  for (int s = 0; s < sweeps; ++s) {
    if (L.rb) {
      rb_range(L, 0, threadIdx.x, blockDim.x);
      __syncthreads();
      rb_range(L, 1, threadIdx.x, blockDim.x);
      __syncthreads();
    } else {
      jacobi_range(L, T(0.8), threadIdx.x, blockDim.x);
      __syncthreads();
      for (long long i = threadIdx.x; i < L.N; i += blockDim.x) L.x[i] = L.x2[i];
      __syncthreads();
    }
  }
}

// Shared-memory bytes of the tail levels first..n-1: three face arrays, x, b
// and 1/diag (red-black levels) or x2 (an odd axis).
template <typename T> __host__ __device__ inline size_t tail_bytes(const Tail<T> &tl, int first) {
  size_t b = 0;
  for (int l = first; l < tl.n; ++l) b += size_t(6) * tl.L[l].N * sizeof(T);
  return b;
}

// V-cycle over levels first..n-1 of lv inside one block, every level held in
// shared memory (descriptors included): face coefficients and the right-hand
// side of level `first` are loaded, its correction x is written back.  What
// bounds it is the chain of dependent half sweeps (and in FP64 the rate of
// the one SM it runs on); see tail_smooth.
template <typename T>
__device__ void tail_vcycle(const Level<T> *__restrict__ lv, int n, int first, unsigned char *smem_raw) {
  __shared__ Level<T> sl[kMaxLevels];
  if (threadIdx.x == 0) {
    T *p = reinterpret_cast<T *>(smem_raw);
    for (int l = first; l < n; ++l) {
      Level<T> L = lv[l];
      const long long m = L.N;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        L.k[a] = p;
        p += m;
      }
      L.x = p;
      p += m;
      L.b = p;
      p += m;
      L.d = L.x2 = p;  // 1/diag (red-black levels), x2 (the others)
      p += m;
      L.eps = nullptr;
      sl[l] = L;
    }
  }
  __syncthreads();
  for (int l = first; l < n; ++l) {
    const Level<T> G = lv[l];
    const Level<T> S = sl[l];
    for (int i = threadIdx.x; i < int(G.N); i += blockDim.x) {
#pragma unroll
      for (int a = 0; a < 3; ++a) S.k[a][i] = G.k[a][i];
      if (l == first) S.b[i] = G.b[i];
      if (G.d) S.d[i] = G.d[i];
    }
  }
  __syncthreads();
  for (int l = first; l < n; ++l) {
    const Level<T> S = sl[l];
    if (!S.rb || lv[l].d) continue;
    const Dims d = S.dims();
    for (Walk w(threadIdx.x, blockDim.x, d.nx, d.ny); w.z < d.nz; w.next()) {
      const Nbr c = nbr(d, w.u, w.y, w.z);
      const Faces<T> f = faces(S, c.i, c.xm, c.ym, c.zm);
      S.d[c.i] = T(1) / ((f.xp + f.xm) + (f.yp + f.ym) + (f.zp + f.zm));
    }
  }
  __syncthreads();
  for (int l = first; l < n; ++l) {
    const Level<T> L = sl[l];
    if (l == n - 1) {
      // coarsest: mean-free right-hand side (one warp adds its few cells), fixed relaxation count
      if (threadIdx.x < 32) {
        T acc = T(0);
        for (long long i = threadIdx.x; i < L.N; i += 32) acc += L.b[i];
        for (int w = 16; w > 0; w >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, w);
        const T mean = acc / T(L.N);
        for (long long i = threadIdx.x; i < L.N; i += 32) L.b[i] -= mean;
      }
      __syncthreads();
      tail_smooth(L, L.rb ? 4 : 30, true);
    } else {
      tail_smooth(L, kNu, true);
      const Level<T> Lc = sl[l + 1];
      restrict_range(L, Lc, threadIdx.x, blockDim.x);
      __syncthreads();
    }
  }
  for (int l = n - 2; l >= first; --l) {
    const Level<T> Lf = sl[l], Lc = sl[l + 1];
    if (Lf.rb) prolong_range<true>(Lf, Lc, threadIdx.x, blockDim.x);
    else prolong_range<false>(Lf, Lc, threadIdx.x, blockDim.x);
    __syncthreads();
    tail_smooth(Lf, kNu, false);
  }
  {
    const Level<T> G = lv[first], S = sl[first];
    for (long long i = threadIdx.x; i < G.N; i += blockDim.x) G.x[i] = S.x[i];
  }
}

// ---------------------------------------------------------------- split levels
// Passes of the levels above the tail, on colour-split arrays.  A thread works
// on V consecutive cells of one colour of a row (V words fill 16 bytes; V = 1
// where a half row is not a multiple of V cells).
template <typename T, int V> struct alignas(sizeof(T) * V) Vec {
  T v[V];
};
template <int V, typename T> __device__ __forceinline__ Vec<T, V> ldv(const T *p) {
  return *reinterpret_cast<const Vec<T, V> *>(p);
}
template <int V, typename T> __device__ __forceinline__ void stv(T *p, const Vec<T, V> &v) {
  *reinterpret_cast<Vec<T, V> *>(p) = v;
}

// Rows of a split level: cells pair up along the first axis that is not a
// single cell, which takes the place of x (the axes of one cell in front of
// it move to the back; their coefficients are zero).
template <typename T> struct Rows {
  int hx, ny, nz;           // cells of one colour in a row, rows of a plane, planes
  int axis;                 // the axis of the rows
  const T *kx, *ky, *kz;    // faces along the row, the plane and the box direction
};
template <typename T> __device__ __forceinline__ Rows<T> rows_of(const Level<T> &L) {
  if (L.nx > 1) return Rows<T>{L.nx >> 1, L.ny, L.nz, 0, L.k[0], L.k[1], L.k[2]};
  if (L.ny > 1) return Rows<T>{L.ny >> 1, L.nz, 1, 1, L.k[1], L.k[2], L.k[0]};
  return Rows<T>{L.nz >> 1, 1, 1, 2, L.k[2], L.k[0], L.k[1]};
}
template <typename T> __device__ __forceinline__ bool wide(const Level<T> &L) {
  return (rows_of(L).hx % int(16 / sizeof(T))) == 0;
}

// The V cells at (row offset `row` of (y, z), place j) of colour c and their
// neighbours, all of the other colour: those along y and z at the same place
// j, one of those along the row at j and the other at j + 1 or j - 1,
// depending on the parity of the cells' first coordinate.
struct Site {
  unsigned i, yp, ym, zp, zm, e;  // e: the place past the V along the row
  int p;                          // 1: the cells sit at odd coordinates (e follows), 0: at even ones (e precedes)
};
template <int V, typename T> __device__ __forceinline__ Site split_site(const Rows<T> &r, int c, int j, int y, int z) {
  const unsigned hx = unsigned(r.hx), sz = hx * unsigned(r.ny);
  const unsigned row = unsigned(z) * sz + unsigned(y) * hx;
  Site s;
  s.i = row + unsigned(j);
  s.yp = y + 1 == r.ny ? s.i - unsigned(y) * hx : s.i + hx;
  s.ym = y == 0 ? s.i + unsigned(r.ny - 1) * hx : s.i - hx;
  s.zp = z + 1 == r.nz ? s.i - unsigned(z) * sz : s.i + sz;
  s.zm = z == 0 ? s.i + unsigned(r.nz - 1) * sz : s.i - sz;
  s.p = (y + z + c) & 1;
  s.e = row + unsigned(s.p ? (j + V == r.hx ? 0 : j + V) : (j == 0 ? r.hx - 1 : j - 1));
  return s;
}
// the values before (xm) and after (xp) each of the V cells, from the other
// colour's values m at the same places and the one past them
template <typename T, int V>
__device__ __forceinline__ void along_row(const Vec<T, V> &m, T e, int p, Vec<T, V> &xp, Vec<T, V> &xm) {
#pragma unroll
  for (int v = 0; v < V; ++v) {
    const T next = v + 1 < V ? m.v[v + 1 < V ? v + 1 : v] : e, prev = v > 0 ? m.v[v > 0 ? v - 1 : 0] : e;
    xp.v[v] = p ? next : m.v[v];
    xm.v[v] = p ? m.v[v] : prev;
  }
}

// six face coefficients of the V cells of colour c at a site
template <typename T, int V> struct FaceV {
  Vec<T, V> xp, xm, yp, ym, zp, zm;
};
template <bool EPS, int V, typename T>
__device__ __forceinline__ FaceV<T, V> faces_v(const Level<T> &L, const Rows<T> &r, const Site &s, int c) {
  const unsigned half = unsigned(L.N >> 1), co = c ? half : 0u, oo = c ? 0u : half;
  FaceV<T, V> f;
  if constexpr (EPS) {
    const T *ec = L.eps + co, *eo = L.eps + oo;
    const Vec<T, V> own = ldv<V>(ec + s.i);
    along_row<T, V>(ldv<V>(eo + s.i), eo[s.e], s.p, f.xp, f.xm);
    f.yp = ldv<V>(eo + s.yp);
    f.ym = ldv<V>(eo + s.ym);
    f.zp = ldv<V>(eo + s.zp);
    f.zm = ldv<V>(eo + s.zm);
#pragma unroll
    for (int v = 0; v < V; ++v) {
      f.xp.v[v] = T(0.5) * (own.v[v] + f.xp.v[v]);
      f.xm.v[v] = T(0.5) * (f.xm.v[v] + own.v[v]);
      f.yp.v[v] = T(0.5) * (own.v[v] + f.yp.v[v]);
      f.ym.v[v] = T(0.5) * (f.ym.v[v] + own.v[v]);
      f.zp.v[v] = T(0.5) * (own.v[v] + f.zp.v[v]);
      f.zm.v[v] = T(0.5) * (f.zm.v[v] + own.v[v]);
    }
  } else {
    const T *kx = r.kx, *ky = r.ky, *kz = r.kz;
    f.xp = ldv<V>(kx + co + s.i);
    f.yp = ldv<V>(ky + co + s.i);
    f.zp = ldv<V>(kz + co + s.i);
    Vec<T, V> unused;
    along_row<T, V>(ldv<V>(kx + oo + s.i), s.p ? T(0) : kx[oo + s.e], s.p, unused, f.xm);
    f.ym = ldv<V>(ky + oo + s.ym);
    f.zm = ldv<V>(kz + oo + s.zm);
  }
  return f;
}
// sum of face times neighbour over the six neighbours
template <int V, typename T>
__device__ __forceinline__ Vec<T, V> off_v(const Level<T> &L, const FaceV<T, V> &f, const Site &s, int c) {
  const T *xo = L.x + (c ? 0u : unsigned(L.N >> 1));
  Vec<T, V> xp, xm, o;
  along_row<T, V>(ldv<V>(xo + s.i), xo[s.e], s.p, xp, xm);
  const Vec<T, V> yp = ldv<V>(xo + s.yp), ym = ldv<V>(xo + s.ym), zp = ldv<V>(xo + s.zp), zm = ldv<V>(xo + s.zm);
#pragma unroll
  for (int v = 0; v < V; ++v)
    o.v[v] = (f.xp.v[v] * xp.v[v] + f.xm.v[v] * xm.v[v]) + (f.yp.v[v] * yp.v[v] + f.ym.v[v] * ym.v[v]) +
             (f.zp.v[v] * zp.v[v] + f.zm.v[v] * zm.v[v]);
  return o;
}
template <int V, typename T> __device__ __forceinline__ T diag_v(const FaceV<T, V> &f, int v) {
  return (f.xp.v[v] + f.xm.v[v]) + (f.yp.v[v] + f.ym.v[v]) + (f.zp.v[v] + f.zm.v[v]);
}

// The thread's share of n work items: items t0, t0 + dt, ...  The passes over
// n items go over the blocks in equal contiguous chunks of whole warps, so
// that a level with fewer items than the team has threads still keeps every
// SM busy (512 items to a block left 120 of 152 SMs idle at 32^3, where the
// FP64 arithmetic of one SM is what bounds a pass).
struct Share {
  long long t0, dt;
};
template <class Team> __device__ __forceinline__ Share share(const Team &tm, unsigned n) {
  const unsigned nb = unsigned(tm.nblocks()), team = nb * blockDim.x;
  const unsigned turns = (n + team - 1u) / team;
  const unsigned per = nb * (turns ? turns : 1u);
  const unsigned chunk = min((((n + per - 1u) / per) + 31u) & ~31u, blockDim.x);
  return Share{threadIdx.x < chunk ? (long long)(unsigned(tm.block()) * chunk + threadIdx.x) : (long long)n,
               (long long)nb * chunk};
}

// One half sweep of colour c: x = (sum of face times neighbour - b) / diag.
// ZERO: from x = 0.  EPS: the faces are formed from eps (FP32, finest level;
// one array instead of four), else they and 1/diag are stored.
template <bool EPS, bool ZERO, int V, typename T, class Team>
__device__ __forceinline__ void half_sweep(const Level<T> &L, int c, const Team &tm) {
  const Rows<T> r = rows_of(L);
  const unsigned half = unsigned(L.N >> 1), co = c ? half : 0u;
  const Share sh = share(tm, half / V);
  for (Walk w(sh.t0, sh.dt, r.hx / V, r.ny); w.z < r.nz; w.next()) {
    const Site s = split_site<V>(r, c, w.u * V, w.y, w.z);
    const Vec<T, V> b = ldv<V>(L.b + co + s.i);
    Vec<T, V> o;
    if constexpr (EPS) {
      const FaceV<T, V> f = faces_v<true, V>(L, r, s, c);
      if constexpr (ZERO) {
#pragma unroll
        for (int v = 0; v < V; ++v) o.v[v] = -b.v[v] / diag_v(f, v);
      } else {
        o = off_v<V>(L, f, s, c);
#pragma unroll
        for (int v = 0; v < V; ++v) o.v[v] = (o.v[v] - b.v[v]) / diag_v(f, v);
      }
    } else {
      const Vec<T, V> g = ldv<V>(L.d + co + s.i);
      if constexpr (ZERO) {
#pragma unroll
        for (int v = 0; v < V; ++v) o.v[v] = -b.v[v] * g.v[v];
      } else {
        o = off_v<V>(L, faces_v<false, V>(L, r, s, c), s, c);
#pragma unroll
        for (int v = 0; v < V; ++v) o.v[v] = (o.v[v] - b.v[v]) * g.v[v];
      }
    }
    stv<V>(L.x + co + s.i, o);
  }
}
template <bool ZERO, typename T, class Team>
__device__ __forceinline__ void sweep_colour(const Level<T> &L, int c, const Team &tm) {
  constexpr int V = 16 / sizeof(T);
  if (L.eps) {
    if (wide(L)) half_sweep<true, ZERO, V>(L, c, tm);
    else half_sweep<true, ZERO, 1>(L, c, tm);
  } else {
    if (wide(L)) half_sweep<false, ZERO, V>(L, c, tm);
    else half_sweep<false, ZERO, 1>(L, c, tm);
  }
}

// 1 / diag of a level that stores its faces
template <typename T, class Team> __device__ __forceinline__ void inverse_diag(const Level<T> &L, const Team &tm) {
  const Dims d = L.dims();
  const Share sh = share(tm, unsigned(L.N));
  for (Walk w(sh.t0, sh.dt, d.nx, d.ny); w.z < d.nz; w.next()) {
    const Nbr c = nbr(d, w.u, w.y, w.z);
    const int color = (w.u + w.y + w.z) & 1;
    const unsigned i = cell_at(L, c.i, color);
    // along an axis of one cell the faces are zero wherever they are read
    const Faces<T> f = faces(L, i, cell_at(L, c.xm, color ^ 1), cell_at(L, c.ym, color ^ 1), cell_at(L, c.zm, color ^ 1));
    L.d[i] = T(1) / ((f.xp + f.xm) + (f.yp + f.ym) + (f.zp + f.zm));
  }
}

// restrict_range on a split fine level.  Along the fine row each pair of
// children has one red cell, so the red children of V coarse cells are V
// consecutive red cells of each of the two or four child rows.  The first
// half sweep on the coarse level starts from x = 0, which sets its red cells
// to -b / diag: that is done here (split coarse levels; the tail starts its
// own sweeps).
template <bool EPS, int V, typename T, class Team>
__device__ __forceinline__ void restrict_split(const Level<T> &F, const Level<T> &C, const Team &tm) {
  const Rows<T> r = rows_of(F);
  const Share sh = share(tm, unsigned(C.N) / V);
  for (Walk w(sh.t0, sh.dt, C.nx / V, C.ny); w.z < C.nz; w.next()) {
    const int X = w.u * V, Y = w.y, Z = w.z;
    Vec<T, V> acc{};
    // child rows: (y, z) of the fine level, or their counterparts when the
    // fine level's row runs along another axis
    const bool xrow = r.axis == 0;
    const int ry = xrow ? Y : r.axis == 1 ? Z : 0, rz = xrow ? Z : 0, j = xrow ? X : r.axis == 1 ? Y : Z;
    const int ny = xrow ? C.cf[1] : r.axis == 1 ? C.cf[2] : 0, nz = xrow ? C.cf[2] : 0;
    auto child_row = [&](int ty, int tz) {
      const Site s = split_site<V>(r, 0, j, ny ? 2 * ry + ty : ry, nz ? 2 * rz + tz : rz);
      const FaceV<T, V> f = faces_v<EPS, V>(F, r, s, 0);
      const Vec<T, V> o = off_v<V>(F, f, s, 0), x = ldv<V>(F.x + s.i), b = ldv<V>(F.b + s.i);
#pragma unroll
      for (int v = 0; v < V; ++v) acc.v[v] += b.v[v] - (o.v[v] - diag_v(f, v) * x.v[v]);
    };
    if (V == 1 && ny && nz) {  // the loads of the four child rows in flight together
      child_row(0, 0);
      child_row(1, 0);
      child_row(0, 1);
      child_row(1, 1);
    } else {
      for (int tz = 0; tz <= nz; ++tz)
        for (int ty = 0; ty <= ny; ++ty) child_row(ty, tz);
    }
    const T mean = T(1) / T(2 * (1 + ny) * (1 + nz));  // one eighth, a quarter or a half
    const unsigned I = (unsigned(Z) * unsigned(C.ny) + unsigned(Y)) * unsigned(C.nx) + unsigned(X);
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const int color = (X + v + Y + Z) & 1;
      const unsigned at = cell_at(C, I + v, color);
      const T bI = acc.v[v] * mean;
      C.b[at] = bI;
      if (C.split && !color) C.x[at] = -bI * C.d[at];
    }
  }
}
template <typename T, class Team>
__device__ __forceinline__ void restrict_to(const Level<T> &F, const Level<T> &C, const Team &tm) {
  constexpr int V = 16 / sizeof(T);
  // rows of a multiple of V coarse cells, and more cells than threads: below
  // that, one cell per thread over more SMs hides the latency of its child
  // rows better (6.4 us with V = 2 against 3.6 at 32^3 in FP64)
  const bool w = F.nx > 1 && wide(F) && C.N > tm.size();
  if (F.eps) {
    if (w) restrict_split<true, V>(F, C, tm);
    else restrict_split<true, 1>(F, C, tm);
  } else {
    if (w) restrict_split<false, V>(F, C, tm);
    else restrict_split<false, 1>(F, C, tm);
  }
}

// prolong_range<true> on a split fine level, coarsened along every axis:
// weights 27/64, 9/64, 3/64, 1/64; V consecutive black cells of a row take
// V + 1 consecutive coarse cells of each of four coarse rows.
template <int V, typename T, class Team>
__device__ __forceinline__ void prolong_black(const Level<T> &F, const Level<T> &C, const Team &tm) {
  const Rows<T> r = rows_of(F);
  const unsigned half = unsigned(F.N >> 1), cnx = unsigned(C.nx), cny = unsigned(C.ny);
  const Share sh = share(tm, half / V);
  for (Walk w(sh.t0, sh.dt, r.hx / V, r.ny); w.z < r.nz; w.next()) {
    const int y = w.y, z = w.z, j = w.u * V;
    const int p = (y + z + 1) & 1;
    const int Y0 = y >> 1, Z0 = z >> 1;
    const int Y1 = (y & 1) ? (Y0 + 1 == C.ny ? 0 : Y0 + 1) : (Y0 == 0 ? C.ny - 1 : Y0 - 1);
    const int Z1 = (z & 1) ? (Z0 + 1 == C.nz ? 0 : Z0 + 1) : (Z0 == 0 ? C.nz - 1 : Z0 - 1);
    // near (X0 = j + v) and far (X1) coarse cells of the coarse rows (Y0, Z0), (Y1, Z0), (Y0, Z1), (Y1, Z1)
    const int Xe = p ? (j + V == C.nx ? 0 : j + V) : (j == 0 ? C.nx - 1 : j - 1);
    T n[4][V], f[4][V];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int Y = (k & 1) ? Y1 : Y0, Z = (k & 2) ? Z1 : Z0;
      const unsigned row = (unsigned(Z) * cny + unsigned(Y)) * cnx;
      const T e = C.x[cell_at(C, row + unsigned(Xe), (Xe + Y + Z) & 1)];
      if constexpr (V == 1) {
        n[k][0] = C.x[cell_at(C, row + unsigned(j), (j + Y + Z) & 1)];
      } else if (C.split) {  // j is even: the V cells are V / 2 of each colour
        const unsigned hc = unsigned(C.N >> 1), at = (row + unsigned(j)) >> 1;
        const int q = (Y + Z) & 1;
        const Vec<T, V / 2> ev = ldv<V / 2>(C.x + (q ? hc : 0u) + at), od = ldv<V / 2>(C.x + (q ? 0u : hc) + at);
#pragma unroll
        for (int v = 0; v < V; ++v) n[k][v] = (v & 1) ? od.v[v / 2] : ev.v[v / 2];
      } else {
        const Vec<T, V> m = ldv<V>(C.x + row + unsigned(j));
#pragma unroll
        for (int v = 0; v < V; ++v) n[k][v] = m.v[v];
      }
#pragma unroll
      for (int v = 0; v < V; ++v)
        f[k][v] = p ? (v + 1 < V ? n[k][v + 1 < V ? v + 1 : v] : e) : (v > 0 ? n[k][v > 0 ? v - 1 : 0] : e);
    }
    T *xb = F.x + half + (unsigned(z) * unsigned(r.ny) + unsigned(y)) * unsigned(r.hx) + unsigned(j);
    Vec<T, V> x = ldv<V>(xb);
#pragma unroll
    for (int v = 0; v < V; ++v)
      x.v[v] += T(0.421875) * n[0][v] + T(0.140625) * ((f[0][v] + n[1][v]) + n[2][v]) +
                T(0.046875) * ((f[1][v] + f[2][v]) + n[3][v]) + T(0.015625) * f[3][v];
    stv<V>(xb, x);
  }
}
template <typename T, class Team>
__device__ __forceinline__ void prolong_to(const Level<T> &F, const Level<T> &C, const Team &tm) {
  constexpr int V = 16 / sizeof(T);
  if (C.cf[0] && C.cf[1] && C.cf[2]) {
    if (wide(F)) prolong_black<V>(F, C, tm);
    else prolong_black<1>(F, C, tm);
    return;
  }
  const Share sh = share(tm, unsigned(F.N >> 1));
  prolong_range<true>(F, C, sh.t0, sh.dt);
}

// Four consecutive cells 4g .. 4g + 3 of the row (y, z) of a split array in
// row-major order (pr = parity of y + z: 0 when the first of them is red).
template <typename T> __device__ __forceinline__ void ld_quad(const T *a, unsigned half, unsigned at, int pr, T (&o)[4]) {
  const Vec<T, 2> r = ldv<2>(a + at), b = ldv<2>(a + half + at);
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    o[2 * k] = pr ? b.v[k] : r.v[k];
    o[2 * k + 1] = pr ? r.v[k] : b.v[k];
  }
}
template <typename T> __device__ __forceinline__ void st_quad(T *a, unsigned half, unsigned at, int pr, const T (&v)[4]) {
  Vec<T, 2> r, b;
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    r.v[k] = pr ? v[2 * k + 1] : v[2 * k];
    b.v[k] = pr ? v[2 * k] : v[2 * k + 1];
  }
  stv<2>(a + at, r);
  stv<2>(a + half + at, b);
}

// ---------------------------------------------------------------- persistent solve
// The whole solve in one cooperative launch: initial guess, coefficients, the
// residual test and the defect-correction cycles, separated by grid-wide
// barriers.  Every block evaluates the same fixed-order sums, so all blocks
// take the same branches.  The barrier wait is bounded: a block that gives up
// raises an abort flag and the device status, and every block then returns.
constexpr int kPB = 512;     // threads per block of a team
// One block per SM: the passes on V cells keep up to 60 values of a thread in
// flight and take 128 registers; at 64 (two blocks) they spill 3 KB, and 152
// blocks pass a barrier faster than 304 (1.1 us against 1.3).
constexpr int kPBlocks = 1;
constexpr long long kSpinLimit = 1LL << 24;  // default polls of a barrier wait (an L2 round trip each)
constexpr double kTrustTol = 1e-8;  // FP32 residual estimate used only above this tolerance
constexpr double kEstErr = 1e-4;    // bound of its error relative to the last exact residual

struct Bar {
  unsigned long long arrived;  // arrivals so far (reset before each launch); kBarAbort set: the solve gave up
};
constexpr unsigned long long kBarAbort = 1ull << 63;

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long *p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_add_release_u64(unsigned long long *p, unsigned long long v) {
  asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Grid barrier number `gen` (1, 2, ...) of a launch: thread 0 of every block
// adds its arrival with release semantics (the block's writes, ordered by the
// preceding __syncthreads) and polls the count with acquire loads until all
// blocks of this generation have arrived.  What bounds it is the round trip
// to the L2: the arrival returns no value (the target follows from the
// generation the caller counts), the abort flag is the top bit of the polled
// word, and polls follow each other without a sleep, so a barrier is one
// one-way add and one load past the last arrival.  The wait is bounded; on
// time-out the block raises the abort bit and the status, and every block
// leaves at its next barrier.
__device__ __forceinline__ bool grid_sync(Bar *bar, unsigned long long gen, int *status, long long spin_limit) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned long long target = gen * gridDim.x;
    red_add_release_u64(&bar->arrived, 1ull);
    unsigned long long v;
    long long spins = 0;
    while ((v = ld_acquire_u64(&bar->arrived)) < target) {  // the abort bit also ends the wait
      if (++spins > spin_limit) {
        v = atomicOr(&bar->arrived, kBarAbort) | kBarAbort;
        atomicOr(status, ST_TIMEOUT);
        break;
      }
    }
    ok = !(v & kBarAbort);
  }
  __syncthreads();
  return ok != 0;
}


// A team is the set of blocks that solves one system: the whole grid of a
// cooperative launch (barrier on a global counter, bounded wait), or one
// thread-block cluster (hardware cluster barrier with release/acquire
// semantics, no polling).
struct GridTeam {
  Bar *bar;
  int *status;
  long long spin_limit;  // polls of a barrier wait before the solve gives up
  mutable unsigned long long gen = 0;  // barriers passed in this launch
  __device__ GridTeam(Bar *b, int *s, long long limit) : bar(b), status(s), spin_limit(limit) {}
  __device__ long long rank() const { return blockIdx.x * (long long)blockDim.x + threadIdx.x; }
  __device__ long long size() const { return (long long)gridDim.x * blockDim.x; }
  __device__ int block() const { return blockIdx.x; }
  __device__ int nblocks() const { return gridDim.x; }
  __device__ bool sync() const { return grid_sync(bar, ++gen, status, spin_limit); }
};

struct ClusterTeam {
  unsigned crank, csize;
  mutable unsigned long long gen = 0;  // barriers passed in this launch
  __device__ ClusterTeam() {
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(crank));
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(csize));
  }
  __device__ long long rank() const { return (long long)crank * blockDim.x + threadIdx.x; }
  __device__ long long size() const { return (long long)csize * blockDim.x; }
  __device__ int block() const { return int(crank); }
  __device__ int nblocks() const { return int(csize); }
  __device__ bool sync() const {
    ++gen;
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
    return true;
  }
};

template <typename T> struct PArgs {
  const Level<T> *lv;                          // level table in device memory
  int nlev;
  int tail;                                    // first level relaxed by block 0 in shared memory
  const T *eps, *q;
  double *phi, *prev;                          // FP64 potential (FP64 mode)
  float *phi_hi, *phi_lo, *prev_hi, *prev_lo;  // double-float potential (FP32 modes)
  DF edf[3];
  double ex, ey, ez;
  PDev *st;
  int *status;
  double *part;  // block sums of two reductions in turn (team_part.h)
  Bar *bar;
  long long spin_limit;  // polls of a grid-barrier wait before time-out (cooperative solve)
};

// Exact residual r = b - A phi of one cell with b = -(q - qbar) + sum_d k (E_ext . c_d), in the precision of the
// potential; kk: the six faces +x -x +y -y +z -z.
// Double-float: sum_k k_k (phi_k - phi_i) from exact differences of the high
// words (two_sum) plus the differences of the low words, the high products
// exact with their FMA error terms, high parts summed with compensation
// (about 2^-46 of the largest flux term, as in general double-float
// arithmetic, at less than half its operations).
struct ResDF {
  float r, b;
};
template <typename T>
__device__ __forceinline__ ResDF residual_df(const PArgs<T> &a, float q, DF qbar, float h0, float l0,
                                             const float (&hi)[6], const float (&lo)[6], const float (&kk)[6]) {
  float ahi = 0.f, alo = 0.f;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const DF dd = two_sum(hi[k], -h0);
    const float dlo = __fadd_rn(dd.lo, __fsub_rn(lo[k], l0));
    const float prod = __fmul_rn(dd.hi, kk[k]);
    const float plo = __fmaf_rn(dlo, kk[k], __fmaf_rn(dd.hi, kk[k], -prod));
    const DF t = two_sum(ahi, prod);
    ahi = t.hi;
    alo = __fadd_rn(alo, __fadd_rn(t.lo, plo));
  }
  DF b = two_sum(qbar.hi, -q);
  b.lo = __fadd_rn(b.lo, qbar.lo);
  if (a.edf[0].hi != 0.f) b = df_add(b, df_mul(a.edf[0], two_sum(kk[0], -kk[1])));
  if (a.edf[1].hi != 0.f) b = df_add(b, df_mul(a.edf[1], two_sum(kk[2], -kk[3])));
  if (a.edf[2].hi != 0.f) b = df_add(b, df_mul(a.edf[2], two_sum(kk[4], -kk[5])));
  const DF r = two_sum(b.hi, -ahi);
  return ResDF{__fadd_rn(r.hi, __fadd_rn(r.lo, __fsub_rn(b.lo, alo))), b.hi};
}

// one cell, any layout (FP32: faces from the row-major eps; FP64: stored faces)
template <typename T, bool DFM>
__device__ __forceinline__ void residual_site(const PArgs<T> &a, const Level<T> &L0, int x, int y, int z,
                                              double qbar, DF qbar_df, SumAcc<DFM> &ar, SumAcc<DFM> &ab,
                                              SumAcc<DFM> &ap) {
  const Nbr c = nbr(L0.dims(), x, y, z);
  const unsigned i = c.i, nb[6] = {c.xp, c.xm, c.yp, c.ym, c.zp, c.zm};
  const int color = (x + y + z) & 1;
  const unsigned at = cell_at(L0, i, color);
  if constexpr (DFM) {
    float hi[6], lo[6], kk[6];
    const float e = a.eps[i];
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      hi[k] = a.phi_hi[nb[k]];
      lo[k] = a.phi_lo[nb[k]];
      kk[k] = 0.5f * (e + a.eps[nb[k]]);
    }
    const float h0 = a.phi_hi[i];
    const ResDF r = residual_df(a, a.q[i], qbar_df, h0, a.phi_lo[i], hi, lo, kk);
    L0.b[at] = r.r;
    ar.add(r.r * r.r);
    ab.add(r.b * r.b);
    ap.add(h0);
  } else {
    const double kxp = L0.k[0][at], kxm = L0.k[0][cell_at(L0, c.xm, color ^ 1)];
    const double kyp = L0.k[1][at], kym = L0.k[1][cell_at(L0, c.ym, color ^ 1)];
    const double kzp = L0.k[2][at], kzm = L0.k[2][cell_at(L0, c.zm, color ^ 1)];
    const double *phi = a.phi;
    const double p = phi[i];
    double b = -(double(a.q[i]) - qbar);
    if (a.ex != 0.0) b += a.ex * (kxp - kxm);
    if (a.ey != 0.0) b += a.ey * (kyp - kym);
    if (a.ez != 0.0) b += a.ez * (kzp - kzm);
    const double Ap = kxp * (phi[c.xp] - p) - kxm * (p - phi[c.xm]) + kyp * (phi[c.yp] - p) - kym * (p - phi[c.ym]) +
                      kzp * (phi[c.zp] - p) - kzm * (p - phi[c.zm]);
    const double r = b - Ap;
    L0.b[at] = T(r);
    ar.add(r * r);
    ab.add(b * b);
    ap.add(p);
  }
}

// Four cells of a row (FP32, rows of a multiple of four cells): 16-byte loads
// of the row and its four neighbour rows and one word past each end, 24 loads
// instead of 22 per cell.  out: the residual, rhs: the right-hand side's high
// word, pot: the potential's high word of each cell, for the caller's sums.
template <typename T>
__device__ __forceinline__ void residual_quad(const PArgs<T> &a, const Level<T> &L0, int g, int y, int z, DF qbar,
                                              float (&out)[4], float (&rhs)[4], float (&pot)[4]) {
  const unsigned nx = unsigned(L0.nx), sz = nx * unsigned(L0.ny), n = unsigned(L0.N);
  const unsigned x0 = 4u * unsigned(g), row = unsigned(z) * sz + unsigned(y) * nx, i = row + x0;
  const unsigned rw[5] = {i, y + 1 == L0.ny ? i - (sz - nx) : i + nx, y == 0 ? i + (sz - nx) : i - nx,
                          z + 1 == L0.nz ? i - (n - sz) : i + sz, z == 0 ? i + (n - sz) : i - sz};
  const unsigned ip = x0 + 4u == nx ? row : i + 4u, im = x0 == 0u ? row + nx - 1u : i - 1u;
  Vec<float, 4> h[5], l[5], e[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    h[k] = ldv<4>(a.phi_hi + rw[k]);
    l[k] = ldv<4>(a.phi_lo + rw[k]);
    e[k] = ldv<4>(a.eps + rw[k]);
  }
  const float hp = a.phi_hi[ip], hm = a.phi_hi[im], lp = a.phi_lo[ip], lm = a.phi_lo[im], ep = a.eps[ip],
              em = a.eps[im];
  const Vec<float, 4> q = ldv<4>(a.q + i);
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    const float hi[6] = {v < 3 ? h[0].v[v < 3 ? v + 1 : 3] : hp, v > 0 ? h[0].v[v > 0 ? v - 1 : 0] : hm,
                         h[1].v[v], h[2].v[v], h[3].v[v], h[4].v[v]};
    const float lo[6] = {v < 3 ? l[0].v[v < 3 ? v + 1 : 3] : lp, v > 0 ? l[0].v[v > 0 ? v - 1 : 0] : lm,
                         l[1].v[v], l[2].v[v], l[3].v[v], l[4].v[v]};
    const float e0 = e[0].v[v];
    const float kk[6] = {0.5f * (e0 + (v < 3 ? e[0].v[v < 3 ? v + 1 : 3] : ep)),
                         0.5f * (e0 + (v > 0 ? e[0].v[v > 0 ? v - 1 : 0] : em)), 0.5f * (e0 + e[1].v[v]),
                         0.5f * (e0 + e[2].v[v]), 0.5f * (e0 + e[3].v[v]), 0.5f * (e0 + e[4].v[v])};
    const ResDF r = residual_df(a, q.v[v], qbar, h[0].v[v], l[0].v[v], hi, lo, kk);
    out[v] = r.r;
    rhs[v] = r.b;
    pot[v] = h[0].v[v];
  }
}

// The last five levels of a block's sum tree by one warp: the same pairs as the
// shared-memory levels (t and t + w), without their barriers and round trips.
template <int M, int STRIDE> __device__ __forceinline__ void warp_tail(double (&v)[M], double *sh) {
  if (threadIdx.x < 32) {
#pragma unroll
    for (int m = 0; m < M; ++m) v[m] = sh[m * STRIDE + threadIdx.x];
#pragma unroll
    for (int w = 16; w > 0; w >>= 1)
#pragma unroll
      for (int m = 0; m < M; ++m) v[m] += __shfl_down_sync(0xffffffffu, v[m], w);
    if (threadIdx.x == 0)
#pragma unroll
      for (int m = 0; m < M; ++m) sh[m * STRIDE] = v[m];
  }
  __syncthreads();
#pragma unroll
  for (int m = 0; m < M; ++m) v[m] = sh[m * STRIDE];
  __syncthreads();
}

// Fixed-order sums of M values over the block at once: a shared-memory tree
// whose levels add all M values behind one set of barriers.  sh: M kPB doubles.
template <int M> __device__ __forceinline__ void block_sums(double (&v)[M], double *sh) {
#pragma unroll
  for (int m = 0; m < M; ++m) sh[m * kPB + threadIdx.x] = v[m];
  __syncthreads();
  for (int w = blockDim.x / 2; w >= 32; w >>= 1) {
    if (threadIdx.x < w)
#pragma unroll
      for (int m = 0; m < M; ++m) sh[m * kPB + threadIdx.x] += sh[m * kPB + threadIdx.x + w];
    __syncthreads();
  }
  warp_tail<M, kPB>(v, sh);
}
// the team's sums of M per-thread values, identical in every block; false on abort
template <int M, class Team>
__device__ __forceinline__ bool team_sums(double (&v)[M], double *part, const Team &tm, double *sh) {
  block_sums<M>(v, sh);
  const int nb = tm.nblocks();
  if (threadIdx.x == 0)
#pragma unroll
    for (int m = 0; m < M; ++m) part[part_at(tm.gen, m, nb, tm.block())] = v[m];
  if (!tm.sync()) return false;
#pragma unroll
  for (int m = 0; m < M; ++m) v[m] = 0.0;
  for (int b = threadIdx.x; b < nb; b += blockDim.x)
#pragma unroll
    for (int m = 0; m < M; ++m) v[m] += part[part_at(tm.gen - 1, m, nb, b)];
  block_sums<M>(v, sh);
  return true;
}

// FP64 scalar arithmetic (divisions, square roots) by one thread, broadcast
// through shared memory: 512 threads repeating a relative residual took 4 us
// a cycle at the target's FP64 rate.
template <class F> __device__ __forceinline__ double by_one(double *cell, F f) {
  if (threadIdx.x == 0) *cell = f();
  __syncthreads();
  const double v = *cell;
  __syncthreads();
  return v;
}

// residual pass + fixed-order sums in every block; returns false on abort
template <typename T, bool DFM, class Team>
__device__ bool residual_pass(const PArgs<T> &a, const Team &tm, const Level<T> &L0, double qbar, DF qbar_df,
                              double *sh, double &r2, double &b2, double &ps) {
  SumAcc<DFM> sr, sb, sp;
  const long long N = L0.N;
  if constexpr (DFM) {
    if (L0.split && (L0.nx & 3) == 0) {
      const Share s = share(tm, unsigned(N >> 2));
      for (Walk w(s.t0, s.dt, L0.nx >> 2, L0.ny); w.z < L0.nz; w.next()) {
        float out[4], rhs[4], pot[4];
        residual_quad(a, L0, w.u, w.y, w.z, qbar_df, out, rhs, pot);
        st_quad<float>(L0.b, unsigned(N >> 1), site32(L0.dims(), 4 * w.u, w.y, w.z) >> 1, (w.y + w.z) & 1, out);
        // each cell's terms in double-float, as in residual_site
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          sr.add(out[v] * out[v]);
          sb.add(rhs[v] * rhs[v]);
          sp.add(pot[v]);
        }
      }
    } else {
      const Share s = share(tm, unsigned(L0.N));
      for (Walk w(s.t0, s.dt, L0.nx, L0.ny); w.z < L0.nz; w.next())
        residual_site<T, DFM>(a, L0, w.u, w.y, w.z, qbar, qbar_df, sr, sb, sp);
    }
  } else {
    const Share s = share(tm, unsigned(L0.N));
    for (Walk w(s.t0, s.dt, L0.nx, L0.ny); w.z < L0.nz; w.next())
      residual_site<T, DFM>(a, L0, w.u, w.y, w.z, qbar, qbar_df, sr, sb, sp);
  }
  double v[3] = {sr.get(), sb.get(), sp.get()};
  if (!team_sums<3>(v, a.part, tm, sh)) return false;
  r2 = v[0];
  b2 = v[1];
  ps = v[2];
  return true;
}

// Carried residual and potential of four cells of a row: r <- r - A e on the
// FP32 residual (its rounding error is relative to |A e| ~ |r|), phi += e in
// double-float.  Every cell, black ones included: after the black half sweep
// their residual is zero only up to the FP32 rounding of the update, which
// scales with the correction and must stay visible to later cycles.
template <typename T>
__device__ __forceinline__ void carry_quad(const PArgs<T> &a, const Level<T> &L, int g, int y, int z,
                                           SumAcc<true> &sr, SumAcc<true> &sp) {
  const unsigned hx = unsigned(L.nx >> 1), sz = hx * unsigned(L.ny), half = unsigned(L.N >> 1);
  const unsigned j = 2u * unsigned(g), row = unsigned(z) * sz + unsigned(y) * hx, i = row + j;
  const unsigned rw[4] = {y + 1 == L.ny ? i - (sz - hx) : i + hx, y == 0 ? i + (sz - hx) : i - hx,
                          z + 1 == L.nz ? i - (half - sz) : i + sz, z == 0 ? i + (half - sz) : i - sz};
  const int pr = (y + z) & 1;
  // the cell past the four has the colour of the first, the one before it that of the last
  const unsigned ip = (pr ? half : 0u) + (j + 2u == hx ? row : i + 2u);
  const unsigned im = (pr ? 0u : half) + (j == 0u ? row + hx - 1u : i - 1u);
  float x[4], e[4], xn[4][4], en[4][4], b[4], out[4];
  ld_quad<float>(L.x, half, i, pr, x);
  ld_quad<float>(L.eps, half, i, pr, e);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    ld_quad<float>(L.x, half, rw[k], pr ^ 1, xn[k]);
    ld_quad<float>(L.eps, half, rw[k], pr ^ 1, en[k]);
  }
  const float xp = L.x[ip], xm = L.x[im], ep = L.eps[ip], em = L.eps[im];
  ld_quad<float>(L.b, half, i, pr, b);
  Vec<float, 4> h = ldv<4>(a.phi_hi + 2u * i), l = ldv<4>(a.phi_lo + 2u * i);
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    const float xv[6] = {v < 3 ? x[v < 3 ? v + 1 : 3] : xp, v > 0 ? x[v > 0 ? v - 1 : 0] : xm,
                         xn[0][v], xn[1][v], xn[2][v], xn[3][v]};
    const float ev[6] = {v < 3 ? e[v < 3 ? v + 1 : 3] : ep, v > 0 ? e[v > 0 ? v - 1 : 0] : em,
                         en[0][v], en[1][v], en[2][v], en[3][v]};
    float Ae = 0.f;
#pragma unroll
    for (int k = 0; k < 6; ++k) Ae += 0.5f * (e[v] + ev[k]) * (xv[k] - x[v]);
    const float r = b[v] - Ae;
    out[v] = r;
    sr.add(r * r);
    const DF s = df_add_f(DF{h.v[v], l.v[v]}, x[v]);
    h.v[v] = s.hi;
    l.v[v] = s.lo;
    sp.add(s.hi);
  }
  st_quad<float>(L.b, half, i, pr, out);
  stv<4>(a.phi_hi + 2u * i, h);
  stv<4>(a.phi_lo + 2u * i, l);
}

// the same for one cell, any layout
template <typename T>
__device__ __forceinline__ void carry_site(const PArgs<T> &a, const Level<T> &L, int x, int y, int z,
                                           SumAcc<true> &sr, SumAcc<true> &sp) {
  const Nbr c = nbr(L.dims(), x, y, z);
  const unsigned nb[6] = {c.xp, c.xm, c.yp, c.ym, c.zp, c.zm};
  const int color = (x + y + z) & 1;
  const unsigned at = cell_at(L, c.i, color);
  const float x0 = L.x[at], e0 = a.eps[c.i];
  // a neighbour along an axis of odd extent has no colour of its own: only
  // row-major levels have such axes, and there the colour is not used
  float Ae = 0.f;
#pragma unroll
  for (int k = 0; k < 6; ++k) Ae += 0.5f * (e0 + a.eps[nb[k]]) * (L.x[cell_at(L, nb[k], color ^ 1)] - x0);
  const float r = L.b[at] - Ae;
  L.b[at] = r;
  sr.add(r * r);
  const DF s = df_add_f(DF{a.phi_hi[c.i], a.phi_lo[c.i]}, x0);
  a.phi_hi[c.i] = s.hi;
  a.phi_lo[c.i] = s.lo;
  sp.add(s.hi);
}

// The whole solve of one system by one team: initial guess, coefficients,
// the residual test and the defect-correction cycles, separated by team
// barriers.  Every block of the team evaluates the same fixed-order sums, so
// all blocks take the same branches.  smem_raw holds the tail levels, sh
// (3 kPB doubles) block scratch, lv the level table.
template <typename T, bool DFM, class Team>
__device__ void poisson_body(const PArgs<T> &a, const Team &tm, unsigned char *smem_raw, double *sh, Level<T> *lv) {
  // the level table in shared memory: a barrier empties the L1, and each
  // phase would begin with reads of it from the L2
  for (int l = threadIdx.x; l < a.nlev; l += blockDim.x) lv[l] = a.lv[l];
  __syncthreads();
  const Level<T> L0 = lv[0];  // by value: stores cannot alias it
  const Dims d = L0.dims();
  const long long N = d.N;
  PDev *st = a.st;
  const int have_prev = st->have_prev;

  // initial guess, level-0 coefficients (faces, or the colour-split copy of eps), sum of q
  SumAcc<DFM> sq;
  {
    T *es = const_cast<T *>(L0.eps);
    bool quads = false;
    if constexpr (DFM) {
      quads = L0.split && (L0.nx & 3) == 0;
      if (quads) {
        const Share s = share(tm, unsigned(N >> 2));
        for (Walk w(s.t0, s.dt, L0.nx >> 2, L0.ny); w.z < L0.nz; w.next()) {
          const unsigned i = site32(d, 4 * w.u, w.y, w.z);
          const Vec<float, 4> h = ldv<4>(a.phi_hi + i), l = ldv<4>(a.phi_lo + i), q = ldv<4>(a.q + i);
          const Vec<float, 4> e = ldv<4>(a.eps + i);
          if (have_prev) {
            const Vec<float, 4> ph = ldv<4>(a.prev_hi + i), pl = ldv<4>(a.prev_lo + i);
            Vec<float, 4> gh, gl;
#pragma unroll
            for (int v = 0; v < 4; ++v) {
              const DF gv = df_sub(DF{2.f * h.v[v], 2.f * l.v[v]}, DF{ph.v[v], pl.v[v]});
              gh.v[v] = gv.hi;
              gl.v[v] = gv.lo;
            }
            stv<4>(a.phi_hi + i, gh);
            stv<4>(a.phi_lo + i, gl);
          }
          stv<4>(a.prev_hi + i, h);
          stv<4>(a.prev_lo + i, l);
          st_quad<float>(es, unsigned(N >> 1), i >> 1, (w.y + w.z) & 1, e.v);
          // each term in double-float: the mean charge offsets the residual of every cell
#pragma unroll
          for (int v = 0; v < 4; ++v) sq.add(q.v[v]);
        }
      }
    }
    if (!quads) {
      const Share s = share(tm, unsigned(N));
      for (Walk w(s.t0, s.dt, d.nx, d.ny); w.z < d.nz; w.next()) {
        const Nbr c = nbr(d, w.u, w.y, w.z);
        const unsigned i = c.i;
        if constexpr (DFM) {
          const DF p{a.phi_hi[i], a.phi_lo[i]};
          if (have_prev) {
            const DF g = df_sub(DF{2.f * p.hi, 2.f * p.lo}, DF{a.prev_hi[i], a.prev_lo[i]});
            a.phi_hi[i] = g.hi;
            a.phi_lo[i] = g.lo;
          }
          a.prev_hi[i] = p.hi;
          a.prev_lo[i] = p.lo;
        } else {
          const double p = a.phi[i];
          if (have_prev) a.phi[i] = 2.0 * p - a.prev[i];
          a.prev[i] = p;
        }
        const T e = a.eps[i];
        const unsigned at = cell_at(L0, i, (w.u + w.y + w.z) & 1);
        if (es) {
          es[at] = e;
        } else {
          L0.k[0][at] = T(0.5) * (e + a.eps[c.xp]);
          L0.k[1][at] = T(0.5) * (e + a.eps[c.yp]);
          L0.k[2][at] = T(0.5) * (e + a.eps[c.zp]);
        }
        sq.add(a.q[i]);
      }
    }
  }
  double qs[1] = {sq.get()};
  if (!team_sums<1>(qs, a.part, tm, sh)) return;
  const double qbar = by_one(sh, [&] { return qs[0] / double(N); });
  const DF qbar_df = df_split(qbar);
  // coarse face coefficients, level by level, and 1 / diag of the level before
  for (int l = 1; l < a.nlev; ++l) {
    const Level<T> F = lv[l - 1], C = lv[l];
    const Dims c = C.dims();
    const Share s = share(tm, unsigned(C.N));
    const bool from_eps = F.eps && !F.far && C.cf[0] && C.cf[1] && C.cf[2] && C.nx > 1 && C.ny > 1 && C.nz > 1;
    for (Walk w(s.t0, s.dt, c.nx, c.ny); w.z < c.nz; w.next()) {
      const unsigned I = cell_at(C, site32(c, w.u, w.y, w.z), (w.u + w.y + w.z) & 1);
      T k[3];
      if (from_eps) {
        coarse_faces_from_eps(a.eps, d, w.u, w.y, w.z, k);
      } else {
        k[0] = coarse_coef<0>(F, C, w.u, w.y, w.z);
        k[1] = coarse_coef<1>(F, C, w.u, w.y, w.z);
        k[2] = coarse_coef<2>(F, C, w.u, w.y, w.z);
      }
      C.k[0][I] = k[0];
      C.k[1][I] = k[1];
      C.k[2][I] = k[2];
    }
    if (F.d) inverse_diag(F, tm);
    if (!tm.sync()) return;
  }
  if (lv[a.nlev - 1].d) inverse_diag(lv[a.nlev - 1], tm);  // read after the residual's barrier
  // residual test
  double r2, b2, ps;
  if (!residual_pass<T, DFM>(a, tm, L0, qbar, qbar_df, sh, r2, b2, ps)) return;
  const double tol = st->tol;
  const int max_iter = st->max_iter;
  const double bn = b2;
  double rr = by_one(sh, [&] { return rel_res(r2, bn); });
  int it = 0;
  // In the FP32 modes the level-0 residual is carried from cycle to cycle in
  // FP32 (r <- r - A e); that estimate is accurate to about 1e-5 of the
  // starting residual, so below kTrustTol the exact double-float residual
  // re-anchors it before convergence is accepted.
  bool exact = true;
  const bool carry = DFM && tol >= kTrustTol;
  double rr0 = rr;
  for (;;) {
    while (rr >= tol && it < max_iter) {
      exact = !carry;
      // V-cycle on the correction: levels above the tail, red-black smoothing
      for (int l = 0; l < a.tail; ++l) {
        const Level<T> Ll = lv[l];
        // the first red half sweep is from x = 0; on coarse levels the
        // restriction that produced the right-hand side has done it
        if (l == 0) {
          sweep_colour<true>(Ll, 0, tm);
          if (!tm.sync()) return;
        }
        for (int s = 0; s < kNu; ++s) {
          if (s > 0) {
            sweep_colour<false>(Ll, 0, tm);
            if (!tm.sync()) return;
          }
          sweep_colour<false>(Ll, 1, tm);
          if (!tm.sync()) return;
        }
        restrict_to(Ll, lv[l + 1], tm);
        if (!tm.sync()) return;
      }
      if (tm.block() == 0) tail_vcycle(lv, a.nlev, a.tail, smem_raw);
      if (!tm.sync()) return;
      for (int l = a.tail - 1; l >= 0; --l) {
        const Level<T> Ll = lv[l];
        prolong_to(Ll, lv[l + 1], tm);
        if (!tm.sync()) return;
        for (int s = 0; s < kNu; ++s) {
          sweep_colour<false>(Ll, 0, tm);
          if (!tm.sync()) return;
          sweep_colour<false>(Ll, 1, tm);
          if (!tm.sync()) return;
        }
      }
      // phi += correction; the residual follows the correction
      bool carried = false;
      if constexpr (DFM) {
        if (carry) {
          SumAcc<true> sr, sp;
          if (L0.split && (L0.nx & 3) == 0) {
            const Share s = share(tm, unsigned(N >> 2));
            for (Walk w(s.t0, s.dt, L0.nx >> 2, L0.ny); w.z < L0.nz; w.next()) carry_quad(a, L0, w.u, w.y, w.z, sr, sp);
          } else {
            const Share s = share(tm, unsigned(N));
            for (Walk w(s.t0, s.dt, L0.nx, L0.ny); w.z < L0.nz; w.next()) carry_site(a, L0, w.u, w.y, w.z, sr, sp);
          }
          double v[2] = {sr.get(), sp.get()};
          if (!team_sums<2>(v, a.part, tm, sh)) return;
          r2 = v[0];
          ps = v[1];
          carried = true;
        }
      }
      if (!carried) {
        const Share s = share(tm, unsigned(N));
        for (Walk w(s.t0, s.dt, d.nx, d.ny); w.z < d.nz; w.next()) {
          const unsigned i = site32(d, w.u, w.y, w.z);
          const T e = L0.x[cell_at(L0, i, (w.u + w.y + w.z) & 1)];
          if constexpr (DFM) {
            const DF v = df_add(DF{a.phi_hi[i], a.phi_lo[i]}, DF{float(e), 0.f});
            a.phi_hi[i] = v.hi;
            a.phi_lo[i] = v.lo;
          } else {
            a.phi[i] += double(e);
          }
        }
        if (!tm.sync()) return;
        if (!residual_pass<T, DFM>(a, tm, L0, qbar, qbar_df, sh, r2, b2, ps)) return;
      }
      rr = by_one(sh, [&] { return rel_res(r2, bn); });
      ++it;
    }
    if (exact || rr + kEstErr * rr0 < tol) break;
    if (!residual_pass<T, DFM>(a, tm, L0, qbar, qbar_df, sh, r2, b2, ps)) return;
    rr = by_one(sh, [&] { return rel_res(r2, bn); });
    rr0 = rr;
    exact = true;
    if (rr < tol || it >= max_iter) break;
  }
  const bool zero = bn == 0.0;
  const double mean_phi = by_one(sh, [&] { return ps / double(N); });
  const DF mean_df = df_split(mean_phi);
  long long done = 0;
  if constexpr (DFM) {
    if ((N & 3) == 0) {
      const Share s = share(tm, unsigned(N >> 2));
      for (long long t = s.t0; t < (N >> 2); t += s.dt) {
        Vec<float, 4> h = ldv<4>(a.phi_hi + 4 * t), l = ldv<4>(a.phi_lo + 4 * t);
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          DF o{0.f, 0.f};
          if (!zero) o = df_sub(DF{h.v[v], l.v[v]}, mean_df);
          h.v[v] = o.hi;
          l.v[v] = o.lo;
        }
        stv<4>(a.phi_hi + 4 * t, h);
        stv<4>(a.phi_lo + 4 * t, l);
      }
      done = N;
    }
  }
  for (long long i = done + tm.rank(); i < N; i += tm.size()) {
    if constexpr (DFM) {
      DF v{0.f, 0.f};
      if (!zero) v = df_sub(DF{a.phi_hi[i], a.phi_lo[i]}, mean_df);
      a.phi_hi[i] = v.hi;
      a.phi_lo[i] = v.lo;
    } else {
      a.phi[i] = zero ? 0.0 : a.phi[i] - mean_phi;
    }
  }
  if (tm.rank() == 0) {
    st->mean_q = qbar;
    st->mean_phi = mean_phi;
    st->bnorm2 = bn;
    st->rnorm2 = r2;
    st->relres = rr;
    st->iters = it;
    st->total_iters += it;
    const int fail = !(rr < tol);  // not converged, or not finite
    st->notconv = fail;
    st->cond = 0;
    st->zero = zero;
    st->have_prev = 1;
    if (fail) atomicOr(a.status, ST_POISSON);
    if (!isfinite(rr)) atomicOr(a.status, ST_NONFINITE);
  }
}

}  // namespace lbeh
