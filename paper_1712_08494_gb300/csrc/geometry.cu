// Projection of spherical colloids onto the lattice (Sec. II.E).
//
// A node is solid when its centre is strictly inside a sphere (minimum-image
// squared distance < r^2).  The solid fraction psi_s = nu/(h+1)^3 counts the
// sub-cube centres (h+1 per axis) strictly inside.  Surface nodes are solid
// nodes with a fluid D3Q19 neighbour; the colloid's charge Q is split equally
// over them.  Distances are evaluated with explicitly rounded FP64 operations
// (no fused multiply-add) in a fixed order, so the masks are bit-identical to
// any IEEE FP64 evaluation of ((dx*dx + dy*dy) + dz*dz) < r*r.
#include "internal.h"

namespace lbeh {

__device__ __forceinline__ double min_image(double dd, int n) {
  const double half = 0.5 * double(n);
  if (dd > half) return __dsub_rn(dd, double(n));
  if (dd < -half) return __dadd_rn(dd, double(n));
  return dd;
}

__device__ __forceinline__ double dist2(double px, double py, double pz, const double *X, const Dims &d) {
  const double dx = min_image(__dsub_rn(px, X[0]), d.nx);
  const double dy = min_image(__dsub_rn(py, X[1]), d.ny);
  const double dz = min_image(__dsub_rn(pz, X[2]), d.nz);
  return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

// Position of a node or sample relative to the sphere centre, split into
// the integer part of the centre (exact) and a fractional remainder: in FP32
// the offset d = (x - floor(X)) + o - frac(X) is then within 1e-6 of the exact
// value times 2^-23 |d|, so |d^2 - r^2| > 1e-3 + 1e-5 r^2 decides "inside"
// exactly as the rounded FP64 test does; closer cases use the FP64 test itself.
constexpr float kCertain = 1e-3f;

__device__ __forceinline__ int wrap_rel(int dx, int n) {
  // minimum-image integer offset in (-n/2, n/2]
  if (dx > n / 2) dx -= n;
  if (dx <= -((n + 1) / 2)) dx += n;
  return dx;
}

template <typename T>
__global__ void k_project(Dims d, int h, const double *__restrict__ cx, const double *__restrict__ cr,
                          uint8_t *__restrict__ solid, int *__restrict__ owner, T *__restrict__ psi_s, int slabs) {
  const int j = blockIdx.x / slabs, sl = blockIdx.x - j * slabs;
  const double X[3] = {cx[3 * j], cx[3 * j + 1], cx[3 * j + 2]};
  const double r = cr[j];
  const double r2 = __dmul_rn(r, r);
  const float r2f = float(r2);
  const float certain = kCertain + 1e-5f * r2f;
  const SphereBox b = block_box(d, X, r, 1.0);
  const int hp = h + 1;
  const int dims[3] = {d.nx, d.ny, d.nz};
  __shared__ int Xi[3];
  __shared__ float Xf[3];
  if (threadIdx.x < 3) {
    const double Xa = cx[3 * j + threadIdx.x], fl = floor(Xa);
    Xi[threadIdx.x] = int(fl);
    Xf[threadIdx.x] = float(Xa - fl);  // exact difference, rounded once to FP32
  }
  // sub-cube centre offsets (k + 1/2)/(h+1) - 1/2, once per block
  __shared__ double off[16];
  __shared__ float offf[16];
  if (threadIdx.x < hp) {
    off[threadIdx.x] = __dsub_rn(__ddiv_rn(threadIdx.x + 0.5, double(hp)), 0.5);
    offf[threadIdx.x] = float(off[threadIdx.x]);  // dyadic: exact in FP32
  }
  __syncthreads();
  // Every sub-cube centre lies within sqrt(3) (1/2 - 1/(2(h+1))) of its node;
  // a node farther than that (plus 1e-3) from the sphere surface has all its
  // samples on one side.  Used only where every sample and the node share one
  // periodic image.
  __shared__ float r_lim[2];  // r - reach and r + reach
  __shared__ bool short_ok;
  if (threadIdx.x == 0) {
    const double reach = 1.7320508075688772 * (0.5 - 0.5 / double(hp)) + 1e-3;
    r_lim[0] = float(r - reach);
    r_lim[1] = float(r + reach);
    short_ok = 2.0 * (r + reach + 1.0) < double(min(d.nx, min(d.ny, d.nz)));
  }
  __syncthreads();
  const float rinf = r_lim[0], routf = r_lim[1];
  const bool shortcut = short_ok;
  for (unsigned t = unsigned(sl) * blockDim.x + threadIdx.x; t < b.tot; t += unsigned(slabs) * blockDim.x) {
    int x, y, z;
    b.node(t, x, y, z);
    const long long i = site(d, x, y, z);
    const int p[3] = {x, y, z};
    float rel[3];
    for (int a = 0; a < 3; ++a) rel[a] = float(wrap_rel(p[a] - Xi[a], dims[a])) - Xf[a];
    const float d2f = rel[0] * rel[0] + rel[1] * rel[1] + rel[2] * rel[2];
    // (the FP32 offsets pick the nearest periodic image; the FP64 test may pick
    // the other one only for samples about half a box away, which are outside
    // whenever the shortcut condition holds, so the fast path is used only then)
    bool in_node;
    if (shortcut && fabsf(d2f - r2f) > certain) in_node = d2f < r2f;
    else in_node = dist2(double(x), double(y), double(z), X, d) < r2;
    if (in_node) {
      solid[i] = 1;
      atomicMax(owner + i, j);
    }
    int nu = 0;
    if (shortcut && rinf > 0.f && d2f < rinf * rinf - certain) {
      nu = hp * hp * hp;
    } else if (shortcut && d2f > routf * routf + certain) {
      nu = 0;
    } else {
      for (int kz = 0; kz < hp; ++kz) {
        const float qz = rel[2] + offf[kz];
        for (int ky = 0; ky < hp; ++ky) {
          const float qy = rel[1] + offf[ky];
          const float s2 = qy * qy + qz * qz;
          for (int kx = 0; kx < hp; ++kx) {
            const float qx = rel[0] + offf[kx];
            const float e2 = qx * qx + s2;
            bool in;
            if (shortcut && fabsf(e2 - r2f) > certain)
              in = e2 < r2f;
            else
              in = dist2(__dadd_rn(double(x), off[kx]), __dadd_rn(double(y), off[ky]), __dadd_rn(double(z), off[kz]),
                         X, d) < r2;
            nu += in ? 1 : 0;
          }
        }
      }
    }
    // dyadic values: exact in any order
    if (nu) atomicAdd(psi_s + i, nu == hp * hp * hp ? T(1) : T(double(nu) / (double(hp) * hp * hp)));
  }
}

// Nodes within r + 2 of a centre (minimum image).  A node partly covered by a
// sphere lies within r + sqrt(3)/2 of its centre and a solid one within r, so a
// node outside the mark has no solid D3Q19 neighbour (sqrt(2) away at most),
// and neither it nor an axis neighbour is covered in part.  FP32 offsets carry
// an error below 1e-4, inside the margin of 0.01.
__global__ void k_near(Dims d, const double *__restrict__ cx, const double *__restrict__ cr, uint8_t *__restrict__ near,
                       int slabs) {
  const int j = blockIdx.x / slabs, sl = blockIdx.x - j * slabs;
  const double X[3] = {cx[3 * j], cx[3 * j + 1], cx[3 * j + 2]};
  const SphereBox b = block_box(d, X, cr[j], 2.01);
  const int dims[3] = {d.nx, d.ny, d.nz};
  const float lim = float(cr[j]) + 2.01f;
  // the centre's integer part (it may lie outside the box by whole periods) and its remainder
  __shared__ int Xi[3];
  __shared__ float Xf[3];
  if (threadIdx.x < 3) {
    const double Xa = cx[3 * j + threadIdx.x], fl = floor(Xa);
    Xi[threadIdx.x] = int(fl);
    Xf[threadIdx.x] = float(Xa - fl);
  }
  __syncthreads();
  for (unsigned t = unsigned(sl) * blockDim.x + threadIdx.x; t < b.tot; t += unsigned(slabs) * blockDim.x) {
    int p[3];
    b.node(t, p[0], p[1], p[2]);
    float d2 = 0.f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int rel = wrap_rel((p[a] - Xi[a]) % dims[a], dims[a]);
      float dd = fabsf(float(rel) - Xf[a]);
      dd = fminf(dd, float(dims[a]) - dd);  // the nearer image, also half a box away
      d2 += dd * dd;
    }
    if (d2 < lim * lim) near[site(d, p[0], p[1], p[2])] = 1;
  }
}

template <typename T>
__global__ void k_surface(Dims d, const double *__restrict__ cx, const double *__restrict__ cr,
                          const uint8_t *__restrict__ solid, const int *__restrict__ owner,
                          uint8_t *__restrict__ surface, int *__restrict__ count, T *__restrict__ psi_s,
                          int slabs) {
  const int j = blockIdx.x / slabs, sl = blockIdx.x - j * slabs;
  const double X[3] = {cx[3 * j], cx[3 * j + 1], cx[3 * j + 2]};
  const SphereBox b = block_box(d, X, cr[j], 1.0);
  int mine = 0;
  for (unsigned t = unsigned(sl) * blockDim.x + threadIdx.x; t < b.tot; t += unsigned(slabs) * blockDim.x) {
    int x, y, z;
    b.node(t, x, y, z);
    const long long i = site(d, x, y, z);
    if (psi_s[i] > T(1)) psi_s[i] = T(1);
    if (!solid[i] || owner[i] != j) continue;
    long long nb[19];
    neighbours19(d, x, y, z, nb);
    bool any = false;
    for (int q = 1; q < 19; ++q) any |= !solid[nb[q]];
    if (any) {
      surface[i] = 1;
      ++mine;
    }
  }
  atomicAdd(count + j, mine);  // integer: exact in any order
}

template <typename T>
__global__ void k_charge(Dims d, const double *__restrict__ cx, const double *__restrict__ cr,
                         const double *__restrict__ cq, const uint8_t *__restrict__ surface,
                         const int *__restrict__ owner, const int *__restrict__ count, T *__restrict__ qc,
                         int slabs) {
  const int j = blockIdx.x / slabs, sl = blockIdx.x - j * slabs;
  const double X[3] = {cx[3 * j], cx[3 * j + 1], cx[3 * j + 2]};
  const SphereBox b = block_box(d, X, cr[j], 1.0);
  __shared__ double val;
  if (threadIdx.x == 0) val = count[j] > 0 ? __ddiv_rn(cq[j], double(count[j])) : 0.0;
  __syncthreads();
  for (unsigned t = unsigned(sl) * blockDim.x + threadIdx.x; t < b.tot; t += unsigned(slabs) * blockDim.x) {
    int x, y, z;
    b.node(t, x, y, z);
    const long long i = site(d, x, y, z);
    if (surface[i] && owner[i] == j) qc[i] = T(val);
  }
}

// eight sites per thread (a byte a thread leaves the pass waiting for issue:
// 67 us at 256^3 in FP32, where its 150 MB take 22)
template <typename T>
__global__ void __launch_bounds__(256) k_psi_f(long long N, const uint8_t *__restrict__ solid,
                                               const T *__restrict__ psi_s, T *__restrict__ psi_f) {
  const long long i = 8 * (blockIdx.x * (long long)blockDim.x + threadIdx.x);
  if (i + 8 <= N) {
    struct alignas(16) V {
      T v[16 / sizeof(T)];
    };
    constexpr int W = 16 / sizeof(T);
    const uint2 m = *reinterpret_cast<const uint2 *>(solid + i);
#pragma unroll
    for (int k = 0; k < 8; k += W) {
      V p = *reinterpret_cast<const V *>(psi_s + i + k);
#pragma unroll
      for (int c = 0; c < W; ++c) {
        const unsigned s = ((k + c < 4 ? m.x : m.y) >> (8 * ((k + c) & 3))) & 255u;
        p.v[c] = s ? T(0) : T(1) - p.v[c];
      }
      *reinterpret_cast<V *>(psi_f + i + k) = p;
    }
    return;
  }
  for (long long k = i; k < N; ++k) psi_f[k] = solid[k] ? T(0) : T(1) - psi_s[k];
}

template <typename T> static void build(Ctx &c) {
  const long long N = c.d.N;
  cudaMemsetAsync(c.solid, 0, N, c.s);
  cudaMemsetAsync(c.surface, 0, N, c.s);
  cudaMemsetAsync(c.owner, 0xff, N * sizeof(int), c.s);  // -1
  cudaMemsetAsync(c.psi_s, 0, N * sizeof(T), c.s);
  cudaMemsetAsync(c.qc, 0, N * sizeof(T), c.s);
  if (c.near) cudaMemsetAsync(c.near, 0, N, c.s);
  if (c.ncoll > 0) {
    cudaMemsetAsync(c.ccount, 0, c.ncoll * sizeof(int), c.s);
    const int sl = colloid_slabs(c.ncoll);
    count_launch(), k_project<T><<<c.ncoll * sl, 256, 0, c.s>>>(c.d, c.h, c.cx, c.cr, c.solid, c.owner, (T *)c.psi_s, sl);
    count_launch(), k_near<<<c.ncoll * sl, 256, 0, c.s>>>(c.d, c.cx, c.cr, c.near, sl);
    count_launch(), k_surface<T><<<c.ncoll * sl, 256, 0, c.s>>>(c.d, c.cx, c.cr, c.solid, c.owner, c.surface, c.ccount,
                                                                 (T *)c.psi_s, sl);
    count_launch(), k_charge<T><<<c.ncoll * sl, 256, 0, c.s>>>(c.d, c.cx, c.cr, c.cq, c.surface, c.owner, c.ccount,
                                                                (T *)c.qc, sl);
  }
  count_launch(), k_psi_f<T><<<grid_for((N + 7) / 8, 256), 256, 0, c.s>>>(N, c.solid, (const T *)c.psi_s, (T *)c.psi_f);
  c.geom_empty = c.ncoll == 0;
}

void geometry_build(Ctx &c) {
  if (c.prec == LBEH_FP64)
    build<double>(c);
  else
    build<float>(c);
}

}  // namespace lbeh
