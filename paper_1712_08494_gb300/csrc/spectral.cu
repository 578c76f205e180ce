// Host side of the spectral solve: support test, tables and work arrays of a
// box, choice of the kernel variant, launch.
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "spectral_dev.cuh"

namespace lbeh {
using namespace lbeh_spectral;

struct Spectral {
  int fp64 = 0;
  int grid = 0;
  size_t smem = 0;
  std::vector<void *> allocs;
  void *r = nullptr, *p = nullptr, *q = nullptr, *e = nullptr, *w = nullptr;
  void *code[3] = {nullptr, nullptr, nullptr}, *tw[3] = {nullptr, nullptr, nullptr};
  void *sym[3] = {nullptr, nullptr, nullptr};
  LinePlan plan[3];
  int W[3] = {0, 0, 0}, lgW[3] = {0, 0, 0}, K[3] = {0, 0, 0};
  int code_at[3] = {0, 0, 0}, tw_at[3] = {0, 0, 0}, s_at[3] = {0, 0, 0};
  int ncode = 0, ntw = 0, ns = 0;
  double eps_ref = 1.0;
  bool mix = false;  // an axis that is not 32, 64, 128 or 256
  bool big = false;  // the large form: large_form(), or FP64
};

static const void *variant(const Spectral *s) {
  if (s->fp64) return spectral_kernel_f64(s->mix);
  if (!s->big) return spectral_kernel_f32(s->mix);
  return s->mix ? spectral_kernel_f32_big_mix() : spectral_kernel_f32_big();
}

bool spectral_supported(const Dims &d, int fp64) {
  int rad[kMaxStages];
  const int lim = fp64 ? 256 : kMaxN;
  for (int n : {d.nx, d.ny, d.nz})
    if (n < 2 || n > lim || !plan_radices(n, rad)) return false;
  return true;
}

template <typename T> static bool spectral_setup(Spectral *s, const Dims &d) {
  auto dal = [&](size_t bytes) -> void * {
    void *ptr = nullptr;
    if (!dev_alloc(&ptr, bytes)) return nullptr;
    s->allocs.push_back(ptr);
    return ptr;
  };
  // the five work arrays in one allocation, each start skewed by an odd
  // number of 256-byte lines from the power-of-two strides of the lattice, so
  // that the same site of the five arrays (read and written together by the
  // passes) does not fall into the same L2 sets
  const size_t nb = sizeof(T) * (size_t)d.N;
  const size_t stride = ((nb + 255) & ~size_t(255)) + 97 * 256;
  unsigned char *base = (unsigned char *)dal(5 * stride);
  if (!base) return false;
  s->r = base;
  s->p = base + stride;
  s->q = base + 2 * stride;
  s->e = base + 3 * stride;
  s->w = base + 4 * stride;
  const int ns[3] = {d.nx, d.ny, d.nz};
  s->big = sizeof(T) == 8 || large_form(d.nx, d.ny, d.nz);
  int dev = 0, nsm = 0, coop = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  size_t tiles = 0;
  for (int A = 0; A < 3; ++A) {
    const int n = ns[A];
    std::vector<unsigned> code;
    std::vector<C2<double>> twd;
    if (!build_plan(n, s->plan[A], code, twd, s->big)) return false;
    std::vector<C2<T>> tw(twd.size());
    for (size_t k = 0; k < twd.size(); ++k) tw[k] = C2<T>{T(twd[k].x), T(twd[k].y)};
    s->code_at[A] = s->ncode;
    s->tw_at[A] = s->ntw;
    s->s_at[A] = s->ns;
    s->ncode += (int)code.size();
    s->ntw += (int)tw.size();
    s->ns += n;
    // Lines per tile: the largest of 32, 16, 8 whose tile fits 52 KB (two
    // blocks per SM).  A tile of the x pass holds four arrays (r, q, e, p), one
    // of the y and z passes two (the next tile, or the other side of a stage);
    // 64-byte rows of 16 lines along x keep those passes on whole DRAM bursts
    // up to lines of 384.  FP64 passes along y and z, bound by the FP64 rate of
    // the SMs that have a tile, take fewer lines while there are fewer tiles
    // than SMs: steps of 32 x 32 x 192 2384 -> 1859 us, of 64 x 75 x 64 2742 ->
    // 2230, of 16 x 64 x 64 1687 -> 933, of 32^3 1143 -> 775.
    const size_t arrays = A == 0 ? 4 : 2;
    auto tile = [&](int w) { return arrays * size_t(w / 2) * (n + 1) * sizeof(C2<T>); };
    int W = 32, lg = 5;
    while (W > 8 && (tile(W) > (A == 0 ? 70 : 52) * 1024 ||
                     (sizeof(T) == 8 && A != 0 && tile_count(Grid3{d.nx, d.ny, d.nz}, A, W) < nsm))) {
      W /= 2;
      --lg;
    }
    s->W[A] = W;
    s->lgW[A] = lg;
    tiles = std::max(tiles, tile(W));
    // symbols 2 (1 - cos(2 pi k / n)) in the axis's storage order: slot
    // l + 32 kappa of a register-transformed axis holds frequency
    // kappa + K bitrev5(l)
    std::vector<T> sy(n);
    const int K = s->K[A] = reg_fft_k(n, s->big, sizeof(T) == 8);
    for (int j = 0; j < n; ++j) {
      int k = j;
      if (K) {
        int br = 0;
        for (int b = 0; b < 5; ++b) br |= ((j & 31) >> b & 1) << (4 - b);
        k = (j >> 5) + K * br;
      }
      sy[j] = T(2.0 * (1.0 - std::cos(2.0 * M_PI * double(k) / double(n))));
    }
    if (!(s->code[A] = dal(4 * code.size())) || !(s->tw[A] = dal(sizeof(C2<T>) * tw.size())) ||
        !(s->sym[A] = dal(sizeof(T) * n)))
      return false;
    if (cudaMemcpy(s->code[A], code.data(), 4 * code.size(), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(s->tw[A], tw.data(), sizeof(C2<T>) * tw.size(), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(s->sym[A], sy.data(), sizeof(T) * n, cudaMemcpyHostToDevice) != cudaSuccess)
      return false;
  }
  // layout of smem_layout(): plans, codes, twiddles, symbols, tile buffers (16-byte aligned parts)
  auto al = [](size_t b) { return (b + 15) & ~size_t(15); };
  const size_t smem = al(3 * sizeof(LinePlan)) + al((size_t)s->ncode * 4) + al((size_t)s->ntw * sizeof(C2<T>)) +
                      al((size_t)s->ns * sizeof(T)) + (size_t)3 * 32 * kLaneTw * sizeof(C2<T>) + tiles;
  s->smem = smem;
  s->mix = false;
  for (int K : s->K) s->mix |= K != 1 && K != 2 && K != 4 && K != 8;
  const void *kern = variant(s);
  if (!raise_smem_limit(kern, smem)) return false;
  cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  if (!coop || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, kSB, smem) != cudaSuccess ||
      per < 1) {
    cudaGetLastError();
    return false;
  }
  s->grid = nsm * std::min(per, 4);
  return true;
}

Spectral *spectral_create(const Ctx &c, int fp64, double eps_ref) {
  if (!spectral_supported(c.d, fp64)) return nullptr;
  Spectral *s = new Spectral;
  s->fp64 = fp64;
  s->eps_ref = eps_ref;
  const bool ok = fp64 ? spectral_setup<double>(s, c.d) : spectral_setup<float>(s, c.d);
  if (!ok) {
    spectral_destroy(s);
    return nullptr;
  }
  return s;
}

void spectral_destroy(Spectral *s) {
  if (!s) return;
  for (void *a : s->allocs) cudaFree(a);
  delete s;
}

template <typename T> static int launch(Spectral *s, const Ctx &c, const PArgs<T> &pa, cudaStream_t st) {
  SArgs<T> a{};
  a.pa = pa;
  Level<T> L0;
  L0.nx = c.d.nx;
  L0.ny = c.d.ny;
  L0.nz = c.d.nz;
  L0.N = c.d.N;
  L0.eps = (const T *)c.eps;
  L0.b = (T *)s->r;
  a.L0 = L0;
  for (int A = 0; A < 3; ++A) {
    AxisDev<T> &X = a.ax[A];
    X.P = s->plan[A];
    X.W = s->W[A];
    X.K = s->K[A];
    X.lgW = s->lgW[A];
    X.ld = s->plan[A].n + 1;
    X.code = (const unsigned *)s->code[A];
    X.tw = (const C2<T> *)s->tw[A];
    X.s = (const T *)s->sym[A];
    X.code_at = s->code_at[A];
    X.tw_at = s->tw_at[A];
    X.s_at = s->s_at[A];
  }
  a.ncode = s->ncode;
  a.ntw = s->ntw;
  a.ns = s->ns;
  a.g = Grid3{c.d.nx, c.d.ny, c.d.nz};
  a.r = (T *)s->r;
  a.p = (T *)s->p;
  a.q = (T *)s->q;
  a.e = (T *)s->e;
  a.w = (T *)s->w;
  a.inv_eref_n = T(1.0 / (s->eps_ref * double(c.d.N)));
  // rows of nx words start on 16-byte boundaries (arrays 256-byte aligned)
  a.xrows = s->K[0] != 0 && (c.d.nx * sizeof(T)) % 16 == 0;
  if (cudaMemsetAsync(pa.bar, 0, sizeof(Bar), st) != cudaSuccess) return -1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(s->grid);
  cfg.blockDim = dim3(kSB);
  cfg.dynamicSmemBytes = s->smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  count_launch();
  void *args[] = {(void *)&a};
  return cudaLaunchKernelExC(&cfg, variant(s), args) == cudaSuccess ? 0 : -1;
}

int spectral_launch_f64(Spectral *s, const Ctx &c, const PArgs<double> &pa, cudaStream_t st) {
  return launch<double>(s, c, pa, st);
}
int spectral_launch_f32(Spectral *s, const Ctx &c, const PArgs<float> &pa, cudaStream_t st) {
  return launch<float>(s, c, pa, st);
}
int spectral_grid(const Spectral *s) { return s->grid; }

}  // namespace lbeh
