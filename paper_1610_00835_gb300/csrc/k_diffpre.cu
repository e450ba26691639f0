// Diffusion preconditioner of Section 4.4 (Eq. EQ:DA), 2D.
//
// Diffusion approximation on the unit square: -div(kappa grad U) + mu_a U = f
// with kappa = 1 / (d mu), mu_a = mu - mu_s, and U + l dU/dn = 0 on the
// boundary, l = 2 / (d mu) (d = 2).  Second-order finite volumes on the n x n
// cells: an interior face carries the harmonic mean of its cells' kappa and
// the flux kappa_f (U_c - U_nb) / h; a boundary face eliminates the boundary
// value through the Robin condition, leaving the outward flux
// 2 kappa_c U_c / (h + 2 l_c).  Per cell area, row c of D is
//     diag_c U_c - sum_nb a_nb U_nb,  a_nb = kappa_f / h^2,
//     diag_c = mu_a,c + sum a_nb + (boundary faces) 2 kappa_c / (h (h + 2 l_c)).
//
// As the right preconditioner of (I - K) U = b it applies
//     M(r) = r + D^{-1}(sigma_s r)
// (the diffusion limit of A is (D + Sigma_s)^{-1}, so (I - A Sigma_s)^{-1} is
// close to I + D^{-1} Sigma_s), with D^{-1} one V-cycle of geometric
// multigrid from a zero guess: levels n, n/2, ... while the size is even and
// above 8 (coarse mu and mu_s the means of the 2 x 2 children, the operator
// rediscretised); red-black Gauss-Seidel, 2 sweeps before and after the
// correction; restriction = mean of the children's residuals; bilinear
// prolongation in the cell centres; 200 red-black sweeps on the coarsest
// grid.  FP64 (the grids are small).
//
// One launch per level and direction.  A CTA owns a kTile x kTile tile of the
// level and keeps it with a halo in shared memory, so that its four colour
// half-sweeps (and the residual, or the interpolated correction) need no data
// from other CTAs: every half-sweep updates a region one cell smaller on each
// side, cells in the halos being recomputed by their neighbours' CTAs with the
// same arithmetic.  What bounds a level is launch latency and the SM's narrow
// FP64 pipe (tile 16: 2.2 times the cells in the first half-sweep, but 64 CTAs
// at 128^2; tile 32 leaves 16 CTAs with three times the work each).  A launch
// per colour (50 in a graph) took 2.3 us each, 100 us per V-cycle at 128^2.
//
// The coarsest grid's sweeps from zero are a fixed linear map f -> u.  Up to
// kMapCells cells it is set up as a matrix (the sweeps applied to the unit
// vectors, once per medium: 60 us for 8 x 8 cells, 0.6 ms for 25 x 25) and
// applied as one product: 200 sweeps in one CTA
// took 160 us of each V-cycle at 128^2 (an 8 x 8 grid).  Larger coarsest grids
// (odd sizes of 27 and more) run the sweeps on tiles, kCoarseSweeps / 4
// launches of four.
// Measured at 128^2 (five levels): 40 us per V-cycle in 9 launches; 265 us
// in 50 before.
#include <math.h>

#include <algorithm>
#include <vector>

#include "vie_internal.cuh"

namespace vie {

namespace {

constexpr int kCoarseSweeps = 200;
constexpr int kT = 256;
constexpr int kTile = 16;        // tile side of the smoothing kernels (even: colours and children align)
constexpr int kMapCells = 625;   // largest coarsest grid (25 x 25) kept as a matrix: 3.1 MB, set up in half a ms

__device__ __forceinline__ double neighbour_sum(const double *__restrict__ c, const double *__restrict__ u, int n,
                                               long N, int ix, int iy, long j) {
  double s = 0.0;
  if (ix > 0) s += c[N + j] * u[j - 1];
  if (ix < n - 1) s += c[2 * N + j] * u[j + 1];
  if (iy > 0) s += c[3 * N + j] * u[j - n];
  if (iy < n - 1) s += c[4 * N + j] * u[j + n];
  return s;
}

// A CTA's tile with a halo of M cells: local cell (lx, ly) of the S x S
// region is cell (x0 + lx, y0 + ly) of the level.
template <int M>
struct Tile {
  static constexpr int S = kTile + 2 * M;
  int n, x0, y0;
  __device__ __forceinline__ Tile(int n_) : n(n_), x0((int)blockIdx.x * kTile - M), y0((int)blockIdx.y * kTile - M) {}
  __device__ __forceinline__ bool inside(int x, int y) const { return x >= 0 && x < n && y >= 0 && y < n; }
  // the coupled neighbours of local cell l, in neighbour_sum's order
  __device__ __forceinline__ double sum(const double *__restrict__ c, const double *U, int x, int y, int l) const {
    const long N = (long)n * n, j = (long)y * n + x;
    double s = 0.0;
    if (x > 0) s += c[N + j] * U[l - 1];
    if (x < n - 1) s += c[2 * N + j] * U[l + 1];
    if (y > 0) s += c[3 * N + j] * U[l - S];
    if (y < n - 1) s += c[4 * N + j] * U[l + S];
    return s;
  }
  // one colour of a red-black Gauss-Seidel sweep (red: x + y even) on the
  // cells at least `m` from the region's edge; plane 5 of c holds 1 / diag
  __device__ __forceinline__ void half_sweep(const double *__restrict__ c, const double *F, double *U, int colour,
                                             int m) const {
    const int w = S - 2 * m, half = (w + 1) / 2;
    for (int i = threadIdx.x; i < w * half; i += kT) {
      const int ly = m + i / half, first = (x0 + m + y0 + ly + colour) & 1;
      const int lx = m + 2 * (i % half) + first;
      const int x = x0 + lx, y = y0 + ly;
      if (lx >= S - m || !inside(x, y)) continue;
      const int l = ly * S + lx;
      U[l] = (F[l] + sum(c, U, x, y, l)) * c[5L * n * n + (long)y * n + x];
    }
    __syncthreads();
  }
};

// Down: two sweeps from zero, u, and f_coarse = mean over the 2 x 2 children
// of the residual f - D u.  Finest level: f = ss v (f null).
__global__ void __launch_bounds__(kT) k_dp_down(int n, const double *__restrict__ c, const double *__restrict__ f,
                                                const double *__restrict__ ss, const double *__restrict__ v,
                                                double *__restrict__ u, double *__restrict__ fc) {
  using T = Tile<4>;
  __shared__ double F[T::S * T::S], U[T::S * T::S], R[kTile * kTile];
  const T t(n);
  const long N = (long)n * n;
  for (int l = threadIdx.x; l < T::S * T::S; l += kT) {
    const int x = t.x0 + l % T::S, y = t.y0 + l / T::S;
    double fl = 0.0, ul = 0.0;
    if (t.inside(x, y)) {
      const long j = (long)y * n + x;
      fl = f ? f[j] : ss[j] * v[j];
      if (((x + y) & 1) == 0) ul = fl * c[5 * N + j];  // the first red half-sweep: all neighbours still zero
    }
    F[l] = fl;
    U[l] = ul;
  }
  __syncthreads();
  t.half_sweep(c, F, U, 1, 1);
  t.half_sweep(c, F, U, 0, 2);
  t.half_sweep(c, F, U, 1, 3);
  static_assert(kTile * kTile == kT, "one thread per cell of the tile");
  {
    const int lx = 4 + threadIdx.x % kTile, ly = 4 + threadIdx.x / kTile, l = ly * T::S + lx;
    const int x = t.x0 + lx, y = t.y0 + ly;
    double r = 0.0;
    if (t.inside(x, y)) {
      const long j = (long)y * n + x;
      u[j] = U[l];
      r = F[l] - (c[j] * U[l] - t.sum(c, U, x, y, l));
    }
    R[threadIdx.x] = r;
  }
  __syncthreads();
  constexpr int H = kTile / 2;
  if (threadIdx.x < H * H) {
    const int a = threadIdx.x % H, b = threadIdx.x / H, nc = n / 2;
    const int I = (int)blockIdx.x * H + a, J = (int)blockIdx.y * H + b;
    const double *q = R + 2 * b * kTile + 2 * a;
    if (I < nc && J < nc) fc[(long)J * nc + I] = 0.25 * (q[0] + q[1] + q[kTile] + q[kTile + 1]);
  }
}

// Up: u plus the bilinear interpolation of the coarse correction e (a
// neighbour outside the coarse grid replaced by the coarse cell itself), then
// two sweeps, into w.  Finest level: f = ss v (f null) and w = v + the result.
__global__ void __launch_bounds__(kT) k_dp_up(int n, const double *__restrict__ c, const double *__restrict__ f,
                                              const double *__restrict__ ss, const double *__restrict__ v,
                                              const double *__restrict__ u, const double *__restrict__ e,
                                              double *__restrict__ w) {
  using T = Tile<4>;
  __shared__ double F[T::S * T::S], U[T::S * T::S];
  const T t(n);
  const int nc = n / 2;
  for (int l = threadIdx.x; l < T::S * T::S; l += kT) {
    const int x = t.x0 + l % T::S, y = t.y0 + l / T::S;
    double fl = 0.0, ul = 0.0;
    if (t.inside(x, y)) {
      const long j = (long)y * n + x;
      fl = f ? f[j] : ss[j] * v[j];
      const int I = x >> 1, J = y >> 1;
      const int I2 = (x & 1) ? min(I + 1, nc - 1) : max(I - 1, 0);
      const int J2 = (y & 1) ? min(J + 1, nc - 1) : max(J - 1, 0);
      ul = u[j] + (9.0 * e[(long)J * nc + I] + 3.0 * e[(long)J * nc + I2] + 3.0 * e[(long)J2 * nc + I] +
                   e[(long)J2 * nc + I2]) / 16.0;
    }
    F[l] = fl;
    U[l] = ul;
  }
  __syncthreads();
  t.half_sweep(c, F, U, 0, 1);
  t.half_sweep(c, F, U, 1, 2);
  t.half_sweep(c, F, U, 0, 3);
  t.half_sweep(c, F, U, 1, 4);
  const int lx = 4 + threadIdx.x % kTile, ly = 4 + threadIdx.x / kTile;
  const int x = t.x0 + lx, y = t.y0 + ly;
  if (t.inside(x, y)) {
    const long j = (long)y * n + x;
    const double r = U[ly * T::S + lx];
    w[j] = f ? r : v[j] + r;
  }
}

// Four sweeps on a large coarsest grid: u (null: zero) -> w.
__global__ void __launch_bounds__(kT) k_dp_sweeps(int n, const double *__restrict__ c, const double *__restrict__ f,
                                                  const double *__restrict__ u, double *__restrict__ w) {
  using T = Tile<8>;
  __shared__ double F[T::S * T::S], U[T::S * T::S];
  const T t(n);
  for (int l = threadIdx.x; l < T::S * T::S; l += kT) {
    const int x = t.x0 + l % T::S, y = t.y0 + l / T::S;
    const bool in = t.inside(x, y);
    const long j = (long)y * n + x;
    F[l] = in ? f[j] : 0.0;
    U[l] = in && u ? u[j] : 0.0;
  }
  __syncthreads();
  for (int s = 0; s < 8; ++s) t.half_sweep(c, F, U, s & 1, s + 1);
  const int lx = 8 + threadIdx.x % kTile, ly = 8 + threadIdx.x / kTile;
  const int x = t.x0 + lx, y = t.y0 + ly;
  if (t.inside(x, y)) w[(long)y * n + x] = U[ly * T::S + lx];
}

// The coarsest grid's map, column by column: CTA k runs kCoarseSweeps
// red-black sweeps from zero on the unit vector of cell k into G[k][.].  Thread t
// owns cells 2 t and 2 t + 1, one of each colour, with their couplings times
// 1 / diagonal in registers; u lies in shared memory with a border of zeros, so
// that a half-sweep is four multiply-adds and a barrier.  The FP64 pipe bounds
// it on large grids (25 x 25: 0.5 ms for 3.1e8 multiply-adds), the chain of
// half-sweeps on small ones.
constexpr int kMapSide = 25;
static_assert(kMapSide * kMapSide == kMapCells, "the border fits");
constexpr int map_threads(int cells) { return ((cells + 1) / 2 + 31) / 32 * 32; }
__global__ void __launch_bounds__(map_threads(kMapCells)) k_dp_coarse_map(int n, const double *__restrict__ c,
                                                                         double *__restrict__ G) {
  __shared__ double U[(kMapSide + 2) * (kMapSide + 2)];
  const int N = n * n, P = n + 2, k = blockIdx.x;  // (N <= kMapCells)
  for (int l = threadIdx.x; l < P * P; l += blockDim.x) U[l] = 0.0;
  int at[2], cell[2];  // by colour: place in U, index
  double w[2][4], b[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int j0 = 2 * threadIdx.x, j = j0 + ((j0 % n + j0 / n + q) & 1), x = j % n, y = j / n;
    cell[q] = j < N ? j : -1;
    at[q] = (y + 1) * P + x + 1;
    b[q] = 0.0;
    if (j < N) {
      const double inv = c[5L * N + j];
      w[q][0] = x > 0 ? c[N + j] * inv : 0.0;
      w[q][1] = x < n - 1 ? c[2 * N + j] * inv : 0.0;
      w[q][2] = y > 0 ? c[3 * N + j] * inv : 0.0;
      w[q][3] = y < n - 1 ? c[4 * N + j] * inv : 0.0;
      if (j == k) b[q] = inv;
    }
  }
  __syncthreads();
  for (int s = 0; s < kCoarseSweeps; ++s)
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      if (cell[q] >= 0) {
        const double *u = U + at[q];
        U[at[q]] = fma(w[q][0], u[-1], fma(w[q][1], u[1], fma(w[q][2], u[-P], fma(w[q][3], u[P], b[q]))));
      }
      __syncthreads();
    }
#pragma unroll
  for (int q = 0; q < 2; ++q)
    if (cell[q] >= 0) G[(long)k * N + cell[q]] = U[at[q]];
}

// u = sum_k f_k G[k][.]: a CTA takes 32 cells, its 8 warps every 8th k, and
// warp 0 adds the warps' sums in order.  f = ss v and u = v + the result where
// the coarsest grid is the only one (f null).
__global__ void __launch_bounds__(kT) k_dp_coarse(int N, const double *__restrict__ G, const double *__restrict__ f,
                                                  const double *__restrict__ ss, const double *__restrict__ v,
                                                  double *__restrict__ u) {
  __shared__ double part[kT];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, j = blockIdx.x * 32 + lane;
  double s = 0.0;
  if (j < N) {
#pragma unroll 4
    for (int k = warp; k < N; k += kT / 32) s += (f ? f[k] : ss[k] * v[k]) * G[(long)k * N + j];
  }
  part[threadIdx.x] = s;
  __syncthreads();
  if (warp == 0 && j < N) {
    for (int q = 1; q < kT / 32; ++q) s += part[q * 32 + lane];
    u[j] = f ? s : v[j] + s;
  }
}

__global__ void k_dp_source(long N, const double *__restrict__ ss, const double *__restrict__ v,
                            double *__restrict__ f) {
  for (long j = blockIdx.x * (long)blockDim.x + threadIdx.x; j < N; j += (long)gridDim.x * blockDim.x)
    f[j] = ss[j] * v[j];
}

__global__ void k_dp_finish(long N, const double *__restrict__ v, const double *__restrict__ e,
                            double *__restrict__ z) {
  for (long j = blockIdx.x * (long)blockDim.x + threadIdx.x; j < N; j += (long)gridDim.x * blockDim.x)
    z[j] = v[j] + e[j];
}

int blocks_for(long N) { return (int)std::max(1L, std::min((N + kT - 1) / kT, 2048L)); }

// the coefficient planes of an n x n level with cell values mu, mu_a (FP64, host)
void level_coefficients(int n, const std::vector<double> &mu, const std::vector<double> &mua,
                        std::vector<double> &c) {
  const long N = (long)n * n;
  const double h = 1.0 / n;
  c.assign(6 * N, 0.0);
  for (int iy = 0; iy < n; ++iy)
    for (int ix = 0; ix < n; ++ix) {
      const long j = (long)iy * n + ix;
      const double kc = 1.0 / (2.0 * mu[j]), lc = 2.0 / (2.0 * mu[j]);
      double diag = mua[j];
      const int nx[4] = {ix - 1, ix + 1, ix, ix}, ny[4] = {iy, iy, iy - 1, iy + 1};
      for (int q = 0; q < 4; ++q) {
        if (nx[q] >= 0 && nx[q] < n && ny[q] >= 0 && ny[q] < n) {
          const double kn = 1.0 / (2.0 * mu[(long)ny[q] * n + nx[q]]);
          const double a = 2.0 * kc * kn / (kc + kn) / (h * h);
          c[(q + 1) * N + j] = a;
          diag += a;
        } else {
          diag += 2.0 * kc / (h * (h + 2.0 * lc));
        }
      }
      c[j] = diag;
      c[5 * N + j] = 1.0 / diag;
    }
}

}  // namespace

vie_status diffusion_prepare(DiffPre *dp, int n, const double *sigma_t, const double *sigma_s,
                             const double *sigma_s_dev, cudaStream_t st) {
  diffusion_release(dp);
  const long N = (long)n * n;
  std::vector<double> mu(sigma_t, sigma_t + N), mua((size_t)N);
  for (long j = 0; j < N; ++j) {
    if (!(sigma_t[j] > 0.0)) {
      set_error("vie_set_diffusion_preconditioner: sigma_t must be > 0 in every cell (kappa = 1 / (2 sigma_t))");
      return VIE_ERR_INVALID_ARG;
    }
    mua[j] = sigma_t[j] - sigma_s[j];
  }
  std::vector<double> c;
  int ln = n;
  for (;;) {
    level_coefficients(ln, mu, mua, c);
    const long M = (long)ln * ln;
    DiffLevel &L = dp->lv[dp->L++];  // owned by dp from here: released on failure
    L.n = ln;
    VIE_CUDA(vie_malloc((void **)&L.c, sizeof(double) * 6 * M));
    VIE_CUDA(vie_malloc((void **)&L.f, sizeof(double) * M));
    VIE_CUDA(vie_malloc((void **)&L.u, sizeof(double) * M));
    VIE_CUDA(vie_malloc((void **)&L.w, sizeof(double) * M));
    VIE_CUDA(cudaMemcpyAsync(L.c, c.data(), sizeof(double) * 6 * M, cudaMemcpyHostToDevice, st));
    VIE_CUDA(cudaStreamSynchronize(st));
    if (ln % 2 || ln <= 8 || dp->L == kDiffMaxLevels) break;
    const int nc = ln / 2;
    std::vector<double> mc((size_t)nc * nc), ac((size_t)nc * nc);
    for (int J = 0; J < nc; ++J)
      for (int I = 0; I < nc; ++I) {
        const long a = (long)(2 * J) * ln + 2 * I, b = a + ln;
        mc[(long)J * nc + I] = 0.25 * (mu[a] + mu[b] + mu[a + 1] + mu[b + 1]);
        ac[(long)J * nc + I] = 0.25 * (mua[a] + mua[b] + mua[a + 1] + mua[b + 1]);
      }
    mu.swap(mc);
    mua.swap(ac);
    ln = nc;
  }
  dp->ss = sigma_s_dev;
  dp->n = n;
  const DiffLevel &C = dp->lv[dp->L - 1];
  const int Nc = C.n * C.n;
  if (Nc <= kMapCells) {
    VIE_CUDA(vie_malloc((void **)&dp->map, sizeof(double) * (size_t)Nc * Nc));
    k_dp_coarse_map<<<Nc, map_threads(Nc), 0, st>>>(C.n, C.c, dp->map);
    VIE_CHECK_LAUNCH("k_dp_coarse_map");
    // applies may come on another stream
    VIE_CUDA(cudaStreamSynchronize(st));
  }
  dp->on = 1;
  return VIE_OK;
}

void diffusion_release(DiffPre *dp) {
  if (dp->map) vie_free(dp->map);
  for (int l = 0; l < dp->L; ++l) {
    if (dp->lv[l].c) vie_free(dp->lv[l].c);
    if (dp->lv[l].f) vie_free(dp->lv[l].f);
    if (dp->lv[l].u) vie_free(dp->lv[l].u);
    if (dp->lv[l].w) vie_free(dp->lv[l].w);
  }
  *dp = DiffPre{};
}

vie_status diffusion_precondition(const DiffPre &dp, const double *v, double *z, cudaStream_t st) {
  const DiffLevel *lv = dp.lv;
  const int L = dp.L;
  auto tiles = [](int n) { return dim3((unsigned)((n + kTile - 1) / kTile), (unsigned)((n + kTile - 1) / kTile)); };
  for (int l = 0; l + 1 < L; ++l) {
    k_dp_down<<<tiles(lv[l].n), kT, 0, st>>>(lv[l].n, lv[l].c, l ? lv[l].f : nullptr, dp.ss, v, lv[l].u,
                                             lv[l + 1].f);
    VIE_CHECK_LAUNCH("k_dp_down");
  }
  const DiffLevel &C = lv[L - 1];
  const int Nc = C.n * C.n;
  const double *e = C.u;  // the level's result, read by the level above
  if (dp.map) {
    k_dp_coarse<<<(Nc + 31) / 32, kT, 0, st>>>(Nc, dp.map, L > 1 ? C.f : nullptr, dp.ss, v, L > 1 ? C.u : z);
    VIE_CHECK_LAUNCH("k_dp_coarse");
    if (L == 1) return VIE_OK;
  } else {
    if (L == 1) {
      k_dp_source<<<blocks_for(Nc), kT, 0, st>>>(Nc, dp.ss, v, C.f);
      VIE_CHECK_LAUNCH("k_dp_source");
    }
    for (int s = 0; s < kCoarseSweeps; s += 4) {
      double *out = (s / 4) % 2 ? C.w : C.u;
      k_dp_sweeps<<<tiles(C.n), kT, 0, st>>>(C.n, C.c, C.f, s ? e : nullptr, out);
      VIE_CHECK_LAUNCH("k_dp_sweeps");
      e = out;
    }
    if (L == 1) {
      k_dp_finish<<<blocks_for(Nc), kT, 0, st>>>(Nc, v, e, z);
      VIE_CHECK_LAUNCH("k_dp_finish");
      return VIE_OK;
    }
  }
  for (int l = L - 2; l >= 0; --l) {
    double *out = l ? lv[l].w : z;
    k_dp_up<<<tiles(lv[l].n), kT, 0, st>>>(lv[l].n, lv[l].c, l ? lv[l].f : nullptr, dp.ss, v, lv[l].u, e, out);
    VIE_CHECK_LAUNCH("k_dp_up");
    e = out;
  }
  return VIE_OK;
}

}  // namespace vie
