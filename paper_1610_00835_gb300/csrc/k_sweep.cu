// Step two of Algorithm 1 (S.3): the scattering-free transport solve along
// backward characteristics, Eq. EQ:ERT Intgrl with q = Q = sigma_s U + f:
//   Phi(x, v) = int_0^L exp(-int_0^l sigma_t(x - l' v) dl') Q(x - l v) dl,
// L the distance from x to the boundary along -v.  One thread per
// (direction, cell) ray.  The ray is cut into ns = ceil(2 n L - 1e-6) equal
// steps (at most h/2 each); the step count is decided in FP64 with
// correctly rounded operations so that it does not depend on instruction
// selection.  On each step sigma_t~ and Q~ (bilinear / trilinear in the cell
// values, clamped to the hull of the centres) are frozen at the step midpoint
// and the step is integrated exactly:
//   Phi += e^{-tau} Q~ (1 - e^{-sigma~ D}) / sigma~,  tau += sigma~ D.
//
// What bounds it is the L1 data path (85 % of its wavefronts at 32^3, 65 % of the
// issue slots): the corners of a warp's points lie in several rows of cells, and a
// step reads eight of them.  So the loads are few and the step is short:
//  * sigma_t and Q sit side by side in one lattice with a ghost layer (edge
//    copies), so that no coordinate needs clamping, a corner is one 8-byte load
//    for both, and the two interpolations run as packed FP32 pairs; floors are
//    FP32 additions of 1.5 2^23 instead of conversions (which have a sixteenth
//    of the add's rate);
//  * with x = sigma~ D and g(x) = (1 - e^{-x}) / x the step adds e^{-tau} Q~ D g:
//    up to x = 1/2 g is its Taylor polynomial of degree 7 (truncation below
//    1.1e-8), without expm1f and the division; thicker steps take those.
//    (The transmission is expf of the summed tau: the hardware exponential
//    rounds tau log2(e), 2.6e-6 at an optical depth of 60, for 4 % of the time;
//    e^{-tau} times 1 - x g saves nothing in 3D and rounds 10 % worse.)
// The FP64 set-up of a ray (an exit length per axis with a division each, the
// step count) depends on the direction and one coordinate: a CTA takes a tile
// of cells and one direction and computes it once per coordinate of the tile
// (20 instead of 768 in 3D; per ray it kept the FP64 pipe busy for 0.8 ms).  A
// warp is 8 x 4 cells: a row of 32 leaves lanes idle where the exit lies across
// the row (76 % of the lanes' steps used at 32^3 on 128 directions; 85 %).
// Measured at 32^3: 527 us for 128 directions (1040 before), error against FP64
// unchanged (1.42e-7).
#include <math.h>

#include <algorithm>

#include "vie_internal.cuh"

namespace vie {

namespace {

// (sigma_t, Q = sigma_s U + f) on the cells with a ghost layer of edge copies,
// (n + 2)^dim points
__global__ void k_make_q(int dim, int n, const double *__restrict__ st, const double *__restrict__ ss,
                         const double *__restrict__ U, const double *__restrict__ f, float2 *__restrict__ lat) {
  const long P = n + 2;
  const long total = dim == 2 ? P * P : P * P * P;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < total; i += (long)gridDim.x * blockDim.x) {
    const long px = min(max(i % P - 1, 0L), (long)n - 1), py = min(max((i / P) % P - 1, 0L), (long)n - 1);
    const long pz = dim == 3 ? min(max(i / (P * P) - 1, 0L), (long)n - 1) : 0;
    const long j = (pz * n + py) * n + px;
    lat[i] = make_float2((float)st[j], (float)(ss[j] * U[j] + f[j]));
  }
}

typedef unsigned long long u64;
__device__ __forceinline__ u64 both(float w) {
  u64 r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(w));
  return r;
}
// a + w (b - a) in both halves
__device__ __forceinline__ u64 lerp2(u64 a, u64 b, u64 w) {
  u64 d, r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(both(-1.f)), "l"(b));
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(w), "l"(d), "l"(a));
  return r;
}

// cell index of a lattice coordinate c >= 0 and its weight (at an integer it
// may be the cell below with weight 1: the same value)
__device__ __forceinline__ int cell_of(float c, float &w) {
  const float y = (c - 0.5f) + 12582912.0f;  // 1.5 * 2^23
  w = c - (y - 12582912.0f);
  return __float_as_int(y) - 0x4B400000;
}

// (sigma_t~, Q~) at ghosted lattice coordinates u + 1
template <int DIM>
__device__ __forceinline__ float2 interp(const u64 *__restrict__ lat, unsigned P, const float *c) {
  float ax, ay, az;
  const unsigned ix = cell_of(c[0], ax), iy = cell_of(c[1], ay);
  const unsigned b0 = DIM == 3 ? (cell_of(c[2], az) * P + iy) * P + ix : iy * P + ix;
  const u64 wx = both(ax), wy = both(ay);
  const u64 *r0 = lat + b0, *r1 = lat + (b0 + P);
  u64 v = lerp2(lerp2(__ldg(r0), __ldg(r0 + 1), wx), lerp2(__ldg(r1), __ldg(r1 + 1), wx), wy);
  if (DIM == 3) {
    const unsigned b2 = b0 + P * P;
    const u64 *r2 = lat + b2, *r3 = lat + (b2 + P);
    const u64 hi = lerp2(lerp2(__ldg(r2), __ldg(r2 + 1), wx), lerp2(__ldg(r3), __ldg(r3 + 1), wx), wy);
    v = lerp2(v, hi, both(az));
  }
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}

constexpr int kSweepThreads = 256;
// the tile of cells of a CTA
template <int DIM>
struct SweepTile {
  static constexpr int X = DIM == 2 ? 16 : 8, Y = DIM == 2 ? 16 : 8, Z = DIM == 2 ? 1 : 4;
  static constexpr int coords = DIM == 2 ? X + Y : X + Y + Z;
};

// a ray that leaves the domain across one axis: its length, steps, step length
// and the step in cells
struct Exit {
  long long key;  // the length's bits: lengths are >= 0, so they compare as integers
  int ns;
  float dl, du[3];
};

template <int DIM>
__global__ void __launch_bounds__(kSweepThreads) k_sweep(int n, long tiles, const u64 *__restrict__ lat,
                                                         const float *__restrict__ dirs, int M,
                                                         float *__restrict__ Phi) {
  using T = SweepTile<DIM>;
  __shared__ Exit exits[T::coords];
  const long N = DIM == 2 ? (long)n * n : (long)n * n * n;
  const int tx = (n + T::X - 1) / T::X, ty = (n + T::Y - 1) / T::Y;
  const unsigned P = n + 2;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // cells of this thread in the tile: a warp is 8 x 4
  const int cx = (lane & 7) + (DIM == 2 ? 8 * (warp & 1) : 0);
  const int cy = (lane >> 3) + (DIM == 2 ? 4 * (warp >> 1) : 4 * (warp & 1));
  const int cz = DIM == 2 ? 0 : warp >> 1;
  for (long item = blockIdx.x; item < tiles * M; item += gridDim.x) {
    const int m = (int)(item / tiles), tile = (int)(item % tiles);
    const int x0 = tile % tx * T::X, y0 = tile / tx % ty * T::Y, z0 = DIM == 2 ? 0 : tile / (tx * ty) * T::Z;
    __syncthreads();
    if (threadIdx.x < T::coords) {
      const int t = threadIdx.x;
      const int d = t < T::X ? 0 : t < T::X + T::Y ? 1 : 2;
      const int idx = d == 0 ? x0 + t : d == 1 ? y0 + t - T::X : z0 + t - T::X - T::Y;
      const double h = 1.0 / n;
      const double x = __dmul_rn(__dadd_rn((double)idx, 0.5), h), v = (double)dirs[m * DIM + d];
      double L = INFINITY;
      if (v > 0.0) L = __ddiv_rn(x, v);
      else if (v < 0.0) L = fmax(0.0, __ddiv_rn(__dsub_rn(1.0, x), -v));  // coordinates past the grid: unused
      // |v| = 1 gives L <= sqrt(dim); the cap only bounds the loop for
      // directions that are not unit vectors (undefined input).
      if (!(L <= 2.0)) L = 2.0;
      const double steps = ceil(__dsub_rn(__dmul_rn(L, 2.0 * n), 1e-6));
      Exit e;
      e.key = __double_as_longlong(L);
      e.ns = steps < 1.0 ? 1 : (int)steps;
      e.dl = (float)(L / (double)e.ns);
#pragma unroll
      for (int k = 0; k < DIM; ++k) {
        // the coordinates stay on the lattice: |L v| is at most the way to the
        // boundary; a non-finite direction (undefined input) stands still
        const float du = (float)(-(double)e.dl * (double)dirs[m * DIM + k] * n);
        e.du[k] = fabsf(du) < 1e30f ? du : 0.f;
      }
      exits[t] = e;
    }
    __syncthreads();
    const int jx = x0 + cx, jy = y0 + cy, jz = z0 + cz;
    if (jx >= n || jy >= n || (DIM == 3 && jz >= n)) continue;
    int which = cx;
    if (exits[T::X + cy].key < exits[which].key) which = T::X + cy;
    if (DIM == 3 && exits[T::X + T::Y + cz].key < exits[which].key) which = T::X + T::Y + cz;
    const Exit &e = exits[which];
    const int ns = e.ns;
    const float dl = e.dl;
    // ghosted lattice coordinates of the midpoints: u + 1 = j + 1 + (s + 1/2) du
    float u0[3] = {(float)(jx + 1), (float)(jy + 1), (float)(jz + 1)}, du[3];
#pragma unroll
    for (int k = 0; k < DIM; ++k) du[k] = e.du[k];
    float tau = 0.f, trans = 1.f, acc = 0.f, t = 0.5f;
    for (int s = 0; s < ns; ++s, t += 1.f) {
      float c[3];
#pragma unroll
      for (int k = 0; k < DIM; ++k) c[k] = fmaf(t, du[k], u0[k]);
      const float2 sq = interp<DIM>(lat, P, c);
      const float x = sq.x * dl;
      if (x <= 0.5f) {
        float g = fmaf(x, -1.f / 40320.f, 1.f / 5040.f);
        g = fmaf(x, g, -1.f / 720.f);  // signs folded: g(x) = sum_k (-x)^k / (k + 1)!
        g = fmaf(x, g, 1.f / 120.f);
        g = fmaf(x, g, -1.f / 24.f);
        g = fmaf(x, g, 1.f / 6.f);
        g = fmaf(x, g, -0.5f);
        g = fmaf(x, g, 1.f);
        acc = fmaf(trans * sq.y, dl * g, acc);
      } else {
        acc = fmaf(trans * sq.y, -expm1f(-x) / sq.x, acc);
      }
      tau = fmaf(sq.x, dl, tau);
      trans = expf(-tau);
    }
    Phi[(long)m * N + ((long)jz * n + jy) * n + jx] = acc;
  }
}

int grid_for(long n, int threads) {
  long b = (n + threads - 1) / threads;
  return (int)(b < 1 ? 1 : (b > 65535 ? 65535 : b));
}

}  // namespace

size_t sweep_lattice_points(int dim, int n) {
  const size_t P = (size_t)n + 2;
  return dim == 2 ? P * P : P * P * P;
}

vie_status launch_make_q(int dim, int n, const double *sigma_t, const double *sigma_s, const double *U,
                         const double *f, float2 *lat, cudaStream_t st) {
  k_make_q<<<grid_for((long)sweep_lattice_points(dim, n), 256), 256, 0, st>>>(dim, n, sigma_t, sigma_s, U, f, lat);
  VIE_CHECK_LAUNCH("k_make_q");
  return VIE_OK;
}

vie_status launch_sweep(int dim, int n, const float2 *lat, const float *dirs, int M, float *Phi, cudaStream_t st) {
  auto up = [n](int t) { return (long)((n + t - 1) / t); };
  const u64 *l = reinterpret_cast<const u64 *>(lat);
  if (dim == 2) {
    const long tiles = up(SweepTile<2>::X) * up(SweepTile<2>::Y);
    k_sweep<2><<<(unsigned)std::min(tiles * M, 1L << 20), kSweepThreads, 0, st>>>(n, tiles, l, dirs, M, Phi);
  } else {
    const long tiles = up(SweepTile<3>::X) * up(SweepTile<3>::Y) * up(SweepTile<3>::Z);
    k_sweep<3><<<(unsigned)std::min(tiles * M, 1L << 20), kSweepThreads, 0, st>>>(n, tiles, l, dirs, M, Phi);
  }
  VIE_CHECK_LAUNCH("k_sweep");
  return VIE_OK;
}

}  // namespace vie
