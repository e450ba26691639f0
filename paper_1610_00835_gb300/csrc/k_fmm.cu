// Interpolation-based FMM of Section 3.3 (Fong-Darve; Eqs. EQ: CHEB,
// EQ:Kernel Approx, EQ: SUMMATION, EQ: M2L, EQ: L2L) as an assembled operator
// for 2D grids, with every kernel evaluation cached, as the paper does for
// its GMRES iterations.
//
// y = A s for the M-iii matrix A: the near field (each leaf and its 3 x 3
// neighbourhood of leaves) from the entries A_jk themselves, the far field
// through Chebyshev interpolation of
//     K(x, y) = h^2 exp(-tau(x, y)) / (2 pi |x - y|)
// on a quadtree (leaves of b x b cells, n = 2^L b, b >= 8 and as small as the
// factors of two allow; level l has 2^l x 2^l boxes, far field from l = 2):
//     P2M  W_leaf = P s_leaf                      P [p^2][b^2]  = S_p(leaf cell, node)
//     M2M  W_parent = sum_q C_q W_child(q)        C_q [p^2][p^2] = S_p(parent^{-1} child node, node)
//     M2L  L_B = sum_{C in IL(B)} K_BC W_C        K_BC [p^2][p^2]: 27 blocks per box
//     L2L  L_child(q) += C_q^T L_parent
//     L2P  y_leaf += P^T L_leaf
// S_p is Eq. EQ: CHEB with the first-kind points cos((2i - 1) pi / (2p)); P
// and C_q do not depend on the box or the level, so they are built once on
// the host in FP64.  The interaction list IL(B) is the 27 children of the
// neighbours of B's parent that are not neighbours of B; its offsets depend
// only on B's position in its parent.  tau between Chebyshev nodes is the
// S-step midpoint march of the bilinear sigma_t with the sample points
// clamped to the hull of the cell centres (nodes near the boundary lie
// outside it).  Setup fills the near blocks and the M2L blocks on the device
// (FP32); an apply is the source kernel and 2 L - 2 launches (L = 2: 3) of small
// dense products that read the cached blocks once (M2L of all levels in one of them).
#include <math.h>

#include <algorithm>
#include <vector>

#include "vie_internal.cuh"

namespace vie {

namespace {

constexpr int kIL = 27;  // interaction-list slots per box

// far-field offsets (dx, dy) of the interaction list of a box at position
// (qx, qy) in its parent: x in [-2 - qx, 3 - qx], y likewise, minus the 3 x 3
__host__ __device__ __forceinline__ void il_offset(int qx, int qy, int slot, int *dx, int *dy) {
  int k = 0;
  for (int oy = -2 - qy; oy <= 3 - qy; ++oy)
    for (int ox = -2 - qx; ox <= 3 - qx; ++ox) {
      if (ox >= -1 && ox <= 1 && oy >= -1 && oy <= 1) continue;
      if (k == slot) {
        *dx = ox;
        *dy = oy;
        return;
      }
      ++k;
    }
  *dx = *dy = 0;
}

// bilinear sigma_t~ at lattice coordinates (cell centre j at (ix, iy)),
// clamped to [0, n - 1]; s is the (n + 1)^2 padded lattice
__device__ __forceinline__ float sample_clamped(const float *__restrict__ s, int n, int P, float gx, float gy) {
  gx = fminf(fmaxf(gx, 0.f), (float)(n - 1));
  gy = fminf(fmaxf(gy, 0.f), (float)(n - 1));
  const float fx = floorf(gx), fy = floorf(gy);
  const int ix = (int)fx, iy = (int)fy;
  const float ax = gx - fx, ay = gy - fy;
  const float *r0 = s + (long)iy * P + ix;
  const float lo = fmaf(ax, r0[1] - r0[0], r0[0]);
  const float hi = fmaf(ax, r0[P + 1] - r0[P], r0[P]);
  return fmaf(ay, hi - lo, lo);
}

// h^2 e^{-tau} / (2 pi r) between lattice points a and b (cells; r > 0)
__device__ __forceinline__ float kernel_entry(const float *__restrict__ sig, int n, int P, int S, int closed,
                                              float sigma_c, float ax, float ay, float bx, float by) {
  const float h = 1.0f / (float)n;
  const float dx = bx - ax, dy = by - ay;
  const float r = sqrtf(dx * dx + dy * dy);
  float tau;
  if (closed) {
    tau = sigma_c * h * r;
  } else {
    float acc0 = 0.f, acc1 = 0.f;
    const float inv = 1.0f / (float)S;
    int i = 0;
    for (; i + 1 < S; i += 2) {
      const float t0 = ((float)i + 0.5f) * inv, t1 = ((float)i + 1.5f) * inv;
      acc0 += sample_clamped(sig, n, P, fmaf(t0, dx, ax), fmaf(t0, dy, ay));
      acc1 += sample_clamped(sig, n, P, fmaf(t1, dx, ax), fmaf(t1, dy, ay));
    }
    if (i < S) acc0 += sample_clamped(sig, n, P, fmaf(((float)i + 0.5f) * inv, dx, ax), fmaf(((float)i + 0.5f) * inv, dy, ay));
    tau = h * r * inv * (acc0 + acc1);
  }
  return h * expf(-tau) / (2.0f * 3.14159265358979f * r);
}

struct FillArgs {
  const float *sig;     // padded FP32 sigma_t lattice, (n + 1)^2
  const double *diag;   // self cells
  int n, P, S, closed;
  float sigma_c;
};

// near blocks, stored transposed: near[leaf][slot][k][j] (slot = (oy+1)*3 + ox+1)
__global__ void k_fmm_near_fill(FillArgs a, int L, int b, float *__restrict__ near) {
  const int nl = 1 << L, bb = b * b;
  const long total = (long)nl * nl * 9 * bb * bb;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total; e += (long)gridDim.x * blockDim.x) {
    const int j = (int)(e % bb);
    long t = e / bb;
    const int k = (int)(t % bb);
    t /= bb;
    const int slot = (int)(t % 9);
    const long leaf = t / 9;
    const int bx = (int)(leaf % nl), by = (int)(leaf / nl);
    const int cx = bx + slot % 3 - 1, cy = by + slot / 3 - 1;
    float v = 0.f;
    if (cx >= 0 && cx < nl && cy >= 0 && cy < nl) {
      const int jx = bx * b + j % b, jy = by * b + j / b;
      const int kx = cx * b + k % b, ky = cy * b + k / b;
      if (jx == kx && jy == ky)
        v = (float)a.diag[(long)jy * a.n + jx];
      else
        v = kernel_entry(a.sig, a.n, a.P, a.S, a.closed, a.sigma_c, (float)jx, (float)jy, (float)kx, (float)ky);
    }
    near[e] = v;
  }
}

// M2L blocks of one level: m2l[box][slot][m'][m] (transposed: for each source
// node m', the p^2 target rows contiguous)
__global__ void k_fmm_m2l_fill(FillArgs a, int level, int p, const float *__restrict__ z, float *__restrict__ m2l) {
  const int nb = 1 << level, P2 = p * p;
  const long total = (long)nb * nb * kIL * P2 * P2;
  const float w = (float)a.n / (float)nb;  // box side in cells
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total; e += (long)gridDim.x * blockDim.x) {
    const int m = (int)(e % P2);
    long t = e / P2;
    const int mp = (int)(t % P2);
    t /= P2;
    const int slot = (int)(t % kIL);
    const long box = t / kIL;
    const int bx = (int)(box % nb), by = (int)(box / nb);
    int ox, oy;
    il_offset(bx & 1, by & 1, slot, &ox, &oy);
    const int cx = bx + ox, cy = by + oy;
    float v = 0.f;
    if (cx >= 0 && cx < nb && cy >= 0 && cy < nb) {
      // node positions in lattice coordinates (cell centre j at index j)
      const float tx = bx * w + 0.5f * w * (z[m % p] + 1.f) - 0.5f;
      const float ty = by * w + 0.5f * w * (z[m / p] + 1.f) - 0.5f;
      const float sx = cx * w + 0.5f * w * (z[mp % p] + 1.f) - 0.5f;
      const float sy = cy * w + 0.5f * w * (z[mp / p] + 1.f) - 0.5f;
      v = kernel_entry(a.sig, a.n, a.P, a.S, a.closed, a.sigma_c, tx, ty, sx, sy);
    }
    m2l[e] = v;
  }
}

// P2M and M2M are small dense products whose matrix is the same for every box:
// a thread takes one (box, node m), a CTA kBoxThreads / P2 boxes, and the
// matrix is read transposed, so that a warp's loads are consecutive (with one
// CTA of 128 threads per box and the rows m apart, 36 threads worked and every
// load touched 32 lines: 34 us for P2M and 9 us per M2M level at 512^2, order
// 6; now 6.6 and 7 us).
constexpr int kBoxThreads = 256;

// boxes per CTA, `floats` of shared memory each (at most 48 KB in all), and
// fewer where that leaves less than a CTA for each of about 152 SMs (P2M of 256
// leaves at order 2: 12 us with 64 boxes per CTA, 4.9 so)
inline int boxes_per_cta(int P2, int floats, long boxes) {
  return (int)std::max(1L, std::min({(long)(kBoxThreads / P2), 12288L / floats, boxes / 152}));
}

// P2M: W[leaf][m] = sum_k Pt[k][m] s_leaf[k]
__global__ void __launch_bounds__(kBoxThreads) k_fmm_p2m(int n, int L, int b, int P2, int G,
                                                         const float *__restrict__ Pt, const float *__restrict__ s,
                                                         float *__restrict__ W) {
  extern __shared__ float sh[];  // [G][b^2]
  const int nl = 1 << L, bb = b * b;
  const int box0 = blockIdx.x * G, cnt = min(G, nl * nl - box0);
  for (int i = threadIdx.x; i < cnt * bb; i += blockDim.x) {
    const int box = box0 + i / bb, k = i % bb, bx = box % nl, by = box / nl;
    sh[i] = s[(long)(by * b + k / b) * n + bx * b + k % b];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < cnt * P2; i += blockDim.x) {
    const int q = i / P2, m = i % P2;
    const float *v = sh + q * bb;
    float acc = 0.f;
#pragma unroll 8
    for (int k = 0; k < bb; ++k) acc = fmaf(__ldg(Pt + k * P2 + m), v[k], acc);
    W[(long)(box0 + q) * P2 + m] = acc;
  }
}

// M2M: parent boxes at level l from their children at l + 1; Ct[q][m'][m]
__global__ void __launch_bounds__(kBoxThreads) k_fmm_m2m(int level, int P2, int G, int staged,
                                                         const float *__restrict__ Ct,
                                                         const float *__restrict__ Wc, float *__restrict__ Wp) {
  extern __shared__ float sh[];  // [G][4][P2], then Ct when it fits (staged)
  const int nb = 1 << level;
  const int box0 = blockIdx.x * G, cnt = min(G, nb * nb - box0);
  for (int i = threadIdx.x; i < cnt * 4 * P2; i += blockDim.x) {
    const int box = box0 + i / (4 * P2), q = (i / P2) & 3, mp = i % P2, bx = box % nb, by = box / nb;
    const long child = (long)(2 * by + q / 2) * (2 * nb) + 2 * bx + q % 2;
    sh[i] = Wc[child * P2 + mp];
  }
  // the matrix at once: the sums run term by term, and each term's load from L2
  // would be waited for a few at a time
  float *mat = sh + G * 4 * P2;
  if (staged)
#pragma unroll 8
    for (int i = threadIdx.x; i < 4 * P2 * P2; i += blockDim.x) mat[i] = __ldg(Ct + i);
  __syncthreads();
  for (int i = threadIdx.x; i < cnt * P2; i += blockDim.x) {
    const int g = i / P2, m = i % P2;
    const float *v = sh + g * 4 * P2;
    float acc = 0.f;
    if (staged) {
#pragma unroll 8
      for (int k = 0; k < 4 * P2; ++k) acc = fmaf(mat[k * P2 + m], v[k], acc);
    } else {
#pragma unroll 24
      for (int k = 0; k < 4 * P2; ++k) acc = fmaf(__ldg(Ct + (long)k * P2 + m), v[k], acc);
    }
    Wp[(long)(box0 + g) * P2 + m] = acc;
  }
}

// Streaming product of the two big kernels: thread t = (part, column) of
// parts x C threads adds blk[(part + q parts) C + column] sh[part + q parts]
// over q, in four chains (q = 0, 1, 2, 3 mod 4; what is left over after the
// last whole four goes to the first).  The block is read once from HBM: a
// thread keeps a batch of eight loads in flight while it works on the batch
// before, and the first batch is issued before the sources are gathered into
// shared memory (StreamDot::start), so that the gather's latency hides behind
// it.  Four loads and the gather first: 4.5 TB/s for M2L, 5.2 for the leaves
// at 512^2 (170 and 117 us); now 6.5 and 5.7 (117 and 106).
struct StreamDot {
  static constexpr int kBatch = 8;
  const float *p;   // this thread's next element
  long step;        // parts * C
  int left;         // elements of this thread not yet loaded
  int src, parts;   // this thread's next source, and the distance to the one after
  float v[kBatch];
  __device__ __forceinline__ void load() {
#pragma unroll
    for (int i = 0; i < kBatch; ++i) v[i] = i < left ? __ldcs(p + i * step) : 0.f;
    p += kBatch * step;
  }
  __device__ __forceinline__ void start(const float *blk, int C, int parts_, int part, int column, int I, bool on) {
    parts = parts_;
    step = (long)parts * C;
    p = blk + (long)part * C + column;
    left = on && part < I ? (I - part + parts - 1) / parts : 0;
    src = part;
    load();
  }
  // the four chains, to be added as (a0 + a1) + (a2 + a3)
  __device__ __forceinline__ void run(const float *sh, float (&a)[4]) {
#pragma unroll
    for (int c = 0; c < 4; ++c) a[c] = 0.f;
    while (left >= kBatch) {
      float u[kBatch];
#pragma unroll
      for (int i = 0; i < kBatch; ++i) u[i] = v[i];
      left -= kBatch;
      load();
#pragma unroll
      for (int i = 0; i < kBatch; ++i) a[i & 3] = fmaf(u[i], sh[src + i * parts], a[i & 3]);
      src += kBatch * parts;
    }
    const int whole = left & ~3;
#pragma unroll
    for (int i = 0; i < kBatch; ++i)
      if (i < left) {
        const float x = sh[src + i * parts];
        if (i < whole)
          a[i & 3] = fmaf(v[i], x, a[i & 3]);
        else
          a[0] = fmaf(v[i], x, a[0]);
      }
  }
};

// M2L of every level in one launch (the levels do not depend on each other):
// CTA t takes box t - first[l] of the level l with first[l] <= t < first[l + 1],
// the small coarse levels first, so that their latency hides behind the
// streaming of the large fine level.  Lc[B] = sum over the interaction list of
// K_BC W_C.
struct M2LArgs {
  int L;
  long first[32];     // first CTA of each level
  long node_off[32];  // W and Lc offsets of each level
  long m2l_off[32];   // M2L block offsets of each level
};

__global__ void k_fmm_m2l(M2LArgs a, int P2, const float *__restrict__ m2l_all, const float *__restrict__ W_all,
                          float *__restrict__ Lc_all) {
  extern __shared__ float sh[];
  int level = 2;
  while (level < a.L && (long)blockIdx.x >= a.first[level + 1]) ++level;
  const long box = (long)blockIdx.x - a.first[level];
  const float *W = W_all + a.node_off[level];
  float *Lc = Lc_all + a.node_off[level];
  const int nb = 1 << level;
  const int bx = (int)(box % nb), by = (int)(box / nb);
  // blockDim / P2 groups of P2 threads each take every parts-th source node
  const int parts = blockDim.x / P2, m = threadIdx.x % P2, part = threadIdx.x / P2;
  StreamDot dot;
  dot.start(m2l_all + a.m2l_off[level] + box * kIL * P2 * P2, P2, parts, part, m, kIL * P2, part < parts);
  for (int i = threadIdx.x; i < kIL * P2; i += blockDim.x) {
    const int slot = i / P2, mp = i % P2;
    int ox, oy;
    il_offset(bx & 1, by & 1, slot, &ox, &oy);
    const int cx = bx + ox, cy = by + oy;
    sh[i] = (cx >= 0 && cx < nb && cy >= 0 && cy < nb) ? W[((long)cy * nb + cx) * P2 + mp] : 0.f;
  }
  __syncthreads();
  float *red = sh + kIL * P2;
  float c[4];
  dot.run(sh, c);
  red[threadIdx.x] = (c[0] + c[1]) + (c[2] + c[3]);
  __syncthreads();
  if (threadIdx.x < P2) {
    float t = 0.f;
    for (int q = 0; q < parts; ++q) t += red[q * P2 + threadIdx.x];
    Lc[box * P2 + threadIdx.x] = t;
  }
}

// L2L: child boxes at level l + 1 take their parent's interpolated L
__global__ void __launch_bounds__(kBoxThreads) k_fmm_l2l(int level, int P2, int G, const float *__restrict__ Cq,
                                                         const float *__restrict__ Lp, float *__restrict__ Lch) {
  extern __shared__ float sh[];  // [G][P2]
  const int nc = 2 << level;  // children per side
  const int box0 = blockIdx.x * G, cnt = min(G, nc * nc - box0);
  for (int i = threadIdx.x; i < cnt * P2; i += blockDim.x) {
    const int box = box0 + i / P2, cx = box % nc, cy = box / nc;
    sh[i] = Lp[((long)(cy >> 1) * (nc >> 1) + (cx >> 1)) * P2 + i % P2];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < cnt * P2; i += blockDim.x) {
    const int g = i / P2, mp = i % P2, box = box0 + g;
    const float *C = Cq + (long)((box % nc & 1) + 2 * (box / nc & 1)) * P2 * P2 + mp;
    const float *v = sh + g * P2;
    float acc = 0.f;
#pragma unroll 4
    for (int m = 0; m < P2; ++m) acc = fmaf(__ldg(C + (long)m * P2), v[m], acc);
    Lch[(long)box * P2 + mp] += acc;
  }
}

// leaves: near field from the cached blocks plus L2P of the leaf's own far
// field and its parent's (the L2L step of the leaf level, taken here); y (FP64)
// by op
__global__ void k_fmm_leaf(int n, int L, int b, int P2, const float *__restrict__ near, const float *__restrict__ Pm,
                           const float *__restrict__ s, const float *__restrict__ Lc, const float *__restrict__ Lp,
                           const float *__restrict__ Cq, int op, const double *__restrict__ g,
                           double *__restrict__ y) {
  extern __shared__ float sh[];  // [9][b^2] sources, then [P2] L, [P2] the parent's
  const int nl = 1 << L, bb = b * b;
  const int bx = blockIdx.x % nl, by = blockIdx.x / nl;
  // blockDim / bb groups of bb threads each take every parts-th source cell;
  // group 0 adds the far field (L2P)
  const int parts = blockDim.x / bb, j = threadIdx.x % bb, part = threadIdx.x / bb;
  StreamDot dot;
  dot.start(near + (long)blockIdx.x * 9 * bb * bb, bb, parts, part, j, 9 * bb, part < parts);
  float *far = sh + 9 * bb, *up = far + P2, *red = up + P2;
  for (int m = threadIdx.x; m < P2; m += blockDim.x) {
    far[m] = Lc[(long)blockIdx.x * P2 + m];
    if (Lp) up[m] = Lp[((long)(by >> 1) * (nl >> 1) + (bx >> 1)) * P2 + m];
  }
  for (int i = threadIdx.x; i < 9 * bb; i += blockDim.x) {
    const int slot = i / bb, k = i % bb;
    const int cx = bx + slot % 3 - 1, cy = by + slot / 3 - 1;
    sh[i] = (cx >= 0 && cx < nl && cy >= 0 && cy < nl) ? s[(long)(cy * b + k / b) * n + cx * b + k % b] : 0.f;
  }
  __syncthreads();
  if (Lp) {
    const float *C = Cq + (long)((bx & 1) + 2 * (by & 1)) * P2 * P2;
    for (int mp = threadIdx.x; mp < P2; mp += blockDim.x) {
      float acc = 0.f;
#pragma unroll 18
      for (int m = 0; m < P2; ++m) acc = fmaf(__ldg(C + (long)m * P2 + mp), up[m], acc);
      far[mp] += acc;
    }
    __syncthreads();
  }
  float c[4];
  dot.run(sh, c);
  if (part == 0) {
#pragma unroll 4
    for (int m = 0; m < P2; ++m) c[1] = fmaf(__ldg(Pm + m * bb + j), far[m], c[1]);
  }
  red[threadIdx.x] = (c[0] + c[1]) + (c[2] + c[3]);
  __syncthreads();
  if (threadIdx.x < bb) {
    double v = 0.0;
    for (int q = 0; q < parts; ++q) v += (double)red[q * bb + threadIdx.x];
    const long jj = (long)(by * b + threadIdx.x / b) * n + bx * b + threadIdx.x % b;
    y[jj] = op == VIE_OP_I_MINUS_K ? g[jj] - v : v;
  }
}

// ---- host: the interpolation matrices in FP64

double s1(int p, double u, double v) {
  u = std::min(1.0, std::max(-1.0, u));
  const double tu = acos(u), tv = acos(v);
  double acc = 1.0 / p;
  for (int k = 1; k < p; ++k) acc += 2.0 / p * cos(k * tu) * cos(k * tv);
  return acc;
}

int blocks_for(long total) { return (int)std::max(1L, std::min((total + 255) / 256, 152L * 64)); }

}  // namespace

void fmm_leaf_levels(int n, int *L, int *b) {
  int l = 0;
  while (n % (2 << l) == 0 && n / (2 << l) >= 8) ++l;
  *L = l;
  *b = n >> l;
}

vie_status fmm_prepare(FmmPlan *fp, int n, int p, const float *sig32, const double *diag, int steps, int closed,
                       double sigma_c, cudaStream_t st) {
  fmm_release(fp);
  int L, b;
  fmm_leaf_levels(n, &L, &b);
  if (L < 2) {
    set_error("vie_assemble_fmm: the grid has no far field (n must be 2^L b with L >= 2 and b >= 8)");
    return VIE_ERR_UNSUPPORTED;
  }
  if (p < 2 || p > 12) {
    set_error("vie_assemble_fmm: order must be in 2..12");
    return VIE_ERR_INVALID_ARG;
  }
  const int P2 = p * p, bb = b * b, nl = 1 << L;
  std::vector<double> z(p);
  for (int i = 0; i < p; ++i) z[i] = cos((2.0 * (i + 1) - 1.0) * kPi / (2.0 * p));
  // P[m][k]: leaf cell k = kx + b ky at u = 2 (kx + 1/2) / b - 1
  std::vector<float> Pm((size_t)P2 * bb), Cq((size_t)4 * P2 * P2), Pt(Pm.size()), Ct(Cq.size()), zf(p);
  for (int m = 0; m < P2; ++m)
    for (int k = 0; k < bb; ++k) {
      const double u = 2.0 * (k % b + 0.5) / b - 1.0, v = 2.0 * (k / b + 0.5) / b - 1.0;
      Pm[(size_t)m * bb + k] = (float)(s1(p, u, z[m % p]) * s1(p, v, z[m / p]));
    }
  // C_q[m][m']: child q's node m' in its parent's coordinates
  for (int q = 0; q < 4; ++q)
    for (int m = 0; m < P2; ++m)
      for (int mp = 0; mp < P2; ++mp) {
        const double u = -1.0 + (q % 2) + 0.5 * (z[mp % p] + 1.0);
        const double v = -1.0 + (q / 2) + 0.5 * (z[mp / p] + 1.0);
        Cq[((size_t)q * P2 + m) * P2 + mp] = (float)(s1(p, u, z[m % p]) * s1(p, v, z[m / p]));
      }
  for (int i = 0; i < p; ++i) zf[i] = (float)z[i];
  for (int m = 0; m < P2; ++m) {
    for (int k = 0; k < bb; ++k) Pt[(size_t)k * P2 + m] = Pm[(size_t)m * bb + k];
    for (int q = 0; q < 4; ++q)
      for (int mp = 0; mp < P2; ++mp)
        Ct[((size_t)q * P2 + mp) * P2 + m] = Cq[((size_t)q * P2 + m) * P2 + mp];
  }
  fp->n = n;
  fp->p = p;
  fp->L = L;
  fp->b = b;
  long nodes = 0;
  for (int l = 2; l <= L; ++l) {
    fp->node_off[l] = nodes;
    nodes += (long)P2 << (2 * l);
  }
  long m2l_total = 0;
  for (int l = 2; l <= L; ++l) {
    fp->m2l_off[l] = m2l_total;
    m2l_total += ((long)kIL * P2 * P2) << (2 * l);
  }
  const long near_total = (long)nl * nl * 9 * bb * bb;
  VIE_CUDA(vie_malloc((void **)&fp->near, sizeof(float) * near_total));
  VIE_CUDA(vie_malloc((void **)&fp->m2l, sizeof(float) * m2l_total));
  VIE_CUDA(vie_malloc((void **)&fp->W, sizeof(float) * nodes));
  VIE_CUDA(vie_malloc((void **)&fp->Lc, sizeof(float) * nodes));
  VIE_CUDA(vie_malloc((void **)&fp->Pm, sizeof(float) * Pm.size()));
  VIE_CUDA(vie_malloc((void **)&fp->Cq, sizeof(float) * Cq.size()));
  VIE_CUDA(vie_malloc((void **)&fp->Pt, sizeof(float) * Pt.size()));
  VIE_CUDA(vie_malloc((void **)&fp->Ct, sizeof(float) * Ct.size()));
  VIE_CUDA(vie_malloc((void **)&fp->z, sizeof(float) * p));
  VIE_CUDA(cudaMemcpyAsync(fp->Pm, Pm.data(), sizeof(float) * Pm.size(), cudaMemcpyHostToDevice, st));
  VIE_CUDA(cudaMemcpyAsync(fp->Cq, Cq.data(), sizeof(float) * Cq.size(), cudaMemcpyHostToDevice, st));
  VIE_CUDA(cudaMemcpyAsync(fp->Pt, Pt.data(), sizeof(float) * Pt.size(), cudaMemcpyHostToDevice, st));
  VIE_CUDA(cudaMemcpyAsync(fp->Ct, Ct.data(), sizeof(float) * Ct.size(), cudaMemcpyHostToDevice, st));
  VIE_CUDA(cudaMemcpyAsync(fp->z, zf.data(), sizeof(float) * p, cudaMemcpyHostToDevice, st));
  FillArgs a{sig32, diag, n, n + 1, steps, closed, (float)sigma_c};
  k_fmm_near_fill<<<blocks_for(near_total), 256, 0, st>>>(a, L, b, fp->near);
  VIE_CHECK_LAUNCH("k_fmm_near_fill");
  for (int l = 2; l <= L; ++l) {
    const long cnt = ((long)kIL * P2 * P2) << (2 * l);
    k_fmm_m2l_fill<<<blocks_for(cnt), 256, 0, st>>>(a, l, p, fp->z, fp->m2l + fp->m2l_off[l]);
    VIE_CHECK_LAUNCH("k_fmm_m2l_fill");
  }
  VIE_CUDA(cudaStreamSynchronize(st));
  fp->near_floats = near_total;
  fp->m2l_floats = m2l_total;
  fp->on = 1;
  return VIE_OK;
}

void fmm_release(FmmPlan *fp) {
  if (fp->near) vie_free(fp->near);
  if (fp->m2l) vie_free(fp->m2l);
  if (fp->W) vie_free(fp->W);
  if (fp->Lc) vie_free(fp->Lc);
  if (fp->Pm) vie_free(fp->Pm);
  if (fp->Cq) vie_free(fp->Cq);
  if (fp->Pt) vie_free(fp->Pt);
  if (fp->Ct) vie_free(fp->Ct);
  if (fp->z) vie_free(fp->z);
  *fp = FmmPlan{};
}

vie_status fmm_apply(const FmmPlan &fp, int op, const float *s, const double *g, double *y, cudaStream_t st) {
  const int n = fp.n, L = fp.L, b = fp.b, P2 = fp.p * fp.p, bb = b * b;
  const int nl = 1 << L;
  const int tm = std::max(P2, 256 / P2 * P2), tl = std::max(bb, 256 / bb * bb);
  auto ctas = [](long boxes, int G) { return (unsigned)((boxes + G - 1) / G); };
  // upward pass
  const int gp = boxes_per_cta(P2, bb, (long)nl * nl);
  k_fmm_p2m<<<ctas((long)nl * nl, gp), kBoxThreads, sizeof(float) * gp * bb, st>>>(n, L, b, P2, gp, fp.Pt, s,
                                                                                fp.W + fp.node_off[L]);
  VIE_CHECK_LAUNCH("k_fmm_p2m");
  for (int l = L - 1; l >= 2; --l) {
    const int gm = boxes_per_cta(P2, 4 * P2, 1L << (2 * l));
    const size_t own = sizeof(float) * gm * 4 * P2, mat = sizeof(float) * 4 * P2 * P2;
    const bool staged = own + mat <= 48 * 1024;  // orders up to 7
    k_fmm_m2m<<<ctas(1L << (2 * l), gm), kBoxThreads, own + (staged ? mat : 0), st>>>(
        l, P2, gm, staged, fp.Ct, fp.W + fp.node_off[l + 1], fp.W + fp.node_off[l]);
    VIE_CHECK_LAUNCH("k_fmm_m2m");
  }
  // interactions (all levels in one launch), then the downward pass
  {
    M2LArgs a;
    a.L = L;
    long first = 0;
    for (int l = 2; l <= L; ++l) {
      a.first[l] = first;
      a.node_off[l] = fp.node_off[l];
      a.m2l_off[l] = fp.m2l_off[l];
      first += 1L << (2 * l);
    }
    a.first[L + 1] = first;
    k_fmm_m2l<<<(unsigned)first, tm, sizeof(float) * (kIL * P2 + tm), st>>>(a, P2, fp.m2l, fp.W, fp.Lc);
    VIE_CHECK_LAUNCH("k_fmm_m2l");
  }
  // the leaves take their own L2L step: a launch fewer, hidden behind other leaves'
  // near fields.  Per apply with it and as a launch of its own: 42.0 and 46.2 us at
  // 128^2 (256 leaves) and 86.8 and 87.5 at 256^2 (1024) at order 4, 62.1 and 66.2,
  // 121.4 and 126.5, and 287 and 293 at 512^2 (4096) at order 6
  const bool fused = L > 2;
  for (int l = 2; l < (fused ? L - 1 : L); ++l) {
    const int gl = boxes_per_cta(P2, P2, 4L << (2 * l));
    k_fmm_l2l<<<ctas(4L << (2 * l), gl), kBoxThreads, sizeof(float) * gl * P2, st>>>(
        l, P2, gl, fp.Cq, fp.Lc + fp.node_off[l], fp.Lc + fp.node_off[l + 1]);
    VIE_CHECK_LAUNCH("k_fmm_l2l");
  }
  k_fmm_leaf<<<nl * nl, tl, sizeof(float) * (9 * bb + 2 * P2 + tl), st>>>(
      n, L, b, P2, fp.near, fp.Pm, s, fp.Lc + fp.node_off[L], fused ? fp.Lc + fp.node_off[L - 1] : nullptr, fp.Cq,
      op, g, y);
  VIE_CHECK_LAUNCH("k_fmm_leaf");
  return VIE_OK;
}

}  // namespace vie
