// FP64 Krylov building blocks for GMRES(m) (Algorithm 1, S.2; Section 5).
//
// Arnoldi uses classical Gram-Schmidt applied twice (CGS2): h = V^T w,
// w -= V h, repeated, so each pass is two bandwidth-bound sweeps over the
// basis instead of k dependent ones.  Dot products are block partials summed
// in a fixed order, so results do not depend on timing.  Givens rotations are
// tiny and run in one thread, the triangular solve in one warp.
//
// One Arnoldi step after the operator apply (both passes, the norm, the
// Givens step and the scaling) is one launch, k_arnoldi: the vectors are
// short (N = 16384: 131 KB), so that separate launches for the dots, the
// updates, the norm and the scaling cost their latency (six, 33 us per step
// at 128^2 with four basis vectors; one launch: 18 us, and 62 instead of 87 us
// for 64 right-hand sides, where the FP64 pipe bounds it).  w stays in
// registers between the passes; the blocks exchange their dot partials
// through global memory at three barriers: a thread-block cluster's hardware
// barrier up to 16 blocks (one cluster per right-hand side), a counter with
// every block resident (cooperative launch) above.  The step's residual
// estimate goes straight to a pinned host slot with a sequence number, which
// the host polls: a copy and a stream synchronisation cost 33 us per step.
#include <math.h>

#include <atomic>

#include "arnoldi_form.cuh"
#include "vie_internal.cuh"

namespace vie {

namespace {

constexpr int kDotThreads = 256;

// Sum of 256 values in shared memory by one warp, valid in lane 0: lane l takes
// values l, l + 32, ... in a tree (a dependent FP64 add costs ~45 cycles here),
// then a shuffle tree.
__device__ __forceinline__ double fold256(const double *red, int lane) {
  double t = ((red[lane] + red[lane + 32]) + (red[lane + 64] + red[lane + 96])) +
             ((red[lane + 128] + red[lane + 160]) + (red[lane + 192] + red[lane + 224]));
  for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
  return t;
}

// Block sum (256 threads) in a fixed order, valid in thread 0: every thread's
// value goes to shared memory and warp 0 folds it.  GB300's FP64 pipe is
// narrow, and a shuffle tree in every warp cost more FP64 adds than the dot
// products.
__device__ __forceinline__ double block_sum(double v, double *red) {
  __syncthreads();  // an earlier call may still be reading red
  red[threadIdx.x] = v;
  __syncthreads();
  return threadIdx.x < 32 ? fold256(red, threadIdx.x) : 0.0;
}

// y = x / sqrt(*n2); a zero norm gives y = 0.
__global__ void k_scale(const double *__restrict__ x, const double *__restrict__ n2, double *__restrict__ y, long N) {
  __shared__ double s_inv;  // one reciprocal square root per block, not per thread
  if (threadIdx.x == 0) s_inv = *n2 > 0.0 ? rsqrt(*n2) : 0.0;
  __syncthreads();
  const double inv = s_inv;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < N; i += (long)gridDim.x * blockDim.x)
    y[i] = x[i] * inv;
}

__global__ void k_axpby(double a, const double *__restrict__ x, double b,
                        const double *__restrict__ y, double *__restrict__ z, long N) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < N; i += (long)gridDim.x * blockDim.x)
    z[i] = a * x[i] + b * y[i];
}

// Sum over the blocks' partials part[q * nv + v] of one v by one warp, valid
// in lane 0: lane l adds blocks l, l + 32, ... in turn, then a shuffle tree.
__device__ __forceinline__ double partials_sum(const double *part, int blocks, int nv, int v, int lane) {
  double s = 0.0;
  for (int q = lane; q < blocks; q += 32) s += __ldcg(part + (long)q * nv + v);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  return s;
}

// Column k of the Hessenberg matrix H ((m+1) x m, column-major): entries
// 0..k from hcol, entry k+1 = sqrt(hk1sq).  Apply the k earlier rotations,
// build rotation k, rotate the residual vector gv, and return
// |gv[k+1]| inv_bnorm.  One thread: a chain of dependent FP64 operations, kept
// short by reciprocal square roots in place of hypot, square root and divides
// (the column's end is scaled by a power of two against overflow).
__device__ double givens_step(double *H, int m, int k, const double *hcol, double hk1sq, double *cs, double *sn,
                              double *gv, double inv_bnorm) {
  double *c = H + (long)k * (m + 1);
  double a = hcol[0];
  for (int i = 0; i < k; ++i) {
    const double b = hcol[i + 1], ci = cs[i], si = sn[i];
    c[i] = ci * a + si * b;
    a = -si * a + ci * b;
  }
  // (an overflowed norm stays infinite: the rotation below and the estimate are NaN)
  const double b = hk1sq > 0.0 && hk1sq <= 1.7976931348623157e308 ? hk1sq * rsqrt(hk1sq) : hk1sq;
  const double big = fmax(fabs(a), fabs(b));
  // 2^-e with 2^e <= big < 2^(e+1), clamped so that it and its inverse are normal
  const int e = max(2, min(2044, (int)((__double_as_longlong(big) >> 52) & 0x7ff)));
  const double down = __longlong_as_double((long long)(2046 - e) << 52);
  const double up = __longlong_as_double((long long)e << 52);
  const double as = a * down, bs = b * down, d2 = as * as + bs * bs;
  const double inv = d2 > 0.0 ? rsqrt(d2) : 0.0;
  const double cc = d2 > 0.0 ? as * inv : 1.0, ss = d2 > 0.0 ? bs * inv : 0.0;
  const double g = gv[k], gn = -ss * g;
  cs[k] = cc;
  sn[k] = ss;
  c[k] = d2 * inv * up;
  c[k + 1] = 0.0;
  gv[k] = cc * g;
  gv[k + 1] = gn;
  return fabs(gn) * inv_bnorm;
}

// Solve the k x k upper-triangular system R y = gv[0..k-1], R = H[0..k-1][0..k-1],
// by columns in one warp: row i in lane i mod 32 (k <= 256), the reciprocal
// diagonal and the next column loaded ahead of the dependent chain.
__device__ void backsolve_warp(const double *__restrict__ H, int m, int k, const double *__restrict__ gv, double *y,
                               int lane) {
  double s[8], inv[8], c[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    const int i = lane + 32 * t;
    s[t] = inv[t] = c[t] = 0.0;
    if (i < k) {
      s[t] = gv[i];
      const double d = H[(long)i * (m + 1) + i];
      inv[t] = d != 0.0 ? 1.0 / d : 0.0;
      c[t] = H[(long)(k - 1) * (m + 1) + i];
    }
  }
  for (int q = k - 1; q >= 0; --q) {
    double next[8], yq = 0.0;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      next[t] = q > 0 && lane + 32 * t < q ? H[(long)(q - 1) * (m + 1) + lane + 32 * t] : 0.0;
      if (t == q >> 5) yq = s[t] * inv[t];
    }
    yq = __shfl_sync(0xffffffffu, yq, q & 31);
    if (lane == 0) y[q] = yq;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      if (lane + 32 * t < q) s[t] -= c[t] * yq;
      c[t] = next[t];
    }
  }
  __syncwarp();
}

constexpr int kRegElems = 4;       // elements of w a thread keeps in registers

// f(Count<1>) .. f(Count<8>) for min(n, 8): the sweeps over up to eight basis
// vectors are compiled for their number (predicated off, the operations of the
// missing ones still took the FP64 pipe: 70 us of a 64-source step at 128^2).
template <int C>
struct Count {
  static constexpr int value = C;
};
template <typename F>
__device__ __forceinline__ void by_count(int n, F &&f) {
  switch (n) {
    case 1: f(Count<1>{}); break;
    case 2: f(Count<2>{}); break;
    case 3: f(Count<3>{}); break;
    case 4: f(Count<4>{}); break;
    case 5: f(Count<5>{}); break;
    case 6: f(Count<6>{}); break;
    case 7: f(Count<7>{}); break;
    default: f(Count<8>{});
  }
}

// how the blocks of one right-hand side wait for one another
enum StepSync { kOneBlock = 0, kCluster = 1, kGridWide = 2 };

// Grid-wide barrier of a cooperative launch: bar counts arrivals, `target` of
// them must have come.  The wait is bounded (a limit of zero gives up at once);
// false: it ran out.  All blocks get the same answer: a block whose time is up
// sets the top bit of the counter, in one atomic step only while arrivals are
// missing, and with the bit set nobody passes.  (Each block deciding for itself,
// one could give up just before the last arrival while the others went on.)
constexpr unsigned kGaveUp = 0x80000000u;
__device__ __forceinline__ bool grid_wait(unsigned *bar, unsigned target, long long limit) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(bar, 1u);
    const long long t0 = clock64();
    unsigned seen = 0;
    if (limit <= 0) seen = atomicOr(bar, kGaveUp) | kGaveUp;
    while (seen < target) {
      seen = atomicAdd(bar, 0u);
      if (seen < target && clock64() - t0 > limit && atomicCAS(bar, seen, seen | kGaveUp) == seen) seen |= kGaveUp;
    }
    __threadfence();
    ok = !(seen & kGaveUp);
  }
  __syncthreads();
  return ok != 0;
}

template <int SYNC>
__device__ __forceinline__ bool step_wait(unsigned *bar, unsigned &target, long long limit) {
  if constexpr (SYNC == kOneBlock) {
    __syncthreads();
    return true;
  } else if constexpr (SYNC == kCluster) {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    return true;
  } else {
    target += gridDim.x;
    return grid_wait(bar, target, limit);
  }
}

// The Arnoldi step of column k of every active right-hand side r (blockIdx.y):
// w = V_r[k + 1] holds the operator's result; on return it is orthogonal to
// V_r[0 .. k] and of unit length, H, the rotations and gv have column k, and
// slot r holds {estimate, error words, sequence number}.  Element i of w
// belongs to thread i mod (256 G) of the G = b.blocks blocks that the sums are
// taken over; a CTA is VB of those blocks in turn (VB = 2 halves the CTAs of a
// large batch: 64 right-hand sides at 128^2 are then one wave).  REG keeps the
// up to kRegElems elements of a thread in registers.
template <int SYNC, bool REG, int VB>
__global__ void __launch_bounds__(kDotThreads, 4) k_arnoldi(KBatch b, double *__restrict__ V, long ldv_r, int k,
                                                            double inv_bnorm1, const int *err0, const int *err1,
                                                            unsigned long long seq, unsigned *bar, WaitLimits wl) {
  static_assert(REG || VB == 1, "one block per CTA without the registers");
  __shared__ double red[8][kDotThreads];
  __shared__ double hs[256], hc[256];
  const int r = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (b.act && !b.act[r]) return;
  const long N = b.N;
  const int m = b.m, nv = k + 1, G = b.blocks;
  double *Vr = V + (long)r * ldv_r;
  double *w = Vr + (long)(k + 1) * N;
  double *partA = b.part + (long)r * 2 * G * (m + 1), *partB = partA + (long)G * (m + 1);
  const long stride = (long)G * kDotThreads;
  double *slot = b.slots + 4 * r;
  unsigned target = 0;
  auto first = [&](int vb) { return ((long)blockIdx.x + (long)vb * gridDim.x) * kDotThreads + tid; };
  double wr[VB][kRegElems];
  if (REG) {
#pragma unroll
    for (int vb = 0; vb < VB; ++vb)
#pragma unroll
      for (int e = 0; e < kRegElems; ++e) {
        const long i = first(vb) + e * stride;
        wr[vb][e] = i < N ? w[i] : 0.0;
      }
  }
  // the block partials of C basis vectors from v0 on: one warp each
  auto fold = [&](double *part, int vb, int v0, const auto &s, auto count) {
    constexpr int C = decltype(count)::value;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < C; ++j) red[j][tid] = s[j];
    __syncthreads();
    if (warp < C) {
      const double t = fold256(red[warp], lane);
      if (lane == 0) part[((long)blockIdx.x + (long)vb * gridDim.x) * nv + v0 + warp] = t;
    }
  };
  auto dots = [&](double *part) {
#pragma unroll
    for (int vb = 0; vb < VB; ++vb) {
      const long i0 = first(vb);
      for (int v0 = 0; v0 < nv; v0 += 8)
        by_count(nv - v0, [&](auto count) {
          constexpr int C = decltype(count)::value;
          double s[C];
#pragma unroll
          for (int j = 0; j < C; ++j) s[j] = 0.0;
          const double *x = Vr + (long)v0 * N;
          if (REG) {
#pragma unroll
            for (int e = 0; e < kRegElems; ++e) {
              const long i = i0 + e * stride;
              if (i < N) {
#pragma unroll
                for (int j = 0; j < C; ++j) s[j] += x[(long)j * N + i] * wr[vb][e];
              }
            }
          } else {
            for (long i = i0; i < N; i += stride) {
              const double wi = w[i];
#pragma unroll
              for (int j = 0; j < C; ++j) s[j] += x[(long)j * N + i] * wi;
            }
          }
          fold(part, vb, v0, s, count);
        });
    }
  };
  // hs = the sums over the blocks, hc the Hessenberg column
  auto sums = [&](const double *part, bool again) {
    for (int v = warp; v < nv; v += 8) {
      const double t = partials_sum(part, G, nv, v, lane);
      if (lane == 0) {
        hs[v] = t;
        hc[v] = again ? hc[v] + t : t;
      }
    }
    __syncthreads();
  };
  // w -= sum_v hs_v V_v
  auto update = [&]() {
    if (REG) {
#pragma unroll
      for (int vb = 0; vb < VB; ++vb)
#pragma unroll
        for (int e = 0; e < kRegElems; ++e) {
          const long i = first(vb) + e * stride;
          if (i < N) {
            double acc = wr[vb][e];
            for (int v = 0; v < nv; ++v) acc -= hs[v] * Vr[(long)v * N + i];
            wr[vb][e] = acc;
          }
        }
    } else {
      for (long i = first(0); i < N; i += stride) {
        double acc = w[i];
        for (int v = 0; v < nv; ++v) acc -= hs[v] * Vr[(long)v * N + i];
        w[i] = acc;
      }
    }
  };
  double n2 = 0.0;
  dots(partA);
  bool ok = step_wait<SYNC>(bar, target, wl.first);
  if (ok) {
    sums(partA, false);
    if (REG && nv <= 8) {
      // the first update and the second dots in one sweep over the basis
      by_count(nv, [&](auto count) {
        constexpr int C = decltype(count)::value;
#pragma unroll
        for (int vb = 0; vb < VB; ++vb) {
          const long i0 = first(vb);
          double s[C];
#pragma unroll
          for (int j = 0; j < C; ++j) s[j] = 0.0;
#pragma unroll
          for (int e = 0; e < kRegElems; ++e) {
            const long i = i0 + e * stride;
            if (i < N) {
              double x[C], acc = wr[vb][e];
#pragma unroll
              for (int j = 0; j < C; ++j) x[j] = Vr[(long)j * N + i];
#pragma unroll
              for (int j = 0; j < C; ++j) acc -= hs[j] * x[j];
#pragma unroll
              for (int j = 0; j < C; ++j) s[j] += x[j] * acc;
              wr[vb][e] = acc;
            }
          }
          fold(partB, vb, 0, s, count);
        }
      });
    } else {
      update();
      dots(partB);
    }
    ok = step_wait<SYNC>(bar, target, wl.limit);
  }
  if (ok) {
    sums(partB, true);
    update();
    // partA again: every block has read it before the second barrier
#pragma unroll
    for (int vb = 0; vb < VB; ++vb) {
      double s = 0.0;
      if (REG) {
#pragma unroll
        for (int e = 0; e < kRegElems; ++e)
          if (first(vb) + e * stride < N) s += wr[vb][e] * wr[vb][e];
      } else {
        for (long i = first(vb); i < N; i += stride) s += w[i] * w[i];
      }
      s = block_sum(s, red[0]);
      if (tid == 0) partA[(long)blockIdx.x + (long)vb * gridDim.x] = s;
    }
    ok = step_wait<SYNC>(bar, target, wl.limit);
  }
  if (ok) {
    if (warp == 0) {
      const double t = partials_sum(partA, G, 1, 0, lane);
      if (lane == 0) {
        hs[0] = t;
        hs[1] = t > 0.0 ? rsqrt(t) : 0.0;
      }
    }
    __syncthreads();
    n2 = hs[0];
  }
  if (blockIdx.x == 0 && tid == 0) {
    double est = __longlong_as_double(0x7ff8000000000000ll);
    if (ok)
      est = givens_step(b.H + (long)r * (m + 1) * m, m, k, hc, n2, b.cs + (long)r * m, b.sn + (long)r * m,
                        b.gv + (long)r * (m + 1), b.inv_bnorm ? b.inv_bnorm[r] : inv_bnorm1);
    volatile double *h = slot;
    volatile int *he = reinterpret_cast<volatile int *>(slot + 1);
    h[0] = est;
    he[0] = err0 ? *err0 : 0;
    he[1] = err1 ? *err1 : 0;
    he[2] = ok ? 0 : 1;
    __threadfence_system();
    *reinterpret_cast<volatile unsigned long long *>(slot + 3) = seq;
  }
  if (ok) {
    const double inv = hs[1];
    if (REG) {
#pragma unroll
      for (int vb = 0; vb < VB; ++vb)
#pragma unroll
        for (int e = 0; e < kRegElems; ++e) {
          const long i = first(vb) + e * stride;
          if (i < N) w[i] = wr[vb][e] * inv;
        }
    } else {
      for (long i = first(0); i < N; i += stride) w[i] = w[i] * inv;
    }
  }
  if (SYNC == kGridWide && tid == 0) {
    // the last block out leaves the counters at zero for the next launch
    __threadfence();
    if (atomicAdd(bar + 1, 1u) == gridDim.x - 1) {
      bar[0] = 0u;
      bar[1] = 0u;
    }
  }
}

// R y = gv, then x += sum_{v < kk} y_v B_v, for every active right-hand side
// (k >= 0: the same column count for all of them, else kk[r])
__global__ void __launch_bounds__(kDotThreads) k_update(KBatch b, const double *__restrict__ B, long ldb_r,
                                                        int k_all, const int *__restrict__ kk,
                                                        double *__restrict__ x, long ldx_r) {
  __shared__ double y[256];
  const int r = blockIdx.y;
  if (b.act && !b.act[r]) return;
  const int k = k_all >= 0 ? k_all : kk[r], m = b.m;
  if (threadIdx.x < 32)
    backsolve_warp(b.H + (long)r * (m + 1) * m, m, k, b.gv + (long)r * (m + 1), y, threadIdx.x);
  __syncthreads();
  const double *Br = B + (long)r * ldb_r;
  double *xr = x + (long)r * ldx_r;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < b.N; i += (long)gridDim.x * blockDim.x) {
    double acc = xr[i];
    for (int v = 0; v < k; ++v) acc += y[v] * Br[(long)v * b.N + i];
    xr[i] = acc;
  }
}

int grid_for(long n, int threads) {
  long b = (n + threads - 1) / threads;
  return (int)(b < 1 ? 1 : (b > 2048 ? 2048 : b));
}

// ---- R solves in lockstep (blockIdx.y = right-hand side r).  Each kernel
// does for every r with act[r] != 0 what its single-vector form above does,
// in the same order, so a batched solve of one right-hand side reproduces
// the single solve's arithmetic.  Vector i of r's basis sits at
// V + r ldv_r + i N; r's small arrays at r times their length.

// More than kMaxCluster blocks per right-hand side: the step as separate
// launches, every sum in k_arnoldi's order.
//
// out1[r][v] = V_r[v] . w_r (v < nv) and/or out2[r][v] += it, by the last block
// of r (an atomic ticket, reset for the next launch); with gvmode the single
// dot (nv = 1, V = w) is ||w_r||^2 and that block then takes r's Givens step of
// column k.
__global__ void __launch_bounds__(kDotThreads) k_bdots_last(KBatch b, const double *__restrict__ V, long ldv_r,
                                                            int nv, const double *__restrict__ w, long ldw_r,
                                                            double *out1, double *out2, int gvmode, int k) {
  __shared__ double red[8][kDotThreads];
  __shared__ int last;
  const int r = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (!b.act[r]) return;
  const long N = b.N;
  const int m = b.m;
  const double *Vr = V + (long)r * ldv_r;
  const double *wr = w + (long)r * ldw_r;
  double *part = b.part + (long)r * 2 * gridDim.x * (m + 1);
  const long stride = (long)gridDim.x * blockDim.x;
  const long i0 = blockIdx.x * (long)blockDim.x + threadIdx.x;
  for (int v0 = 0; v0 < nv; v0 += 8)
    by_count(nv - v0, [&](auto count) {
      constexpr int C = decltype(count)::value;
      double s[C];
#pragma unroll
      for (int j = 0; j < C; ++j) s[j] = 0.0;
      const double *x = Vr + (long)v0 * N;
      for (long i = i0; i < N; i += stride) {
        const double wi = wr[i];
#pragma unroll
        for (int j = 0; j < C; ++j) s[j] += x[(long)j * N + i] * wi;
      }
      __syncthreads();
#pragma unroll
      for (int j = 0; j < C; ++j) red[j][threadIdx.x] = s[j];
      __syncthreads();
      if (warp < C) {
        const double t = fold256(red[warp], lane);
        if (lane == 0) part[(long)blockIdx.x * nv + v0 + warp] = t;
      }
    });
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(b.ticket + r, 1) == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int v = warp; v < nv; v += 8) {
    const double sum = partials_sum(part, gridDim.x, nv, v, lane);
    if (lane != 0) continue;
    if (out1) out1[(long)r * (m + 1) + v] = sum;
    if (out2) out2[(long)r * (m + 1) + v] += sum;
    if (gvmode && v == 0) {
      b.scal[r * 8 + 2] = sum;
      b.scal[r * 8 + 3] = givens_step(b.H + (long)r * (m + 1) * m, m, k, b.hcol + (long)r * (m + 1), sum,
                                      b.cs + (long)r * m, b.sn + (long)r * m, b.gv + (long)r * (m + 1),
                                      b.inv_bnorm[r]);
    }
  }
  if (threadIdx.x == 0) b.ticket[r] = 0;
}

// ||w_r||^2 into scal[r][slot] (no Givens step)
__global__ void __launch_bounds__(kDotThreads) k_bnorm2(KBatch b, const double *__restrict__ w, long ldw_r,
                                                        int slot) {
  __shared__ double red[kDotThreads];
  __shared__ int last;
  const int r = blockIdx.y;
  if (b.act && !b.act[r]) return;
  const long N = b.N;
  const double *wr = w + (long)r * ldw_r;
  double *part = b.part + (long)r * 2 * gridDim.x * (b.m + 1);
  double sum = 0.0;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < N; i += (long)gridDim.x * blockDim.x)
    sum += wr[i] * wr[i];
  sum = block_sum(sum, red);
  if (threadIdx.x == 0) {
    part[blockIdx.x] = sum;
    __threadfence();
    last = atomicAdd(b.ticket + r, 1) == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (threadIdx.x < 32) {
    const double t = partials_sum(part, gridDim.x, 1, 0, threadIdx.x);
    if (threadIdx.x == 0) {
      b.scal[r * 8 + slot] = t;
      b.ticket[r] = 0;
    }
  }
}

// w_r -= sum_{v < nv} h_r[v] V_r[v]
__global__ void k_borth_update(KBatch b, const double *__restrict__ V, long ldv_r, int nv,
                               const double *__restrict__ h, double *__restrict__ w, long ldw_r) {
  const int r = blockIdx.y;
  if (!b.act[r]) return;
  const long N = b.N;
  const double *Vr = V + (long)r * ldv_r;
  const double *hr = h + (long)r * (b.m + 1);
  double *wr = w + (long)r * ldw_r;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < N; i += (long)gridDim.x * blockDim.x) {
    double acc = wr[i];
    for (int v = 0; v < nv; ++v) acc -= hr[v] * Vr[(long)v * N + i];
    wr[i] = acc;
  }
}

// y_r = x_r / sqrt(scal[r][slot])
__global__ void k_bscale(KBatch b, const double *__restrict__ x, long ldx_r, int slot, double *__restrict__ y,
                         long ldy_r) {
  const int r = blockIdx.y;
  if (!b.act[r]) return;
  __shared__ double s_inv;  // one reciprocal square root per block, not per thread
  if (threadIdx.x == 0) {
    const double n2 = b.scal[r * 8 + slot];
    s_inv = n2 > 0.0 ? rsqrt(n2) : 0.0;
  }
  __syncthreads();
  const double inv = s_inv;
  const double *xr = x + (long)r * ldx_r;
  double *yr = y + (long)r * ldy_r;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < b.N; i += (long)gridDim.x * blockDim.x)
    yr[i] = xr[i] * inv;
}

// z_r = a x_r + c y_r
__global__ void k_baxpby(KBatch b, double a, const double *__restrict__ x, long ldx_r, double c,
                         const double *__restrict__ y, long ldy_r, double *__restrict__ z, long ldz_r) {
  const int r = blockIdx.y;
  if (!b.act[r]) return;
  const double *xr = x + (long)r * ldx_r, *yr = y + (long)r * ldy_r;
  double *zr = z + (long)r * ldz_r;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < b.N; i += (long)gridDim.x * blockDim.x)
    zr[i] = a * xr[i] + c * yr[i];
}

}  // namespace

// What the current device has room for, asked once per device (two words, no
// state of a solve).  Clusters of more than 8 blocks need a per-kernel opt-in.
static vie_status arnoldi_room(ArnoldiRoom *room) {
  static std::atomic<int> known[64];  // 1 + cluster + 32 resident
  int dev = 0;
  VIE_CUDA(cudaGetDevice(&dev));
  int v = known[dev & 63].load();
  if (v == 0) {
    const void *wide = (const void *)k_arnoldi<kCluster, true, 1>;
    VIE_CUDA(cudaFuncSetAttribute(wide, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    auto clusters = [&](const void *kernel, unsigned size) {
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = size;
      at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
      cudaLaunchConfig_t cfg{};
      cfg.gridDim = dim3(size);
      cfg.blockDim = dim3(kDotThreads);
      cfg.attrs = at;
      cfg.numAttrs = 1;
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
        cudaGetLastError();  // a size the device does not run
        n = 0;
      }
      return n;
    };
    const int cluster = clusters(wide, 16) > 0                                                         ? 16
                        : clusters(wide, 8) > 0 && clusters((const void *)k_arnoldi<kCluster, true, 2>, 8) > 0 ? 8
                                                                                                       : 0;
    int per_sm = 0, per_sm_reg = 0;
    DevProps prop;
    VIE_TRY(get_dev_props(dev, &prop));
    VIE_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_arnoldi<kGridWide, false, 1>, kDotThreads, 0));
    VIE_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_reg, k_arnoldi<kGridWide, true, 1>, kDotThreads, 0));
    v = 1 + cluster + 32 * ((per_sm < per_sm_reg ? per_sm : per_sm_reg) * prop.multiProcessorCount);
    known[dev & 63].store(v);
  }
  room->cluster = (v - 1) % 32;
  room->resident = (v - 1) / 32;
  return VIE_OK;
}

// Blocks of the dot products of one right-hand side.  Up to 16 (one cluster)
// as long as a thread then holds at most four elements: with one block the
// narrow FP64 pipe of its SM bounds the step (17.7 us at N = 1024; four blocks
// 13.3).  Above, four elements per thread: the block sums add one
// operation per thread to them (25 %); past one block per SM, two on every SM
// (152; the same on a part of the device, so that the sums keep their order).
int dot_blocks(long N) {
  const long one = (N + kDotThreads - 1) / kDotThreads;
  if (one <= kMaxCluster) return (int)(one < 1 ? 1 : one);
  const long four = (N + 4 * kDotThreads - 1) / (4 * kDotThreads);
  return (int)(four <= kMaxCluster ? kMaxCluster : four <= 152 ? four : 304);
}

vie_status arnoldi_fused(long N, int R, bool *fused) {
  ArnoldiRoom room;
  VIE_TRY(arnoldi_room(&room));
  *fused = arnoldi_one_launch(dot_blocks(N), R, room);
  return VIE_OK;
}

vie_status launch_arnoldi(const KBatch &b, double *V, long ldv_r, int k, double inv_bnorm1, const int *err0,
                          const int *err1, unsigned long long seq, unsigned *bar, cudaStream_t st) {
  const bool reg = b.N <= (long)kRegElems * b.blocks * kDotThreads;
  int dev = 0;
  VIE_CUDA(cudaGetDevice(&dev));
  const WaitLimits wl = wait_limits(dev);
  // large batches: two blocks per CTA (and clusters of 8)
  const int vb = b.blocks <= kMaxCluster ? b.blocks / arnoldi_cluster(b.blocks, b.R) : 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(b.blocks / vb), (unsigned)b.R);
  cfg.blockDim = dim3(kDotThreads);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  cfg.attrs = at;
  auto go = [&](auto kernel) {
    return cudaLaunchKernelEx(&cfg, kernel, b, V, ldv_r, k, inv_bnorm1, err0, err1, seq, bar, wl);
  };
  if (b.blocks == 1) {
    VIE_CUDA(go(k_arnoldi<kOneBlock, true, 1>));
  } else if (b.blocks <= kMaxCluster) {
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cfg.gridDim.x;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.numAttrs = 1;
    if (vb == 2)
      VIE_CUDA(go(k_arnoldi<kCluster, true, 2>));
    else
      VIE_CUDA(go(k_arnoldi<kCluster, true, 1>));
  } else {
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.numAttrs = 1;
    if (reg)
      VIE_CUDA(go(k_arnoldi<kGridWide, true, 1>));
    else
      VIE_CUDA(go(k_arnoldi<kGridWide, false, 1>));
  }
  count_launch();
  return VIE_OK;
}

vie_status launch_update(const KBatch &b, const double *B, long ldb_r, int k_all, const int *kk, double *x,
                         long ldx_r, cudaStream_t st) {
  // every block takes the (short) triangular solve again: few of them in a batch
  const long per = (b.R > 1 ? 16L : 4L) * kDotThreads, gx = (b.N + per - 1) / per;
  k_update<<<dim3((unsigned)(gx < 2048 ? gx : 2048), (unsigned)b.R), kDotThreads, 0, st>>>(b, B, ldb_r, k_all, kk, x,
                                                                                        ldx_r);
  VIE_CHECK_LAUNCH("k_update");
  return VIE_OK;
}

vie_status launch_scale(const double *x, const double *norm2, double *y, long N, cudaStream_t st) {
  k_scale<<<grid_for(N, 256), 256, 0, st>>>(x, norm2, y, N);
  VIE_CHECK_LAUNCH("k_scale");
  return VIE_OK;
}

vie_status launch_axpby(double a, const double *x, double b, const double *y, double *z, long N,
                        cudaStream_t st) {
  k_axpby<<<grid_for(N, 256), 256, 0, st>>>(a, x, b, y, z, N);
  VIE_CHECK_LAUNCH("k_axpby");
  return VIE_OK;
}

// ---- lockstep batch launchers (KBatch: vie_internal.cuh)
static dim3 bgrid(long N, int R, int threads) {
  long gx = (N + threads - 1) / threads;
  gx = gx < 1 ? 1 : (gx > 2048 / (R < 8 ? R : 8) ? 2048 / (R < 8 ? R : 8) : gx);
  return dim3((unsigned)gx, (unsigned)R);
}

vie_status launch_bdots(const KBatch &b, const double *V, long ldv_r, int nv, const double *w, long ldw_r,
                        double *out1, double *out2, cudaStream_t st) {
  k_bdots_last<<<dim3((unsigned)b.blocks, (unsigned)b.R), kDotThreads, 0, st>>>(b, V, ldv_r, nv, w, ldw_r, out1,
                                                                                out2, 0, 0);
  VIE_CHECK_LAUNCH("k_bdots_last");
  return VIE_OK;
}

vie_status launch_bnorm2_givens(const KBatch &b, const double *w, long ldw_r, int k, cudaStream_t st) {
  k_bdots_last<<<dim3((unsigned)b.blocks, (unsigned)b.R), kDotThreads, 0, st>>>(b, w, ldw_r, 1, w, ldw_r,
                                                                                nullptr, nullptr, 1, k);
  VIE_CHECK_LAUNCH("k_bdots_last");
  return VIE_OK;
}

vie_status launch_bnorm2(const KBatch &b, const double *w, long ldw_r, int slot, cudaStream_t st) {
  k_bnorm2<<<dim3((unsigned)b.blocks, (unsigned)b.R), kDotThreads, 0, st>>>(b, w, ldw_r, slot);
  VIE_CHECK_LAUNCH("k_bnorm2");
  return VIE_OK;
}

vie_status launch_borth_update(const KBatch &b, const double *V, long ldv_r, int nv, const double *h, double *w,
                               long ldw_r, cudaStream_t st) {
  k_borth_update<<<bgrid(b.N, b.R, 256), 256, 0, st>>>(b, V, ldv_r, nv, h, w, ldw_r);
  VIE_CHECK_LAUNCH("k_borth_update");
  return VIE_OK;
}

vie_status launch_bscale(const KBatch &b, const double *x, long ldx_r, int slot, double *y, long ldy_r,
                         cudaStream_t st) {
  k_bscale<<<bgrid(b.N, b.R, 256), 256, 0, st>>>(b, x, ldx_r, slot, y, ldy_r);
  VIE_CHECK_LAUNCH("k_bscale");
  return VIE_OK;
}

vie_status launch_baxpby(const KBatch &b, double a, const double *x, long ldx_r, double c, const double *y,
                         long ldy_r, double *z, long ldz_r, cudaStream_t st) {
  k_baxpby<<<bgrid(b.N, b.R, 256), 256, 0, st>>>(b, a, x, ldx_r, c, y, ldy_r, z, ldz_r);
  VIE_CHECK_LAUNCH("k_baxpby");
  return VIE_OK;
}

}  // namespace vie
