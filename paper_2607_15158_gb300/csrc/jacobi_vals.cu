// Singular values of a batch of small k x k matrices by one-sided Jacobi
// (Hestenes 1958), without the singular vectors: corner spectra and
// ctm_svdvals_noalloc.
//
// What bounds it is the chain of a round of disjoint rotations: dot product,
// warp reduction, rotation angle, rotation, hand-over of the columns. The
// kernels that also return vectors (jacobi.cu) take the angle with fp64 roots,
// divisions and hypots, a chain of about 5000 clocks a round (8300 with the
// columns passed through global memory, as above k = 64). Here
//   * each matrix lives in the shared memory of a cluster of up to eight CTAs,
//     two blocks of B columns in each. A CTA rotates every column of one
//     block against every column of the other (B rounds of B pairs, one pair
//     per warp, separated by the CTA's own barrier), then the blocks move on
//     round-robin through distributed shared memory (two buffers): 2 G - 1
//     cluster barriers a sweep. Pairs within a block take their rounds at the
//     start of a sweep;
//   * the tangent of the rotation is taken in fp32 and only the cosine that
//     belongs to it in fp64 (from the hardware's approximate reciprocal square
//     root by Newton steps): the rotation is orthogonal to fp64 rounding, and
//     an angle off by 5e-7 leaves 5e-7 of the overlap. In the last sweep, whose
//     overlaps are below 7e-10, that is less than the threshold k eps; in every other
//     the next sweep meets it. Against an extended-precision Jacobi (k = 8 to 128,
//     real and complex, singular values falling to e^-16) the errors are 5e-16 to
//     4e-15 of the largest value; with a Newton step in fp64 on the tangent 3e-16 to
//     5e-15 and a tenth more time; from the vector kernels, whose angles are fp64,
//     1e-15 to 4e-14;
//   * the sweep is the last that either rotates nothing, or whose rotated overlaps
//     are below 7e-10 of the norms and so small beside its angles that (largest
//     overlap) x (largest tangent) is below eps. A rotation returns to a pair that
//     was already orthogonal its tangent times another overlap, at most 2 (k - 1)
//     such terms a sweep, so what is left is of the order of the threshold k eps.
//     The overlaps alone do not decide that: columns of nearly equal norm turn by up
//     to 45 degrees however small their overlap, and their cluster converges only as
//     a matrix of its own would (a spectrum within 1e-9 of one value takes seven
//     sweeps at k = 64; one leaves errors of 1e-10). On random and on graded
//     spectra the rule costs no sweep (k = 8 to 128), one without rotations one.
// The matrix is scaled by a power of two so that its largest entry is about
// 1; overlaps below 1e-140 then are left alone (their squares leave the fp64
// range). The squared norms are exact at the start of each sweep and updated
// between; the results are the norms of the final columns. The rows of A
// serve as columns (A and its transpose have the same singular values). The
// call of a program (k x k, singular values falling to e^-16) took, with the
// vector kernel and here: k = 32 real 2.06 ms -> 0.49, 64 real 6.0 -> 1.33,
// 128 real 13.4 -> 5.7, 64 complex 5.9 -> 2.5, 96 complex 10.8 -> 5.8. Above
// that the pairs of one matrix outgrow the fp64 pipes of eight SMs and the
// vector kernel, which uses them all, is as fast.
#include <cooperative_groups.h>

#include <algorithm>
#include <cfloat>

#include "common.cuh"
#include "kernels.h"

namespace ctm {

namespace {

namespace cg = cooperative_groups;

constexpr int VMAXG = 8;   // most CTAs per matrix
constexpr int VMAXW = 8;   // most warps per CTA
constexpr int NONE = -1000000;

struct ValsArgs {
  int k, G, B, max_sweeps;   // B: columns per block, two blocks per CTA
  const void* A;
  long strideA;
  double* s;
  int* err;
};

// 1 / sqrt(a) from an approximation y with relative error below 2^-19: with
// e = 1 - a y^2, y (1 + e / 2 + 3 e^2 / 8) is off by about 5 e^3 / 16
__device__ __forceinline__ double rsqrt_from(double a, double y) {
  const double e = fma(-a * y, y, 1.0);
  return fma(y * e, fma(e, 0.375, 0.5), y);
}
__device__ __forceinline__ double rsqrt_n(double a) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
  return rsqrt_from(a, y);
}

// biased exponent field of |x|
__device__ __forceinline__ int exf(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// x 2^-e as fp32, truncated (0 where that is below the fp32 range; it must not
// overflow it)
__device__ __forceinline__ float scaled32(double x, int e) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int ex = (int)(hi >> 20 & 0x7ffu), f = ex - e - 896;   // 127 - 1023
  const unsigned bits = (hi & 0x80000000u) | (unsigned)f << 23 | (hi & 0xfffffu) << 3 | lo >> 29;
  return ex == 0 || f <= 0 ? 0.f : __uint_as_float(bits);
}

// tangent t of the rotation that makes columns with squared norms al, be and
// real overlap g orthogonal (|t| <= 1): 2 g / (d + sign(d) sqrt(d^2 + 4 g^2)),
// d = be - al, to fp32 accuracy, and an fp32 1 / sqrt(1 + t^2)
__device__ __forceinline__ double tangent(double d, double g, double& c0) {
  const int ed = exf(d), eg = exf(g);
  const int e = max(ed, eg + 1) - 1023;
  c0 = 1.0;
  if (eg - 1023 - e < -90) return g / d;   // far below fp32's range beside d
  const float df = scaled32(d, e), gf = 2.f * scaled32(g, e);
  float h, c;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(h) : "f"(fmaf(df, df, gf * gf)));
  h += fabsf(df);
  const float t = h > 0.f ? __fdividef(df < 0.f ? -gf : gf, h) : 0.f;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(c) : "f"(fmaf(t, t, 1.f)));
  c0 = f64_of(c);
  return f64_of(t);
}

template <typename T, int R>
__global__ void __launch_bounds__(32 * VMAXW) jacobi_vals_kernel(ValsArgs a) {
  cg::cluster_group cl = cg::this_cluster();
  const int k = a.k, G = a.G, B = a.B;
  const int rank = G > 1 ? (int)cl.block_rank() : 0;
  const int b = blockIdx.x / G;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  extern __shared__ __align__(16) unsigned char smem[];
  T* cols = reinterpret_cast<T*>(smem);                               // [2 buffers][2 blocks][B][k]
  double* nsq = reinterpret_cast<double*>(cols + (size_t)4 * B * k);  // [2][2][B]
  double* vals = nsq + 4 * B;                                         // [2 G B]
  // largest exponent of the sweep's rotated |gamma|^2 / (alpha beta) and of its tangents
  __shared__ int mx[2][2];
  __shared__ int mxs[2][2][VMAXG];   // those of all CTAs
  __shared__ int exs[VMAXG];            // largest exponent field of every CTA's entries
  __shared__ int exm;
  auto arrive = [&]() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); };
  auto wait = [&]() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); };
  auto sync = [&]() {
    if (G > 1) {
      arrive();
      wait();
    } else {
      __syncthreads();
    }
  };
  // every CTA of the cluster must run before its shared memory is written: arrive
  // here, wait before the first remote store, the loads in between
  if (G > 1) arrive();
  auto remote = [&](auto* p, int cta) { return G > 1 ? cl.map_shared_rank(p, cta) : p; };
  // block position q of the round-robin table: CTA q's first block for q < G,
  // CTA 2 G - 1 - q's second block above
  auto cta_of = [&](int q) { return q < G ? q : 2 * G - 1 - q; };
  const int q0 = rank, q1 = 2 * G - 1 - rank;
  // where the blocks go after a round: all but position 0 move down by one,
  // position 1 to the end
  const int d0 = q0 == 0 ? 0 : q0 == 1 ? 2 * G - 1 : q0 - 1;
  const int d1 = G == 1 ? 1 : q1 - 1;
  if (threadIdx.x < 4) mx[threadIdx.x / 2][threadIdx.x % 2] = NONE;
  if (threadIdx.x == 0) exm = 0;
  __syncthreads();
  const T* A = static_cast<const T*>(a.A) + (size_t)b * a.strideA;
  int em = 0;
  for (int sl = wp; sl < 2 * B; sl += nw) {
    const int c = (sl < B ? q0 * B + sl : q1 * B + sl - B);
    for (int r = lane; r < k; r += 32) {
      const T v = c < k ? A[(size_t)c * k + r] : zero_of(T());
      if constexpr (sizeof(T) == 8) em = max(em, exf(v));
      else em = max(em, max(exf(v.x), exf(v.y)));
      cols[(size_t)sl * k + r] = v;
    }
  }
  em = __reduce_max_sync(0xffffffffu, em);
  if (lane == 0) atomicMax(&exm, em);
  __syncthreads();
  if (G > 1) wait();
  if (threadIdx.x < G) remote(&exs[rank], threadIdx.x)[0] = exm;
  sync();
  for (int g = 0; g < G; ++g) em = max(em, exs[g]);
  // 2^(1023 - em) and back (1 where the matrix is zero or not finite)
  em = em == 0 || em == 0x7ff ? 1023 : min(max(em, 1), 2045);
  const double down = __hiloint2double((2046 - em) << 20, 0), up = __hiloint2double(em << 20, 0);
  for (int sl = wp; sl < 2 * B; sl += nw)
    for (int r = lane; r < k; r += 32)
      cols[(size_t)sl * k + r] = scalev(cols[(size_t)sl * k + r], down);
  __syncthreads();
  const double tol = fmax(1.0, (double)k) * DBL_EPSILON, tol2 = tol * tol;
  int buf = 0, sweep = 0, par = 0;
  bool converged = false;
  auto norm2 = [&](const T* c) {
    double acc = 0.0;
#pragma unroll
    for (int e = 0; e < R; ++e)
      if (lane + 32 * e < k) acc += absq(c[lane + 32 * e]);
    return warp_sum(acc);
  };
  // one rotation of the columns in slots sx and sy of the current buffer; they
  // go to (xo, nx) and (yo, ny)
  auto rotate = [&](int sx, int sy, T* xo, double* nx, T* yo, double* ny, bool in_place) {
    const T* xc = cols + (size_t)(buf * 2 * B + sx) * k;
    const T* yc = cols + (size_t)(buf * 2 * B + sy) * k;
    double al = nsq[buf * 2 * B + sx], be = nsq[buf * 2 * B + sy];
    const double thr = (tol2 * al) * be, d = be - al;
    T x[R], y[R];
    T ga = zero_of(T());
#pragma unroll
    for (int e = 0; e < R; ++e) {
      const int r = lane + 32 * e;
      x[e] = r < k ? xc[r] : zero_of(T());
      y[e] = r < k ? yc[r] : zero_of(T());
      fmacv(ga, x[e], y[e]);
    }
    ga = warp_sum(ga);
    const double g2 = absq(ga);
    const bool rot = g2 > thr && exf(g2) > 1023 - 930;   // above 1e-280
    if (rot) {
      double g;
      if constexpr (sizeof(T) == 8) {
        g = ga;
      } else {
        const double ig = rsqrt_n(g2);
        g = g2 * ig;
        // y <- conj(gamma) / |gamma| y makes the overlap real
        const cplx ph = make_double2(ga.x * ig, -ga.y * ig);
#pragma unroll
        for (int e = 0; e < R; ++e) y[e] = mulv(ph, y[e]);
      }
      double c;
      const double tt = tangent(d, g, c);
      if (lane == 0) {
        atomicMax(&mx[par][0], exf(g2) + 1023 - exf(al) - exf(be));
        atomicMax(&mx[par][1], exf(tt) - 1023);
      }
      c = rsqrt_from(fma(tt, tt, 1.0), c);
      const double s = c * tt;
#pragma unroll
      for (int e = 0; e < R; ++e) {
        const T xv = x[e], yv = y[e];
        if constexpr (sizeof(T) == 8) {
          x[e] = fma(-s, yv, c * xv);
          y[e] = fma(c, yv, s * xv);
        } else {
          x[e] = make_double2(fma(-s, yv.x, c * xv.x), fma(-s, yv.y, c * xv.y));
          y[e] = make_double2(fma(c, yv.x, s * xv.x), fma(c, yv.y, s * xv.y));
        }
      }
      const double tg = tt * g;
      al -= tg;
      be += tg;
    }
    if (rot || !in_place) {
#pragma unroll
      for (int e = 0; e < R; ++e) {
        const int r = lane + 32 * e;
        if (r < k) {
          xo[r] = x[e];
          yo[r] = y[e];
        }
      }
      if (lane == 0) {
        *nx = al;
        *ny = be;
      }
    }
  };
  auto rotate_here = [&](int sx, int sy) {
    T* c = cols + (size_t)buf * 2 * B * k;
    double* n = nsq + buf * 2 * B;
    rotate(sx, sy, c + (size_t)sx * k, n + sx, c + (size_t)sy * k, n + sy, true);
  };
  for (; sweep < a.max_sweeps && !converged; ++sweep) {
    par = sweep & 1;
    for (int sl = wp; sl < 2 * B; sl += nw) {
      const double n = norm2(cols + (size_t)(buf * 2 * B + sl) * k);
      if (lane == 0) nsq[buf * 2 * B + sl] = n;
    }
    __syncthreads();
    // pairs within the two blocks, round-robin over B (or B + 1) places
    const int m = B + (B & 1);
    for (int t = 0; t + 1 < m; ++t) {
      for (int task = wp; task < m; task += nw) {
        const int side = task < m / 2 ? 0 : 1, i = task - side * (m / 2), o = m - 1 - i;
        const int u = i == 0 ? 0 : (i - 1 + t) % (m - 1) + 1, v = (o - 1 + t) % (m - 1) + 1;
        if (u < B && v < B) rotate_here(side * B + u, side * B + v);
      }
      __syncthreads();
    }
    for (int t = 0; t < 2 * G - 1; ++t) {
      // the first block's columns against the second's
      for (int i = 0; i + 1 < B; ++i) {
        for (int w = wp; w < B; w += nw) rotate_here(w, B + (w + i) % B);
        __syncthreads();
      }
      const int nb = (buf ^ 1) * 2 * B;
      for (int w = wp; w < B; w += nw) {
        const int v = (w + B - 1) % B;
        const int xs = nb + (d0 < G ? 0 : B) + w, ys = nb + (d1 < G ? 0 : B) + v;
        rotate(w, B + v, remote(cols, cta_of(d0)) + (size_t)xs * k, remote(nsq, cta_of(d0)) + xs,
               remote(cols, cta_of(d1)) + (size_t)ys * k, remote(nsq, cta_of(d1)) + ys, false);
      }
      buf ^= 1;
      sync();
    }
    // the largest ratio and tangent of the sweep over all CTAs
    if (threadIdx.x < 2 * G) {
      const int g = threadIdx.x / 2, i = threadIdx.x % 2;
      remote(&mxs[par][i][rank], g)[0] = mx[par][i];
    }
    if (threadIdx.x < 2) mx[par ^ 1][threadIdx.x] = NONE;
    sync();
    int mm = NONE, mt = NONE;
    for (int g = 0; g < G; ++g) {
      mm = max(mm, mxs[par][0][g]);
      mt = max(mt, mxs[par][1][g]);
    }
    // the overlap is below 2^((mm + 1) / 2), the tangent below 2^(mt + 1): the
    // first below 2^-30, the product below 2^-52 (NONE: nothing was rotated)
    converged = mm == NONE || (mm < -61 && mm + 2 * mt <= -107);
  }
  if (!converged && rank == 0 && threadIdx.x == 0) atomicOr(a.err, DEV_JACOBI_NOCONV);
  // norms of the columns to every CTA
  for (int sl = wp; sl < 2 * B; sl += nw) {
    const double v = sqrt(norm2(cols + (size_t)(buf * 2 * B + sl) * k));
    if (lane < G) remote(vals, lane)[rank * 2 * B + sl] = v;
  }
  sync();
  // descending order, ties to the lower place; the last of 2 G B > k values
  // are zero columns that fill the blocks
  const int n = 2 * G * B;
  for (int p = rank * blockDim.x + threadIdx.x; p < n; p += G * blockDim.x) {
    const double v = vals[p];
    int rk = 0;
    for (int j = 0; j < n; ++j) rk += (vals[j] > v) || (vals[j] == v && j < p);
    if (!isfinite(v)) atomicOr(a.err, DEV_NONFINITE);
    if (rk < k) a.s[(size_t)b * k + rk] = v * up;
  }
}

// CTAs per matrix: blocks of four columns (one pair per fp64 pipe of an SM)
// as long as eight CTAs hold them all, larger blocks above
int vals_ctas(int k) {
  int g = 1;
  while (g < VMAXG && k > 8 * g) g *= 2;
  return g;
}
int vals_block(int k, int G) { return (k + 2 * G - 1) / (2 * G); }

size_t vals_smem(bool cx, int k, int G) {
  const size_t B = vals_block(k, G);
  return 4 * B * k * (cx ? 16 : 8) + (4 * B + 2 * G * B) * sizeof(double);
}

template <typename T, int R>
cudaError_t launch_vals(const ValsArgs& a, int batch, size_t shm, cudaStream_t s) {
  static size_t configured = 0;
  auto* fn = jacobi_vals_kernel<T, R>;
  const cudaError_t e = raise_smem((const void*)fn, configured, shm);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(batch * a.G));
  cfg.blockDim = dim3((unsigned)(32 * std::min(a.B, VMAXW)));
  cfg.dynamicSmemBytes = shm;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)a.G;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = a.G > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, fn, a);
}

template <typename T>
cudaError_t dispatch_vals(const ValsArgs& a, int batch, size_t shm, cudaStream_t s) {
  if (a.k <= 32) return launch_vals<T, 1>(a, batch, shm, s);
  if (a.k <= 64) return launch_vals<T, 2>(a, batch, shm, s);
  if constexpr (sizeof(T) == 8)
    if (a.k > 96) return launch_vals<T, 4>(a, batch, shm, s);
  return launch_vals<T, 3>(a, batch, shm, s);
}

}  // namespace

bool jacobi_vals_supported(bool cx, int k) {
  return k >= 1 && k <= (cx ? 96 : 128) && vals_smem(cx, k, vals_ctas(k)) <= (size_t)200 * 1024;
}

cudaError_t jacobi_vals(bool cx, int k, const void* A, long strideA, double* sv, int batch,
                        int max_sweeps, int* err, cudaStream_t s, long* launches) {
  if (!jacobi_vals_supported(cx, k) || batch < 1) return cudaErrorInvalidValue;
  ValsArgs a;
  a.k = k;
  a.G = vals_ctas(k);
  a.B = vals_block(k, a.G);
  a.max_sweeps = max_sweeps;
  a.A = A;
  a.strideA = strideA;
  a.s = sv;
  a.err = err;
  const size_t shm = vals_smem(cx, k, a.G);
  if (launches) ++*launches;
  return cx ? dispatch_vals<cplx>(a, batch, shm, s) : dispatch_vals<double>(a, batch, shm, s);
}

}  // namespace ctm
