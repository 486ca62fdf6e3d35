// Single-layer absorption of the ket and bra tensors into a corner / edge
// block (paper Eq. rho_M_diag, Fig. ctmrg-step: A and conj(A) are absorbed
// one after the other, never as the double-layer A (x) conj(A)):
//
//   Out[t,d,D,n,e,E] = sum_{s,u,l,v,w} A[s,u,l,d,e] B[s,v,w,D,E] In[t,l,w,n,u,v]
//
// In and Out are [chi, Dk, Db, chi, Dk, Db] row-major. For every (t, n) the
// work is two small matrix products per physical index s,
//   Y_s = A_s X       (Dk^2 x Dk^2) (Dk^2 x Db^2),  X[(u,l),(w,v)] = In[t,l,w,n,u,v]
//   Out += Y_s B_s    (Dk^2 x Db^2) (Db^2 x Db^2),  B_s[(w,v),(D,E)] = B[s,v,w,D,E]
// so one kernel reads In once and writes Out once (the unfused form is two
// permutes, two GEMMs and a final permute); the fp32 arithmetic, not HBM,
// bounds it. Each CTA holds A and B in shared memory and runs NG groups of
// GT x GT threads, one (t, n) pair each; a thread owns a TL x TL register
// tile of the products, rows ti + GT a and columns tj + GT b (consecutive
// threads read consecutive shared-memory words). Geometries: GT = 12,
// TL = 3 for Dk^2, Db^2 <= 36 (D <= 6), with four groups and the next
// pair's input staged by cp.async in fp32, else two groups; GT = 16, TL = 4,
// one group for <= 64 (D <= 8). D = 6 and D = 8 also have compile-time
// variants. Arithmetic in F: fp32 (split-precision contexts, ~1e-7 relative
// like the bf16x3 products) or fp64. Square bonds of 4 to 6 with many pairs in
// fp32, and all of fp64, have kernels of their own below.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace ctm {

namespace {

constexpr size_t SMEM_MAX = 227 * 1024;   // shared memory of one block

// hardware conversions here: they issue on the narrow fp64 pipe, but that
// pipe is otherwise idle in this kernel and other warps' fp32 work covers
// them (the integer-pipe conversions of common.cuh measured 12 % slower)
__device__ __forceinline__ float cvt(double a, float) { return (float)a; }
__device__ __forceinline__ float2 cvt(cplx a, float2) { return make_float2((float)a.x, (float)a.y); }
__device__ __forceinline__ double cvt(double a, double) { return a; }
__device__ __forceinline__ cplx cvt(cplx a, cplx) { return a; }
__device__ __forceinline__ double back(float a) { return (double)a; }
__device__ __forceinline__ cplx back(float2 a) { return make_double2((double)a.x, (double)a.y); }
__device__ __forceinline__ double back(double a) { return a; }
__device__ __forceinline__ cplx back(cplx a) { return a; }

__device__ __forceinline__ void mac(float& c, float a, float b) { c = fmaf(a, b, c); }
__device__ __forceinline__ void mac(float2& c, float2 a, float2 b) {
  c.x = fmaf(a.x, b.x, c.x);
  c.x = fmaf(-a.y, b.y, c.x);
  c.y = fmaf(a.x, b.y, c.y);
  c.y = fmaf(a.y, b.x, c.y);
}
__device__ __forceinline__ void mac(double& c, double a, double b) { c = fma(a, b, c); }
__device__ __forceinline__ void mac(cplx& c, cplx a, cplx b) { fmav(c, a, b); }
template <typename F> __device__ __forceinline__ F fz();
template <> __device__ __forceinline__ float fz<float>() { return 0.f; }
template <> __device__ __forceinline__ float2 fz<float2>() { return make_float2(0.f, 0.f); }
template <> __device__ __forceinline__ double fz<double>() { return 0.0; }
template <> __device__ __forceinline__ cplx fz<cplx>() { return make_double2(0.0, 0.0); }

// asynchronous global -> shared copies of one input element (Ampere+ cp.async)
__device__ __forceinline__ void cp_async_elem(cplx* dst, const cplx* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_elem(double* dst, const double* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// two blocks per SM where their shared memory allows (two groups, 8-byte F)
template <typename F, int NG>
constexpr int ab_min_blocks() {
  return (NG == 2 && sizeof(F) <= 8) ? 2 : 1;
}

// ST: the next pair's input block is copied into a staging buffer with
// cp.async while the current pair is computed (fp32 arithmetic, D <= 6)
// DK > 0: Dk = Db = DK fixed at compile time (constant index arithmetic, and
// no bounds tests when the DK^2 x DK^2 tile fills the threads exactly)
template <typename T, typename F, int GT, int TL, int NG, bool ST, int DK>
__global__ void __launch_bounds__(NG * GT * GT, ab_min_blocks<F, NG>())
    absorb_ab_kernel(int chi, int dk_arg, int db_arg, int d, const T* __restrict__ In,
                     const T* __restrict__ A, const T* __restrict__ B, T* __restrict__ Out) {
  constexpr int GROUP = GT * GT;   // threads per (t, n) pair
  constexpr int TILE = TL;         // register tile per thread
  constexpr bool kFull = DK > 0 && DK * DK == GT * TL;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int Dk = DK > 0 ? DK : dk_arg, Db = DK > 0 ? DK : db_arg;
  const int K1 = Dk * Dk, N1 = Db * Db;          // (u,l) and (w,v); M1 = K1 rows (d,e)
  F* As = reinterpret_cast<F*>(smem_raw);         // [d][(d,e)][(u,l)]
  F* Bs = As + (size_t)d * K1 * K1;               // [d][(w,v)][(D,E)]
  const int grp = threadIdx.x / GROUP, lt = threadIdx.x % GROUP;
  F* Xs = Bs + (size_t)d * N1 * N1 + (size_t)grp * 2 * K1 * N1;   // [(u,l)][(w,v)]
  F* Ys = Xs + (size_t)K1 * N1;                                   // [(d,e)][(w,v)], then Out
  const int ti = lt / GT, tj = lt % GT;
  // staging buffers (raw input elements, 16-byte aligned) after all groups' X, Y
  T* St = nullptr;
  if constexpr (ST) {
    const uintptr_t end = reinterpret_cast<uintptr_t>(Bs + (size_t)d * N1 * N1 +
                                                      (size_t)NG * 2 * K1 * N1);
    St = reinterpret_cast<T*>((end + 15) & ~(uintptr_t)15) + (size_t)grp * K1 * N1;
  }
  for (int i = threadIdx.x; i < d * K1 * K1; i += blockDim.x) {
    // As[s][(d,e)][(u,l)] = A[s,u,l,d,e]
    const int s = i / (K1 * K1), rem = i % (K1 * K1);
    const int r = rem / K1, kk = rem % K1;
    const int dd = r / Dk, e = r % Dk, u = kk / Dk, l = kk % Dk;
    As[i] = cvt(A[(((size_t)(s * Dk + u) * Dk + l) * Dk + dd) * Dk + e], F());
  }
  for (int i = threadIdx.x; i < d * N1 * N1; i += blockDim.x) {
    // Bs[s][(w,v)][(D,E)] = B[s,v,w,D,E]
    const int s = i / (N1 * N1), rem = i % (N1 * N1);
    const int kk = rem / N1, c = rem % N1;
    const int w = kk / Db, v = kk % Db, D = c / Db, E = c % Db;
    Bs[i] = cvt(B[(((size_t)(s * Db + v) * Db + w) * Db + D) * Db + E], F());
  }
  const size_t row = (size_t)chi * Dk * Db;       // stride of the (first chi, Dk, Db) index
  const long npairs = (long)chi * chi;
  // element i = (l w, u v) of pair pp's block: In[t,l,w,n,u,v], runs of Dk Db
  // contiguous (u, v)
  auto src_of = [&](long pp, int i) {
    const int tt = (int)(pp / chi), nn = (int)(pp % chi);
    const int lw = i / (Dk * Db), uv = i % (Dk * Db);
    const int l = lw / Db, w = lw % Db;
    return In + ((size_t)tt * Dk + l) * Db * row + (size_t)w * row + (size_t)nn * Dk * Db + uv;
  };
  if constexpr (ST) {
    const long pf = (long)NG * blockIdx.x + grp;
    if (pf < npairs)
      for (int i = lt; i < K1 * N1; i += GROUP) cp_async_elem(St + i, src_of(pf, i));
    cp_async_commit();
  }
  for (long p0 = (long)NG * blockIdx.x; p0 < npairs; p0 += (long)NG * gridDim.x) {
    const long p = p0 + grp;
    const bool live = p < npairs;
    const int t = live ? (int)(p / chi) : 0, n = live ? (int)(p % chi) : 0;
    if constexpr (ST) {
      cp_async_wait_all();
      __syncthreads();   // staged blocks complete; previous output staging consumed
      if (live)
        for (int i = lt; i < K1 * N1; i += GROUP) {
          const int lw = i / (Dk * Db), uv = i % (Dk * Db);
          const int l = lw / Db, w = lw % Db, u = uv / Db, v = uv % Db;
          Xs[(u * Dk + l) * N1 + w * Db + v] = cvt(St[i], F());
        }
      __syncthreads();   // the staging buffers are free again
      const long pn = p + (long)NG * gridDim.x;
      if (pn < npairs)
        for (int i = lt; i < K1 * N1; i += GROUP) cp_async_elem(St + i, src_of(pn, i));
      cp_async_commit();
    } else {
      __syncthreads();   // previous pair's output staging is consumed
      if (live) {
        // X[(u,l),(w,v)] = In[t,l,w,n,u,v]
        for (int i = lt; i < K1 * N1; i += GROUP) {
          const int lw = i / (Dk * Db), uv = i % (Dk * Db);
          const int l = lw / Db, w = lw % Db, u = uv / Db, v = uv % Db;
          Xs[(u * Dk + l) * N1 + w * Db + v] = cvt(*src_of(p, i), F());
        }
      }
    }
    F acc[TILE][TILE];
#pragma unroll
    for (int a = 0; a < TILE; ++a)
#pragma unroll
      for (int b = 0; b < TILE; ++b) acc[a][b] = fz<F>();
    for (int s = 0; s < d; ++s) {
      __syncthreads();   // X loaded / previous Y consumed
      const F* Asb = As + (size_t)s * K1 * K1;
      if (live) {
        F y[TILE][TILE];
#pragma unroll
        for (int a = 0; a < TILE; ++a)
#pragma unroll
          for (int b = 0; b < TILE; ++b) y[a][b] = fz<F>();
#pragma unroll 4
        for (int kk = 0; kk < K1; ++kk) {
          F xa[TILE], xb[TILE];
#pragma unroll
          for (int a = 0; a < TILE; ++a) {
            const int r = ti + GT * a;
            xa[a] = (kFull || r < K1) ? Asb[r * K1 + kk] : fz<F>();
          }
#pragma unroll
          for (int b = 0; b < TILE; ++b) {
            const int c = tj + GT * b;
            xb[b] = (kFull || c < N1) ? Xs[kk * N1 + c] : fz<F>();
          }
#pragma unroll
          for (int a = 0; a < TILE; ++a)
#pragma unroll
            for (int b = 0; b < TILE; ++b) mac(y[a][b], xa[a], xb[b]);
        }
#pragma unroll
        for (int a = 0; a < TILE; ++a)
#pragma unroll
          for (int b = 0; b < TILE; ++b) {
            const int r = ti + GT * a, c = tj + GT * b;
            if (kFull || (r < K1 && c < N1)) Ys[r * N1 + c] = y[a][b];
          }
      }
      __syncthreads();
      const F* Bsb = Bs + (size_t)s * N1 * N1;
      if (live) {
#pragma unroll 4
        for (int kk = 0; kk < N1; ++kk) {
          F ya[TILE], bb[TILE];
#pragma unroll
          for (int a = 0; a < TILE; ++a) {
            const int r = ti + GT * a;
            ya[a] = (kFull || r < K1) ? Ys[r * N1 + kk] : fz<F>();
          }
#pragma unroll
          for (int b = 0; b < TILE; ++b) {
            const int c = tj + GT * b;
            bb[b] = (kFull || c < N1) ? Bsb[kk * N1 + c] : fz<F>();
          }
#pragma unroll
          for (int a = 0; a < TILE; ++a)
#pragma unroll
            for (int b = 0; b < TILE; ++b) mac(acc[a][b], ya[a], bb[b]);
        }
      }
    }
    __syncthreads();   // all Y reads done: Ys becomes the output staging
    if (live) {
#pragma unroll
      for (int a = 0; a < TILE; ++a)
#pragma unroll
        for (int b = 0; b < TILE; ++b) {
          const int r = ti + GT * a, c = tj + GT * b;
          if (kFull || (r < K1 && c < N1)) Ys[r * N1 + c] = acc[a][b];
        }
    }
    __syncthreads();
    if (live) {
      // Out[t,d,D,n,e,E] = O[(d,e),(D,E)]: runs of Dk Db contiguous (e, E)
      for (int i = lt; i < K1 * N1; i += GROUP) {
        const int dD = i / (Dk * Db), eE = i % (Dk * Db);
        const int dd = dD / Db, D = dD % Db, e = eE / Db, E = eE % Db;
        Out[((size_t)t * Dk + dd) * Db * row + (size_t)D * row + (size_t)n * Dk * Db + eE] =
            back(Ys[(dd * Dk + e) * N1 + D * Db + E]);
      }
    }
  }
}

// fp32 arithmetic for square bonds DK = 4, 5, 6 and many pairs, the steps of a
// pair overlapped: four warps copy and convert the next input blocks into the
// second of two X buffers while the others multiply, and the results go from
// the registers to Out. In absorb_ab_kernel all warps of a block convert,
// multiply and write in turn, and whatever D is compute 36 x 36 outputs.
// The multiplying warps form two halves, each with its own named barriers, so
// that one half's waits fall into the other's work. A pair's DK^2 x DK^2
// outputs are TR x TC register tiles of RG x CG threads in a SLOT of lanes;
// larger tiles than 3 x 3 keep the shared-memory reads (2 (TR + TC) wavefronts
// a warp and k, complex) under the fp32 pipes' TR TC clocks. Measured for
// complex data, d = 2: D = 4, chi = 80 162 us -> 42, D = 5, chi = 58 142 -> 72,
// D = 6, chi = 144 915 -> 866 (the pipes' rate: 384; tiles of 6 x 4 with packed
// multiply-adds, 3 x 3, 3 x 6 and 4 x 4 took 900 to 1010).
template <int DK> struct AP;
template <> struct AP<6> {
  static constexpr int TR = 4, TC = 6, RG = 9, CG = 6, SLOT = 64, PH = 2, HW = 4, UNROLL = 1;
};
template <> struct AP<5> {
  static constexpr int TR = 5, TC = 5, RG = 5, CG = 5, SLOT = 32, PH = 6, HW = 6, UNROLL = 4;
};
template <> struct AP<4> {
  static constexpr int TR = 4, TC = 4, RG = 4, CG = 4, SLOT = 16, PH = 12, HW = 6, UNROLL = 1;
};
constexpr int AP_LOAD = 128;   // threads that copy and convert

template <int DK, typename F>
struct APL {   // shared layout, in elements of F
  // two values a read (real data, even DK); rows of A and Y an odd length, or then
  // K1 + 2: both spread a column over the banks
  static constexpr bool TWO = DK % 2 == 0 && sizeof(F) == 4;
  static constexpr int K1 = DK * DK, LD = TWO ? K1 + 2 : K1 | 1, NP = 2 * AP<DK>::PH;
  static constexpr int PAD4 = DK == 4 ? 8 : 0;   // two pairs a warp: other banks
  static constexpr int A_S = (K1 * LD + 3) / 4 * 4, B_S = K1 * K1;
  static constexpr int X_P = (K1 * K1 + 3) / 4 * 4 + PAD4, Y_P = (K1 * LD + 3) / 4 * 4 + PAD4;
  static constexpr int THREADS = 64 * AP<DK>::HW + AP_LOAD;
  static constexpr size_t bytes(int d) {
    return ((size_t)d * (A_S + (B_S + 3) / 4 * 4) + (size_t)NP * (2 * X_P + Y_P)) * sizeof(F);
  }
};

__device__ __forceinline__ void nb_sync(int id, int n) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void nb_arrive(int id, int n) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}
// fp32 -> fp64, on the integer pipe but for subnormal values
__device__ __forceinline__ double wide(float a) {
  return (__float_as_uint(a) & 0x7f800000u) != 0u ? f64_of(a) : (double)a;
}
__device__ __forceinline__ cplx wide(float2 a) { return make_double2(wide(a.x), wide(a.y)); }

// the columns of a thread's tile: adjacent pairs where they are read in twos
template <int DK, bool TWO>
__device__ __forceinline__ constexpr int tile_col(int tj, int c) {
  return TWO ? 2 * (tj + AP<DK>::CG * (c / 2)) + c % 2 : tj + AP<DK>::CG * c;
}
template <typename F> struct alignas(2 * sizeof(F)) Two { F v[2]; };

// v += left (rows ti + RG a, LD apart) times right (columns tile_col). Real data
// of even DK: two values of k of the left factor and two columns of the right one
// are one read, which halves the reads (as many as a fourth of the multiply-adds).
// D = 6, chi = 144, d = 2: 406 us without, 301 with. Complex data has four times
// the arithmetic per value; there it cost registers and time (867 against 1007)
template <typename F, int DK>
__device__ __forceinline__ void tile_multiply(F (&v)[AP<DK>::TR][AP<DK>::TC], const F* left,
                                              const F* right, int ti, int tj) {
  using P = AP<DK>;
  constexpr bool TWO = APL<DK, F>::TWO;
  constexpr int K1 = DK * DK, LD = APL<DK, F>::LD, KS = TWO ? 2 : 1, UNROLL = TWO ? 2 : P::UNROLL;
  left += ti * LD;
#pragma unroll UNROLL
  for (int kk = 0; kk < K1; kk += KS) {
    F xa[P::TR][KS];
#pragma unroll
    for (int a = 0; a < P::TR; ++a) {
      if constexpr (KS == 2) {
        const Two<F> t = *reinterpret_cast<const Two<F>*>(left + P::RG * a * LD + kk);
        xa[a][0] = t.v[0];
        xa[a][1] = t.v[1];
      } else {
        xa[a][0] = left[P::RG * a * LD + kk];
      }
    }
#pragma unroll
    for (int k = 0; k < KS; ++k) {
      const F* row = right + (kk + k) * K1;
      F xb[P::TC];
#pragma unroll
      for (int c = 0; c < P::TC; c += KS) {
        if constexpr (KS == 2) {
          const Two<F> t = *reinterpret_cast<const Two<F>*>(row + tile_col<DK, TWO>(tj, c));
          xb[c] = t.v[0];
          xb[c + 1] = t.v[1];
        } else {
          xb[c] = row[tile_col<DK, TWO>(tj, c)];
        }
      }
#pragma unroll
      for (int a = 0; a < P::TR; ++a)
#pragma unroll
        for (int c = 0; c < P::TC; ++c) mac(v[a][c], xa[a][k], xb[c]);
    }
  }
}
template <typename F, int DK>
__device__ __forceinline__ void tile_zero(F (&v)[AP<DK>::TR][AP<DK>::TC]) {
#pragma unroll
  for (int a = 0; a < AP<DK>::TR; ++a)
#pragma unroll
    for (int c = 0; c < AP<DK>::TC; ++c) v[a][c] = fz<F>();
}
template <typename F, int DK, typename Fn>
__device__ __forceinline__ void tile_each(F (&v)[AP<DK>::TR][AP<DK>::TC], int ti, int tj, Fn&& fn) {
  using P = AP<DK>;
#pragma unroll
  for (int a = 0; a < P::TR; ++a)
#pragma unroll
    for (int c = 0; c < P::TC; ++c)
      fn(ti + P::RG * a, tile_col<DK, APL<DK, F>::TWO>(tj, c), v[a][c]);
}

template <typename T, typename F, int DK>
__global__ void __launch_bounds__(APL<DK, F>::THREADS, 1)
    absorb_pipe_kernel(int chi, int d, const T* __restrict__ In, const T* __restrict__ A,
                       const T* __restrict__ B, T* __restrict__ Out) {
  using L = APL<DK, F>;
  using P = AP<DK>;
  constexpr int K1 = L::K1, KN = K1 * K1, LD = L::LD, PH = P::PH;
  constexpr int HT = 32 * P::HW, NB = HT + AP_LOAD;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  F* Bs = reinterpret_cast<F*>(smem_raw);   // [d][(w,v)][(D,E)]
  constexpr int BS = (L::B_S + 3) / 4 * 4;
  F* As = Bs + (size_t)d * BS;               // [d][(d,e)][(u,l)], rows of LD
  F* Ys = As + (size_t)d * L::A_S;           // [pair][(d,e)][(w,v)], rows of LD
  F* Xs = Ys + L::NP * L::Y_P;               // [buffer][pair][(u,l)][(w,v)]
  for (int i = threadIdx.x; i < d * KN; i += L::THREADS) {
    // As[s][(d,e)][(u,l)] = A[s,u,l,d,e]; Bs[s][(w,v)][(D,E)] = B[s,v,w,D,E]
    const int s = i / KN, rem = i % KN, x = rem / K1, y = rem % K1;
    As[s * L::A_S + y * LD + x] = cvt(A[i], F());
    Bs[s * BS + ((x % DK) * DK + x / DK) * K1 + y] = cvt(B[i], F());
  }
  __syncthreads();
  const size_t row = (size_t)chi * K1;       // stride of the (first chi, Dk, Db) index
  const long npairs = (long)chi * chi, step = (long)L::NP * gridDim.x;
  const long first = (long)L::NP * blockIdx.x;
  const int nsteps = first < npairs ? (int)((npairs - first + step - 1) / step) : 0;
  // barriers: X buffer b of half h filled 1 + 4 h + b, free again 3 + 4 h + b; Y of pair q 9 + q
  if (threadIdx.x >= 2 * HT) {
    const int lt = threadIdx.x - 2 * HT;
    for (int i = 0; i < nsteps; ++i) {
      const int b = i & 1;
#pragma unroll 1
      for (int h = 0; h < 2; ++h) {
        if (i >= 2) nb_sync(3 + 4 * h + b, NB);
        const long p0 = first + i * step + h * PH;
#pragma unroll 1
        for (int q = 0; q < PH; ++q) {
          const long p = p0 + q;
          if (p >= npairs) break;
          const int t = (int)(p / chi), n = (int)(p % chi);
          const T* src = In + (size_t)t * K1 * row + (size_t)n * K1;
          F* X = Xs + (size_t)(b * L::NP + h * PH + q) * L::X_P;
          constexpr int U = (KN + AP_LOAD - 1) / AP_LOAD;   // all loads in flight at once
          T v[U];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int e = lt + u * AP_LOAD;
            if (e < KN) v[u] = __ldcs(src + (size_t)(e / K1) * row + e % K1);
          }
#pragma unroll
          for (int u = 0; u < U; ++u) {
            // X[(u,l),(w,v)] = In[t,l,w,n,u,v]
            const int e = lt + u * AP_LOAD, lw = e / K1, uv = e % K1;
            if (e < KN)
              X[(uv / DK * DK + lw / DK) * K1 + lw % DK * DK + uv % DK] = cvt(v[u], F());
          }
        }
        nb_arrive(1 + 4 * h + b, NB);
      }
    }
    return;
  }
  const int h = threadIdx.x / HT, ht = threadIdx.x % HT;
  const int q = ht / P::SLOT, lt = ht % P::SLOT, ti = lt / P::CG, tj = lt % P::CG;
  F* Y = Ys + (size_t)(h * PH + q) * L::Y_P;
  auto team_sync = [&] {
    if constexpr (P::SLOT > 32) nb_sync(9 + h * PH + q, P::SLOT); else __syncwarp();
  };
  for (int i = 0; i < nsteps; ++i) {
    const int b = i & 1;
    const long p = first + i * step + h * PH + q;
    const bool live = lt < P::RG * P::CG && p < npairs;
    const F* X = Xs + (size_t)(b * L::NP + h * PH + q) * L::X_P;
    F acc[P::TR][P::TC];
    tile_zero<F, DK>(acc);
    nb_sync(1 + 4 * h + b, NB);
    for (int s = 0; s < d; ++s) {
      F y[P::TR][P::TC];
      tile_zero<F, DK>(y);
      if (live) tile_multiply<F, DK>(y, As + s * L::A_S, X, ti, tj);
      team_sync();   // the previous Y is consumed
      if (live) tile_each<F, DK>(y, ti, tj, [&](int r, int c, F v) { Y[r * LD + c] = v; });
      if (s == d - 1 && i + 2 < nsteps) nb_arrive(3 + 4 * h + b, NB);   // X is free
      team_sync();
      if (live) tile_multiply<F, DK>(acc, Y, Bs + s * BS, ti, tj);
    }
    if (live) {
      // Out[t,d,D,n,e,E]: the threads of a tile row write runs of (e, E)
      const int t = (int)(p / chi), n = (int)(p % chi);
      T* dst = Out + (size_t)t * K1 * row + (size_t)n * K1;
      tile_each<F, DK>(acc, ti, tj, [&](int r, int c, F v) {
        dst[(size_t)(r / DK * DK + c / DK) * row + r % DK * DK + c % DK] = wide(v);
      });
    }
  }
}

template <typename T, typename F, int DK>
cudaError_t launch_pipe(int chi, int d, const void* In, const void* A, const void* B, void* Out,
                        int num_sms, cudaStream_t s) {
  using L = APL<DK, F>;
  static size_t configured = 0;
  auto* fn = absorb_pipe_kernel<T, F, DK>;
  cudaError_t e = raise_smem((const void*)fn, configured, L::bytes(d));
  if (e != cudaSuccess) return e;
  const long tiles = ((long)chi * chi + L::NP - 1) / L::NP;
  fn<<<(unsigned)std::min((long)num_sms, tiles), L::THREADS, L::bytes(d), s>>>(
      chi, d, static_cast<const T*>(In), static_cast<const T*>(A), static_cast<const T*>(B),
      static_cast<T*>(Out));
  return cudaGetLastError();
}

// more pairs than absorb_ab_kernel's grid of four a block takes at once: up to
// there that kernel's time is one block's, 19 to 33 us against 27 to 42 here
// (complex, D = 4 to 6, chi <= 24); above it was never faster (chi = 28: 34, 51
// and 60 us against 27, 43 and 60)
template <int DK, typename F>
bool use_pipe(int chi, int Dk, int Db, int d, int num_sms) {
  return Dk == DK && Db == DK && APL<DK, F>::bytes(d) <= SMEM_MAX &&
         (long)chi * chi > 4L * num_sms;
}

// The same contraction in fp64 (F = T), which the fp64 pipe bounds: a
// multiply-add occupies a sub-partition for ~77 clocks however few lanes of
// the warp take part, so no lane may idle and operand reads cost nothing
// beside it. The outputs of NG pairs (t, n) are numbered through and dealt to
// the warps 32 at a time, one output per lane and task, whatever D is; the
// second product's outputs are numbered in the order of Out, so the results
// go out from registers in runs of Dk Db. Register tiles of 3 x 3 on 12 x 12
// threads, which compute 36 x 36 outputs whatever D is, took 605 us at real
// D = 4, chi = 64 (150 here; 132 at the pipe's rate), 395 at complex D = 3,
// chi = 33 (33 here), 75 at real D = 3, chi = 27 (11 here).
constexpr int A64_THREADS = 256, A64_WARPS = A64_THREADS / 32;

template <typename T, int MT>
__global__ void __launch_bounds__(A64_THREADS)
    absorb64_kernel(int chi, int Dk, int Db, int d, int ng, const T* __restrict__ In,
                    const T* __restrict__ A, const T* __restrict__ B, T* __restrict__ Out) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int K1 = Dk * Dk, N1 = Db * Db, KN = K1 * N1, DD = Dk * Db;
  T* As = reinterpret_cast<T*>(smem_raw);   // [d][(d,e)][(u,l)]
  T* Bs = As + (size_t)d * K1 * K1;          // [d][(w,v)][(D,E)]
  T* Xs = Bs + (size_t)d * N1 * N1;          // [pair][(u,l)][(w,v)]
  T* Ys = Xs + (size_t)ng * KN;              // [pair][(d,e)][(w,v)]
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < d * K1 * K1; i += A64_THREADS) {
    // As[s][(d,e)][(u,l)] = A[s,u,l,d,e]
    const int s = i / (K1 * K1), rem = i % (K1 * K1);
    const int r = rem / K1, kk = rem % K1;
    const int dd = r / Dk, e = r % Dk, u = kk / Dk, l = kk % Dk;
    As[i] = A[(((size_t)(s * Dk + u) * Dk + l) * Dk + dd) * Dk + e];
  }
  for (int i = threadIdx.x; i < d * N1 * N1; i += A64_THREADS) {
    // Bs[s][(w,v)][(D,E)] = B[s,v,w,D,E]
    const int s = i / (N1 * N1), rem = i % (N1 * N1);
    const int kk = rem / N1, c = rem % N1;
    const int w = kk / Db, v = kk % Db, D = c / Db, E = c % Db;
    Bs[i] = B[(((size_t)(s * Db + v) * Db + w) * Db + D) * Db + E];
  }
  const size_t row = (size_t)chi * DD;       // stride of the (first chi, Dk, Db) index
  const long npairs = (long)chi * chi;
  for (long p0 = (long)ng * blockIdx.x; p0 < npairs; p0 += (long)ng * gridDim.x) {
    const int np = (int)min((long)ng, npairs - p0);
    const int nout = np * KN;
    for (int i = threadIdx.x; i < nout; i += A64_THREADS) {
      // X[(u,l),(w,v)] = In[t,l,w,n,u,v]
      const int pr = i / KN, ii = i % KN;
      const long p = p0 + pr;
      const int t = (int)(p / chi), n = (int)(p % chi);
      const int lw = ii / DD, uv = ii % DD;
      const int l = lw / Db, w = lw % Db, u = uv / Db, v = uv % Db;
      Xs[(size_t)pr * KN + (u * Dk + l) * N1 + w * Db + v] =
          In[((size_t)t * Dk + l) * Db * row + (size_t)w * row + (size_t)n * DD + uv];
    }
    T acc[MT];
#pragma unroll
    for (int m = 0; m < MT; ++m) acc[m] = zero_of(T());
    for (int s = 0; s < d; ++s) {
      __syncthreads();   // X loaded / previous Y consumed
#pragma unroll
      for (int m = 0; m < MT; ++m) {
        const int t0 = 32 * (wp + A64_WARPS * m);
        if (t0 >= nout) break;
        const int o = min(t0 + lane, nout - 1);
        const int pr = o / KN, r = o % KN / N1, c = o % N1;
        const T* a = As + ((size_t)s * K1 + r) * K1;
        const T* x = Xs + (size_t)pr * KN + c;
        T y = zero_of(T());
#pragma unroll 4
        for (int kk = 0; kk < K1; ++kk) mac(y, a[kk], x[kk * N1]);
        if (t0 + lane < nout) Ys[o] = y;
      }
      __syncthreads();
#pragma unroll
      for (int m = 0; m < MT; ++m) {
        const int t0 = 32 * (wp + A64_WARPS * m);
        if (t0 >= nout) break;
        const int o = min(t0 + lane, nout - 1);
        // output o = (pair, (d, D), (e, E)): row (d, e), column (D, E)
        const int pr = o / KN, oo = o % KN, dD = oo / DD, eE = oo % DD;
        const int r = dD / Db * Dk + eE / Db, c = dD % Db * Db + eE % Db;
        const T* y = Ys + (size_t)pr * KN + r * N1;
        const T* b = Bs + (size_t)s * N1 * N1 + c;
#pragma unroll 4
        for (int kk = 0; kk < N1; ++kk) mac(acc[m], y[kk], b[kk * N1]);
      }
    }
#pragma unroll
    for (int m = 0; m < MT; ++m) {
      const int o = 32 * (wp + A64_WARPS * m) + lane;
      if (o < nout) {
        const int pr = o / KN, oo = o % KN, dD = oo / DD, eE = oo % DD;
        const long p = p0 + pr;
        const int t = (int)(p / chi), n = (int)(p % chi);
        Out[((size_t)t * Dk * Db + dD) * row + (size_t)n * DD + eE] = acc[m];
      }
    }
  }
}

size_t a64_smem(int Dk, int Db, int d, int ng, size_t tsize) {
  const size_t K1 = (size_t)Dk * Dk, N1 = (size_t)Db * Db;
  return ((size_t)d * K1 * K1 + (size_t)d * N1 * N1 + 2 * (size_t)ng * K1 * N1) * tsize;
}

template <typename T, int MT>
cudaError_t launch_a64(int chi, int Dk, int Db, int d, int ng, const void* In, const void* A,
                       const void* B, void* Out, int num_sms, cudaStream_t s) {
  const size_t shm = a64_smem(Dk, Db, d, ng, sizeof(T));
  static size_t configured = 0;
  auto* fn = absorb64_kernel<T, MT>;
  cudaError_t e = raise_smem((const void*)fn, configured, shm);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, A64_THREADS, shm);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  const long tiles = ((long)chi * chi + ng - 1) / ng;
  const long grid = std::min((long)num_sms * per_sm, tiles);
  fn<<<(unsigned)grid, A64_THREADS, shm, s>>>(chi, Dk, Db, d, ng, static_cast<const T*>(In),
                                              static_cast<const T*>(A), static_cast<const T*>(B),
                                              static_cast<T*>(Out));
  return cudaGetLastError();
}

// Pairs per block: as many as fill four tasks of every warp, while every SM
// keeps two blocks' worth of them and they fit half its shared memory
template <typename T>
cudaError_t launch_absorb64(int chi, int Dk, int Db, int d, const void* In, const void* A,
                            const void* B, void* Out, int num_sms, cudaStream_t s) {
  const long kn = (long)Dk * Dk * Db * Db;
  long ng = std::min(4L * A64_THREADS / kn, (long)chi * chi / (2L * num_sms));
  ng = std::max(1L, ng);
  while (ng > 1 && a64_smem(Dk, Db, d, (int)ng, sizeof(T)) > SMEM_MAX / 2) --ng;
  const long tasks = (ng * kn + A64_THREADS - 1) / A64_THREADS;   // per warp
  if (tasks <= 2) return launch_a64<T, 2>(chi, Dk, Db, d, (int)ng, In, A, B, Out, num_sms, s);
  if (tasks <= 4) return launch_a64<T, 4>(chi, Dk, Db, d, (int)ng, In, A, B, Out, num_sms, s);
  if (tasks <= 6) return launch_a64<T, 6>(chi, Dk, Db, d, (int)ng, In, A, B, Out, num_sms, s);
  return launch_a64<T, 16>(chi, Dk, Db, d, (int)ng, In, A, B, Out, num_sms, s);
}

// shared memory of a geometry with ng groups: A and B, then X and Y per
// group, then (staged) one raw input block per group
size_t ab_smem(int Dk, int Db, int d, int ng, size_t fsize, size_t tsize, bool staged) {
  const size_t K1 = (size_t)Dk * Dk, N1 = (size_t)Db * Db;
  size_t b = ((size_t)d * K1 * K1 + (size_t)d * N1 * N1 + 2 * (size_t)ng * K1 * N1) * fsize;
  if (staged) b = (b + 15) / 16 * 16 + (size_t)ng * K1 * N1 * tsize;
  return b;
}

// 0: no fused kernel; 3: 12 x 12 threads x 3 x 3 tiles, four groups with
// staged input (fp32, D <= 6); 1: the same tiles, two groups; 2: 16 x 16
// threads x 4 x 4 tiles, one group (D <= 8); 4: the fp64 kernel (D <= 8)
int ab_geometry(int Dk, int Db, int d, size_t fsize, size_t tsize) {
  if (Dk < 1 || Db < 1 || d < 1) return 0;
  const int m = std::max(Dk * Dk, Db * Db);
  if (fsize == tsize) return m <= 64 && a64_smem(Dk, Db, d, 1, tsize) <= SMEM_MAX ? 4 : 0;
  if (m <= 36 && ab_smem(Dk, Db, d, 4, fsize, tsize, true) <= SMEM_MAX) return 3;
  if (m <= 36 && ab_smem(Dk, Db, d, 2, fsize, tsize, false) <= SMEM_MAX) return 1;
  if (m <= 64 && ab_smem(Dk, Db, d, 1, fsize, tsize, false) <= SMEM_MAX) return 2;
  return 0;
}

template <typename T, typename F, int GT, int TL, int NG, bool ST, int DK>
cudaError_t launch_ab(int chi, int Dk, int Db, int d, const void* In, const void* A,
                      const void* B, void* Out, int num_sms, cudaStream_t s) {
  const size_t shm = ab_smem(Dk, Db, d, NG, sizeof(F), sizeof(T), ST);
  static size_t configured = 0;
  auto* fn = absorb_ab_kernel<T, F, GT, TL, NG, ST, DK>;
  cudaError_t e = raise_smem((const void*)fn, configured, shm);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, NG * GT * GT, shm);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  long grid = (long)num_sms * per_sm;
  const long tiles = ((long)chi * chi + NG - 1) / NG;
  if (grid > tiles) grid = tiles;
  fn<<<(unsigned)grid, NG * GT * GT, shm, s>>>(chi, Dk, Db, d, static_cast<const T*>(In),
                                                 static_cast<const T*>(A),
                                                 static_cast<const T*>(B), static_cast<T*>(Out));
  return cudaGetLastError();
}

template <typename T, typename F>
cudaError_t launch_geom(int geom, int chi, int Dk, int Db, int d, const void* In, const void* A,
                        const void* B, void* Out, int num_sms, cudaStream_t s) {
  if constexpr (sizeof(F) == sizeof(T)) {
    return launch_absorb64<T>(chi, Dk, Db, d, In, A, B, Out, num_sms, s);
  } else {
    const bool sq = Dk == Db;
    if (use_pipe<4, F>(chi, Dk, Db, d, num_sms))
      return launch_pipe<T, F, 4>(chi, d, In, A, B, Out, num_sms, s);
    if (use_pipe<5, F>(chi, Dk, Db, d, num_sms))
      return launch_pipe<T, F, 5>(chi, d, In, A, B, Out, num_sms, s);
    if (use_pipe<6, F>(chi, Dk, Db, d, num_sms))
      return launch_pipe<T, F, 6>(chi, d, In, A, B, Out, num_sms, s);
    if (geom == 3 && sq && Dk == 6)
      return launch_ab<T, F, 12, 3, 4, true, 6>(chi, Dk, Db, d, In, A, B, Out, num_sms, s);
    if (geom == 3)
      return launch_ab<T, F, 12, 3, 4, true, 0>(chi, Dk, Db, d, In, A, B, Out, num_sms, s);
    if (geom == 2 && sq && Dk == 8)
      return launch_ab<T, F, 16, 4, 1, false, 8>(chi, Dk, Db, d, In, A, B, Out, num_sms, s);
    if (geom == 1)
      return launch_ab<T, F, 12, 3, 2, false, 0>(chi, Dk, Db, d, In, A, B, Out, num_sms, s);
    return launch_ab<T, F, 16, 4, 1, false, 0>(chi, Dk, Db, d, In, A, B, Out, num_sms, s);
  }
}

size_t elem_size(bool cx, bool fp32) { return (cx ? 2 : 1) * (fp32 ? 4 : 8); }

}  // namespace

bool absorb_ab_supported(bool cx, bool fp32, int Dk, int Db, int d) {
  return ab_geometry(Dk, Db, d, elem_size(cx, fp32), elem_size(cx, false)) != 0;
}

cudaError_t absorb_ab(bool cx, bool fp32, int chi, int Dk, int Db, int d, const void* In,
                      const void* A, const void* B, void* Out, int num_sms, cudaStream_t s,
                      long* launches) {
  const int geom = ab_geometry(Dk, Db, d, elem_size(cx, fp32), elem_size(cx, false));
  if (geom == 0 || chi < 1) return cudaErrorInvalidValue;
  cudaError_t e;
  if (cx)
    e = fp32 ? launch_geom<cplx, float2>(geom, chi, Dk, Db, d, In, A, B, Out, num_sms, s)
             : launch_geom<cplx, cplx>(geom, chi, Dk, Db, d, In, A, B, Out, num_sms, s);
  else
    e = fp32 ? launch_geom<double, float>(geom, chi, Dk, Db, d, In, A, B, Out, num_sms, s)
             : launch_geom<double, double>(geom, chi, Dk, Db, d, In, A, B, Out, num_sms, s);
  if (launches) ++*launches;
  return e;
}

}  // namespace ctm
