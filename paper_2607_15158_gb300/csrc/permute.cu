// Axis permutation of dense row-major tensors (the reshapes between the
// pairwise contractions of the enlarged corners and of the absorption).
// Memory-bound. After fusing axes that stay adjacent, rows whose fastest axis
// stays in place and is long are copied; everything else goes tile by tile
// through shared memory. A tile spans the fastest axes of the input and the
// fastest axes of the output (the bond axes are 2 to 8 long, so it takes
// several of each to make runs of 256 bytes on both sides), is read in the
// input's order and written in the output's. The positions of a tile's
// elements on both sides are the same for every tile: each block computes
// them once. One pair of axes per 32 x 32 tile, most of it empty with bonds
// this short, took 152 us a permutation of the unfused complex D = 4, chi = 64
// absorption (18 here) and 41 of the real D = 4, chi = 48 two-site patches.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace ctm {

namespace {

struct PermArgs {
  int rank;
  long od[8];     // output dims
  long os[8];     // input stride of each output axis
  long ostr[8];   // output stride of each output axis
  long total;
};

template <typename T, bool CONJ, typename I>
__global__ void __launch_bounds__(256) perm_rows(const T* __restrict__ in,
                                                 T* __restrict__ out,
                                                 PermArgs p) {
  // one warp per output row of length L = od[rank-1] (input stride 1)
  const I L = (I)p.od[p.rank - 1];
  const I nrows = (I)(p.total / p.od[p.rank - 1]);
  const int lane = threadIdx.x & 31;
  I w = (I)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
  const I nw = (I)(gridDim.x * (blockDim.x >> 5));
  for (I row = w; row < nrows; row += nw) {
    I rem = row, ioff = 0;
    for (int j = p.rank - 2; j >= 0; --j) {
      I q = rem / (I)p.od[j];
      ioff += (rem - q * (I)p.od[j]) * (I)p.os[j];
      rem = q;
    }
    const T* src = in + ioff;
    T* dst = out + row * L;
    for (I e = lane; e < L; e += 32) {
      T v = src[e];
      if (CONJ) v = conjv(v);
      dst[e] = v;
    }
  }
}

// tile of the permutation: extents of the axes that it spans (1 elsewhere)
struct TileArgs {
  int E;             // elements
  int nax;           // axes with extent > 1
  int ax[8];         // those axes, fastest in the input first
  unsigned mg[8];    // ceil(2^32 / extent): e / extent = umulhi(e, mg) for e, extent < 2^16
  int iax[8];        // index in ax[] of the axes, fastest in the output first
  int chunk[2];      // axes that the tiles divide (-1: none)
  long ext[8];       // extent of every axis
  long nt[8];        // tiles along every axis
  long ntiles;
};

// one element of padding per 128 bytes keeps strided reads of the tile off
// the same banks
template <typename T>
__device__ __forceinline__ int pad_idx(int e) {
  return e + (e >> (sizeof(T) == 16 ? 3 : 4));
}

template <typename T, bool CONJ, typename I>
__global__ void __launch_bounds__(256) perm_tile(const T* __restrict__ in, T* __restrict__ out,
                                                 PermArgs p, TileArgs t) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* tile = reinterpret_cast<T*>(smem_raw);
  I* tin = reinterpret_cast<I*>(tile + pad_idx<T>(t.E) + 1);   // input offset, input order
  I* tout = tin + t.E;                                          // output offset, output order
  unsigned* cin = reinterpret_cast<unsigned*>(tout + t.E);      // coordinates on the chunked axes
  unsigned* cout = cin + t.E;
  unsigned* src = cout + t.E;                                   // tile position, output order
  for (int e = threadIdx.x; e < t.E; e += 256) {
    unsigned rem = (unsigned)e, c2 = 0;
    I o = 0;
    for (int a = 0; a < t.nax; ++a) {
      const int ax = t.ax[a];
      const unsigned q = __umulhi(rem, t.mg[a]), c = rem - q * (unsigned)t.ext[ax];
      o += (I)c * (I)p.os[ax];
      if (ax == t.chunk[0]) c2 |= c;
      if (ax == t.chunk[1]) c2 |= c << 16;
      rem = q;
    }
    tin[e] = o;
    cin[e] = c2;
    rem = (unsigned)e;
    c2 = 0;
    o = 0;
    unsigned pos = 0;
    for (int b = 0; b < t.nax; ++b) {
      const int a = t.iax[b], ax = t.ax[a];
      const unsigned q = __umulhi(rem, t.mg[a]), c = rem - q * (unsigned)t.ext[ax];
      o += (I)c * (I)p.ostr[ax];
      unsigned w = c;   // weight of axis a in the input order of the tile
      for (int f = 0; f < a; ++f) w *= (unsigned)t.ext[t.ax[f]];
      pos += w;
      if (ax == t.chunk[0]) c2 |= c;
      if (ax == t.chunk[1]) c2 |= c << 16;
      rem = q;
    }
    tout[e] = o;
    cout[e] = c2;
    src[e] = pad_idx<T>((int)pos);
  }
  __syncthreads();
  for (long tl = blockIdx.x; tl < t.ntiles; tl += gridDim.x) {
    I ib = 0, ob = 0;
    unsigned lim0 = 0xffffu, lim1 = 0xffffu;   // live extent on the chunked axes
    I rem = (I)tl;
    for (int a = p.rank - 1; a >= 0; --a) {
      if (t.nt[a] == 1) continue;
      const I q = rem / (I)t.nt[a], c = (rem - q * (I)t.nt[a]) * (I)t.ext[a];
      ib += c * (I)p.os[a];
      ob += c * (I)p.ostr[a];
      const unsigned left = (unsigned)min((long)0xffff, p.od[a] - (long)c);
      if (a == t.chunk[0]) lim0 = left;
      if (a == t.chunk[1]) lim1 = left;
      rem = q;
    }
#pragma unroll 4
    for (int e = threadIdx.x; e < t.E; e += 256) {
      const unsigned c = cin[e];
      if ((c & 0xffffu) < lim0 && (c >> 16) < lim1) tile[pad_idx<T>(e)] = in[ib + tin[e]];
    }
    __syncthreads();
#pragma unroll 4
    for (int e = threadIdx.x; e < t.E; e += 256) {
      const unsigned c = cout[e];
      if ((c & 0xffffu) < lim0 && (c >> 16) < lim1) {
        T v = tile[src[e]];
        if (CONJ) v = conjv(v);
        out[ob + tout[e]] = v;
      }
    }
    __syncthreads();
  }
}

// The tile: runs of at least `run` elements on both sides, then doubled along
// the two last axes taken while it has at most emax elements.
TileArgs plan_tile(const PermArgs& p, long run, long emax) {
  TileArgs t{};
  int byin[8];
  for (int a = 0; a < p.rank; ++a) {
    t.ext[a] = 1;
    byin[a] = a;
  }
  std::sort(byin, byin + p.rank, [&](int a, int b) { return p.os[a] < p.os[b]; });
  t.chunk[0] = t.chunk[1] = -1;
  for (int side = 0; side < 2; ++side) {
    long prod = 1;
    for (int b = 0; b < p.rank && prod < run; ++b) {
      const int a = side == 0 ? byin[b] : p.rank - 1 - b;
      t.ext[a] = std::max(t.ext[a], std::min(p.od[a], (run + prod - 1) / prod));
      prod *= t.ext[a];
      t.chunk[side] = a;
    }
  }
  auto elems = [&]() {
    long e = 1;
    for (int a = 0; a < p.rank; ++a) e *= t.ext[a];
    return e;
  };
  for (int side = 1, tries = 0; tries < 2; side ^= 1) {
    const int a = t.chunk[side];
    const long old = t.ext[a], e = elems(), grown = std::min(p.od[a], 2 * old);
    if (grown > old && e / old * grown <= emax) {
      t.ext[a] = grown;
      tries = 0;
    } else {
      ++tries;
    }
  }
  t.E = (int)elems();
  t.ntiles = 1;
  for (int a = 0; a < p.rank; ++a) {
    t.nt[a] = (p.od[a] + t.ext[a] - 1) / t.ext[a];
    t.ntiles *= t.nt[a];
  }
  for (int b = 0; b < p.rank; ++b)
    if (t.ext[byin[b]] > 1) {
      t.mg[t.nax] = (unsigned)(((1ull << 32) + t.ext[byin[b]] - 1) / t.ext[byin[b]]);
      t.ax[t.nax++] = byin[b];
    }
  int n = 0;
  for (int a = p.rank - 1; a >= 0; --a)
    for (int b = 0; b < t.nax; ++b)
      if (t.ax[b] == a) t.iax[n++] = b;
  if (t.chunk[0] == t.chunk[1]) t.chunk[1] = -1;
  return t;
}

template <typename T, bool CONJ, typename I>
cudaError_t launch(const void* in, void* out, const PermArgs& p,
                   cudaStream_t s, long* launches) {
  const T* src = static_cast<const T*>(in);
  T* dst = static_cast<T*>(out);
  const int last = p.rank - 1;
  const long maxgrid = 152L * 16;
  if (p.os[last] == 1 && (p.od[last] >= 64 || p.rank == 1)) {
    long rows = p.total / p.od[last];
    long grid = (rows + 7) / 8;
    if (grid > maxgrid) grid = maxgrid;
    perm_rows<T, CONJ, I><<<(unsigned)grid, 256, 0, s>>>(src, dst, p);
  } else {
    // 256-byte runs; tiles of up to 2048 elements while two per SM remain
    const long emax = std::min(2048L, std::max(256L, p.total / (2 * 152)));
    const TileArgs t = plan_tile(p, 256 / (long)sizeof(T), emax);
    const size_t shm = (size_t)(t.E + t.E / (sizeof(T) == 16 ? 8 : 16) + 1) * sizeof(T) +
                       (size_t)t.E * (2 * sizeof(I) + 12);
    static size_t configured = 0;
    const cudaError_t e = raise_smem((const void*)perm_tile<T, CONJ, I>, configured, shm);
    if (e != cudaSuccess) return e;
    const long grid = std::min(t.ntiles, 152L * 6);
    perm_tile<T, CONJ, I><<<(unsigned)grid, 256, shm, s>>>(src, dst, p, t);
  }
  if (launches) ++*launches;
  return cudaGetLastError();
}

}  // namespace

cudaError_t permute(const void* in, void* out, int rank, const long* in_dims,
                    const int* perm, bool cx, bool conj, cudaStream_t s,
                    long* launches) {
  if (rank < 1 || rank > 8) return cudaErrorInvalidValue;
  long istr[8];
  long acc = 1;
  for (int j = rank - 1; j >= 0; --j) {
    istr[j] = acc;
    acc *= in_dims[j];
  }
  const long total = acc;
  if (total == 0) return cudaSuccess;
  // output axes, dropping size-1 axes, then fusing axes adjacent in both
  long od[8], os[8];
  int r = 0;
  for (int j = 0; j < rank; ++j) {
    long d = in_dims[perm[j]];
    if (d == 1) continue;
    od[r] = d;
    os[r] = istr[perm[j]];
    ++r;
  }
  PermArgs p{};
  if (r == 0) {
    od[0] = 1;
    os[0] = 1;
    r = 1;
  }
  int n = 0;
  long cd = od[r - 1], cs = os[r - 1];
  long fd[8], fs[8];
  for (int j = r - 2; j >= 0; --j) {
    if (os[j] == cs * cd) {
      cd *= od[j];
    } else {
      fd[n] = cd;
      fs[n] = cs;
      ++n;
      cd = od[j];
      cs = os[j];
    }
  }
  fd[n] = cd;
  fs[n] = cs;
  ++n;
  p.rank = n;
  for (int j = 0; j < n; ++j) {
    p.od[j] = fd[n - 1 - j];
    p.os[j] = fs[n - 1 - j];
  }
  long o = 1;
  for (int j = n - 1; j >= 0; --j) {
    p.ostr[j] = o;
    o *= p.od[j];
  }
  p.total = total;
  if (p.rank == 1 && p.os[0] == 1 && !conj) {
    if (launches) ++*launches;
    return cudaMemcpyAsync(out, in, total * (cx ? 16 : 8),
                           cudaMemcpyDeviceToDevice, s);
  }
  const bool small = total < (1L << 31);
  if (cx) {
    if (conj)
      return small ? launch<cplx, true, uint32_t>(in, out, p, s, launches)
                   : launch<cplx, true, uint64_t>(in, out, p, s, launches);
    return small ? launch<cplx, false, uint32_t>(in, out, p, s, launches)
                 : launch<cplx, false, uint64_t>(in, out, p, s, launches);
  }
  return small ? launch<double, false, uint32_t>(in, out, p, s, launches)
               : launch<double, false, uint64_t>(in, out, p, s, launches);
}

}  // namespace ctm
