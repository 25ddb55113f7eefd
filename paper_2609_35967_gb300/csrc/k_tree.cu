// k_tree.cu -- the order of the particles in memory and the search tree over them, with the
// frozen partner snapshot of the interval (Sect. 2.5.1, 2.5.3).
//
// In place of the paper's KD-tree every instance is sorted along a Hilbert curve (a segmented
// radix sort of keys of 24 or 32 bits) and boxed bottom-up: 32 consecutive particles are a
// leaf, 32 leaves a node, and so on.  The order adapts to any density, so a leaf is a compact
// set of particles in the dense inner disk as in its sparse outskirts, and a warp's 32 queries
// (one leaf) share nearly all their candidates.  Equal keys keep the caller's order: the rank
// order is the same in every run.
//   k_bounds         bounds of the finite coordinates, per instance
//   k_keys           frame (origin, quantum), keys, digit counts of the first pass
//   k_radix_hist / k_radix_scan / k_radix_scatter   one 8-bit digit, least significant first
//   k_gather         rank-space copies (coalesced writes, the caller's arrays gathered), leaves
//   k_levels         one upper level of the tree
#include <algorithm>
#include <climits>
#include <vector>

#include "gd_ctx.h"
#include "gd_physics.cuh"

namespace gd {

constexpr int kSortTile = 2048;   // particles per block of the sort
constexpr int kChunk = 2048;      // digit counts per block of their scan

// ---------------------------------------------------------------- stats
// Sums of M, M m and M s per instance (a10): per-tile partials over a fixed stride and a
// fixed tree, then each instance's partials in tile order.  Every launch adds in the same
// order, so the result is bitwise reproducible.
__device__ __forceinline__ void block_tree3(double (&sh)[3][256], double a0, double a1, double a2) {
  sh[0][threadIdx.x] = a0;
  sh[1][threadIdx.x] = a1;
  sh[2][threadIdx.x] = a2;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w)
      for (int k = 0; k < 3; ++k) sh[k][threadIdx.x] += sh[k][threadIdx.x + w];
    __syncthreads();
  }
}

__global__ void __launch_bounds__(256) k_stats_tile(TileMap tm, const InstDev* __restrict__ P,
                                                    const double* __restrict__ s, const double* __restrict__ M,
                                                    double* part) {
  __shared__ double sh[3][256];
  int b;
  long long lo, hi;
  double a0 = 0.0, a1 = 0.0, a2 = 0.0;
  if (tile_range(tm, blockIdx.x, b, lo, hi)) {
    const InstDev& p = P[b];
    for (long long i = lo + threadIdx.x; i < hi; i += blockDim.x) {
      const double si = s[i], Mi = M[i];
      a0 += Mi;
      a1 += Mi * grain_mass(p, si);
      a2 += Mi * si;
    }
  }
  block_tree3(sh, a0, a1, a2);
  if (threadIdx.x == 0)
    for (int k = 0; k < 3; ++k) part[3 * (long long)blockIdx.x + k] = sh[k][0];
}

__global__ void __launch_bounds__(256) k_stats_inst(const long long* __restrict__ tile_off,
                                                    const double* __restrict__ part, double* out) {
  __shared__ double sh[3][256];
  const int b = blockIdx.x;
  double a0 = 0.0, a1 = 0.0, a2 = 0.0;
  for (long long t = tile_off[b] + threadIdx.x; t < tile_off[b + 1]; t += blockDim.x) {
    a0 += part[3 * t];
    a1 += part[3 * t + 1];
    a2 += part[3 * t + 2];
  }
  block_tree3(sh, a0, a1, a2);
  if (threadIdx.x == 0)
    for (int k = 0; k < 3; ++k) out[3 * b + k] = sh[k][0];
}

// ---------------------------------------------------------------- bounds
// Tile t of the sort: particles [lo, hi) of instance b.
__device__ __forceinline__ bool stile_range(const TileMap& tm, int tile, int& b, long long& lo, long long& hi) {
  int l = 0, h = tm.n_inst - 1;
  while (l < h) {
    const int mid = (l + h + 1) >> 1;
    if (tm.tile_off[mid] <= tile) l = mid; else h = mid - 1;
  }
  b = l;
  lo = tm.off[b] + (tile - tm.tile_off[b]) * (long long)kSortTile;
  hi = min(lo + kSortTile, tm.off[b + 1]);
  return lo < hi;
}

// A particle with a coordinate that is not finite takes no part in the bounds or the tree.
__global__ void __launch_bounds__(256) k_bounds(TileMap tm, const InstDev* __restrict__ P,
                                                const double* __restrict__ x, const double* __restrict__ y,
                                                const double* __restrict__ z, StateDev* st) {
  int b;
  long long lo, hi;
  if (!stile_range(tm, blockIdx.x, b, lo, hi)) return;
  const int model = P[b].model;
  unsigned long long mn[3] = {~0ull, ~0ull, ~0ull}, mx[3] = {0, 0, 0};
  for (long long i = lo + threadIdx.x; i < hi; i += blockDim.x) {
    double X, Y, Z;
    model_pos(model, x[i], y[i], z[i], X, Y, Z);
    if (!isfinite(X) || !isfinite(Y) || !isfinite(Z)) continue;
    unsigned long long o[3] = {dbl_ord(X), dbl_ord(Y), dbl_ord(Z)};
#pragma unroll
    for (int a = 0; a < 3; ++a) { mn[a] = min(mn[a], o[a]); mx[a] = max(mx[a], o[a]); }
  }
  __shared__ unsigned long long smn[3][8], smx[3][8];
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    for (int o = 16; o > 0; o >>= 1) {
      mn[a] = min(mn[a], __shfl_xor_sync(0xffffffffu, mn[a], o));
      mx[a] = max(mx[a], __shfl_xor_sync(0xffffffffu, mx[a], o));
    }
    if (lane == 0) { smn[a][w] = mn[a]; smx[a][w] = mx[a]; }
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    int a = threadIdx.x;
    unsigned long long m0 = ~0ull, m1 = 0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) { m0 = min(m0, smn[a][k]); m1 = max(m1, smx[a][k]); }
    if (m0 <= m1) {
      atomicMin(&st[P[b].unit0].bmin[a], m0);
      atomicMax(&st[P[b].unit0].bmax[a], m1);
    }
  }
}

// ---------------------------------------------------------------- explicit cell sizes
// A cell size (gd_instance_params.cell_size, gd_config.cell_factor) asks for a uniform grid of
// the search.  The tree needs none, but a size whose grid would still exceed the capacity
// after 40 growths is reported as before (GD_ST_CAPACITY, with exact lists).
__device__ double cells_of(const InstDev& P, const StateDev& S, double cell_factor, int xsplit, double grow) {
  double ext[3];
  for (int a = 0; a < 3; ++a) ext[a] = ord_dbl(S.bmax[a]) - ord_dbl(S.bmin[a]);
  const bool per = P.geometry == GD_GEOM_PATCH;
  if (per) { ext[0] = P.box_x; ext[1] = P.box_y; }
  const double tiny = 1e-300;
  double vol = 1.0, emax = 0.0;
  for (int a = 0; a < 3; ++a) emax = fmax(emax, ext[a]);
  for (int a = 0; a < 3; ++a) vol *= fmax(ext[a], 1e-6 * emax + tiny);
  double c;
  if (P.cell_size > 0.0) {
    c = P.cell_size;
  } else if (P.model == GD_MODEL_3D) {
    c = cell_factor * cbrt(vol / (double)P.n);
  } else {
    double span = 1.0;
    int D = 0;
    for (int a = 0; a < 3; ++a)
      if (ext[a] > 1e-9 * emax) { span *= ext[a]; ++D; }
    const double one = span / (double)P.n;
    c = cell_factor * (D >= 3 ? cbrt(one) : D == 2 ? sqrt(one) : D == 1 ? one : 1.0);
    if (!(c > 0.0)) c = emax + tiny;
  }
  c *= grow;
  double cells = 1.0;
  for (int a = 0; a < 3; ++a) {
    const bool pa = per && a < 2;
    const double e = pa ? ext[a] : ext[a] * (1.0 + 1e-9) + 1e-12 * emax + tiny;
    const double ca = a == 0 ? c / xsplit : c;
    const double dimd = pa ? floor(e / ca) : ceil(e / ca);
    const double cap = P.model == GD_MODEL_R ? (a == 0 ? 16777216.0 : 1.0) : (a < 2 ? 2048.0 : 1024.0);
    cells *= fmin(fmax(dimd, 1.0), cap);
  }
  return cells;
}

__global__ void k_check_cells(const InstDev* __restrict__ P, StateDev* st, int n_inst, double cell_factor,
                              int xsplit, long long cell_cap) {
  __shared__ double part[256];
  const int tid = threadIdx.x;
  double grow = 1.0;
  for (int attempt = 0; attempt < 40; ++attempt) {
    double mine = 0.0;
    for (int b = tid; b < n_inst; b += blockDim.x) mine += cells_of(P[b], st[P[b].unit0], cell_factor, xsplit, grow);
    __syncthreads();
    part[tid] = mine;
    __syncthreads();
    double total = 0.0;
    for (int k = 0; k < (int)blockDim.x; ++k) total += part[k];
    if (total <= (double)cell_cap) return;
    grow *= 1.1 * cbrt(total / (double)cell_cap);
  }
  for (int b = tid; b < n_inst; b += blockDim.x) set_status(&st[P[b].unit0], GD_ST_CAPACITY);
}

// ---------------------------------------------------------------- frame and keys
// The instance's frame from its data bounds: one quantum for all axes, so that distances in
// units are distances over q.  Differences of two units, and of a unit and one shifted by a
// periodic extent, fit in 32 bits.
__device__ void make_frame(const InstDev& P, const StateDev& S, TreeDev& T) {
  const bool per = P.geometry == GD_GEOM_PATCH;
  const double box[3] = {per ? P.box_x : 0.0, per ? P.box_y : 0.0, 0.0};
  double ext[3], emax = 0.0;
  const bool any = S.bmin[0] <= S.bmax[0];
  for (int a = 0; a < 3; ++a) {
    T.lo[a] = any ? ord_dbl(S.bmin[a]) : 0.0;
    ext[a] = any ? ord_dbl(S.bmax[a]) - T.lo[a] : 0.0;
    emax = fmax(emax, fmax(ext[a], box[a]));
  }
  T.bits = per ? 29 : 31;
  const double top = ldexp(1.0, T.bits) - 4096.0;
  double q = emax / top;
  if (!(q > 1e-290)) q = emax > 0.0 ? 1e-290 : 1.0;
  T.q = q;
  T.inv_q = 1.0 / q;
  T.periodic = per ? 1 : 0;
  for (int a = 0; a < 2; ++a) {
    T.box[a] = box[a];
    T.boxq[a] = (int)fmin(rint(box[a] * T.inv_q), top);
    T.maxq[a] = (int)fmin(ext[a] * T.inv_q, top) + 1;
  }
}

__device__ __forceinline__ int to_unit(const TreeDev& T, int a, double v) {
  return __double2int_rz((v - T.lo[a]) * T.inv_q);   // v >= lo; the conversion saturates
}

__device__ __forceinline__ unsigned long long spread3(unsigned v) {   // bit i to bit 3 i (v < 2^21)
  unsigned long long x = v;
  x = (x | x << 32) & 0x1F00000000FFFFull;
  x = (x | x << 16) & 0x1F0000FF0000FFull;
  x = (x | x << 8) & 0x100F00F00F00F00Full;
  x = (x | x << 4) & 0x10C30C30C30C30C3ull;
  x = (x | x << 2) & 0x1249249249249249ull;
  return x;
}
__device__ __forceinline__ unsigned spread2(unsigned x) {              // bit i to bit 2 i (x < 2^16)
  x = (x | x << 8) & 0x00FF00FFu;
  x = (x | x << 4) & 0x0F0F0F0Fu;
  x = (x | x << 2) & 0x33333333u;
  x = (x | x << 1) & 0x55555555u;
  return x;
}

// Hilbert index of nbits per axis by the transposition of J. Skilling, "Programming the
// Hilbert curve" (AIP Conf. Proc. 707, 2004): undo the excess rotations from the top bit down,
// then Gray-encode; the index's bits are those of X[0], X[1], .. interleaved.
template <int D>
__device__ __forceinline__ void hilbert_axes(unsigned (&X)[D], int nbits) {
  for (unsigned Q = 1u << (nbits - 1); Q > 1u; Q >>= 1) {
    const unsigned m = Q - 1u;
#pragma unroll
    for (int i = 0; i < D; ++i) {
      if (X[i] & Q) {
        X[0] ^= m;
      } else {
        const unsigned t = (X[0] ^ X[i]) & m;
        X[0] ^= t;
        X[i] ^= t;
      }
    }
  }
#pragma unroll
  for (int i = 1; i < D; ++i) X[i] ^= X[i - 1];
  unsigned t = 0;
  for (unsigned Q = 1u << (nbits - 1); Q > 1u; Q >>= 1)
    if (X[D - 1] & Q) t ^= Q - 1u;
#pragma unroll
  for (int i = 0; i < D; ++i) X[i] ^= t;
}

// How a 3D key divides its bits: axes by descending extent; the longest is cut in 2^n1 before the
// second has a bit, these two in 2^n2 each before the third has one, and all three in 2^n3.
//
// Cubes of the whole extent (n1 = n2 = 0) where they leave 16 cells per particle of the instance's
// own box: the curve is unbroken there, and a leaf across a break has a wide box (first builds of a
// disk of 50,001: 1.04 ms, in slabs 1.11; a patch a thousandth thick of 2^20: 0.85 and 0.90 ms).
// Slabs first where they do not: a narrow column or a thin ring had no bits left for its short axes
// (2^18 particles, first and next builds: a column 30 box widths tall 49 and 10.6 ms, in slabs 0.76
// and 0.43; a ring 0.001 wide and thinner 1.4 and 0.82, in slabs 1.1 and 0.33; a box 4:1, four cells
// per particle, 0.75 and 0.54 ms for the next builds).
struct KeyShape {
  int axis[3], top, n1, n2, n3;                       // top: bits of the longest axis' units
};

__device__ KeyShape key_shape(const StateDev& S, const TreeDev& T, long long n, int passes) {
  KeyShape K;
  int len[3];                                         // bits of the largest unit
  const bool any = S.bmin[0] <= S.bmax[0];
  for (int a = 0; a < 3; ++a) {
    const double ext = any ? ord_dbl(S.bmax[a]) - T.lo[a] : 0.0;
    len[a] = 32 - __clz((int)fmin(ext * T.inv_q, 2147483647.0));
    K.axis[a] = a;
  }
  for (int k = 0; k < 3; ++k) {                       // three exchanges order three
    const int i = k == 1 ? 1 : 0;
    if (len[K.axis[i]] < len[K.axis[i + 1]]) { const int t = K.axis[i]; K.axis[i] = K.axis[i + 1]; K.axis[i + 1] = t; }
  }
  const int bits = 8 * passes;
  K.top = len[K.axis[0]];
  const int d1 = len[K.axis[0]] - len[K.axis[1]], d2 = len[K.axis[1]] - len[K.axis[2]];
  const bool slabs = bits - (2 * d1 + d2) < 64 - __clzll(n - 1) + 4;   // cubes waste d1 and d1 + d2 bits
  K.n1 = slabs ? min(d1, bits) : 0;
  K.n2 = slabs ? min(d2, (bits - K.n1) / 2) : 0;
  K.n3 = (bits - K.n1 - 2 * K.n2 + 2) / 3;
  return K;
}

// The sort key (8 passes bits): along a 3D curve inside cubes (see KeyShape; what the last bit per
// axis has too many is dropped), a 2D curve of 12 or 16 bits per axis, or the coordinate itself
// (1D).  24 bits resolve instances of up to 2^18 particles (64 cells per particle of their box), 32
// bits the larger ones.  Where most particles crowd a few cells of the box (far outliers, clumps a
// ten-thousandth of it) their keys are equal, a leaf is a random part of the crowd and its queries go
// to the exact search: 2^18 particles of a disk with one at 1000 times its radius 180 ms a build; 64
// clumps of 2^14 324 ms first and 284 next.  (The cell grid that was before took 787 and 185 ms for
// the clumps, and 570 ms already for 2^16 with the outlier.)
__device__ __forceinline__ unsigned sort_key(int model, const TreeDev& T, const KeyShape& K, int passes, int ux, int uy,
                                             int uz) {
  const bool wide = passes > 3;
  if (model == GD_MODEL_R) return wide ? (unsigned)ux << 1 : (unsigned)ux >> (T.bits - 24);
  if (model != GD_MODEL_3D) {
    const int nb = wide ? 16 : 12;
    unsigned X[2] = {(unsigned)ux >> (T.bits - nb), (unsigned)uy >> (T.bits - nb)};
    hilbert_axes<2>(X, nb);
    return spread2(X[0]) << 1 | spread2(X[1]);
  }
  const int u[3] = {ux, uy, uz};
  unsigned v[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) v[k] = (unsigned)(K.axis[k] == 0 ? u[0] : K.axis[k] == 1 ? u[1] : u[2]);
  const int n1 = K.n1, n2 = K.n2, n3 = K.n3;
  const int below = K.top - n1;                      // bits of a slab, then of a cube
  unsigned long long key = n1 > 0 ? v[0] >> below : 0u;
  if (n2 > 0) {
    const unsigned m = (1u << n2) - 1u;
    unsigned X[2] = {(v[0] >> (below - n2)) & m, (v[1] >> (below - n2)) & m};
    hilbert_axes<2>(X, n2);
    key = key << (2 * n2) | spread2(X[0]) << 1 | spread2(X[1]);
  }
  if (n3 > 0) {
    const unsigned m = (1u << n3) - 1u;
    const int s = below - n2 - n3;
    unsigned X[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) X[k] = (s >= 0 ? v[k] >> s : v[k] << -s) & m;
    hilbert_axes<3>(X, n3);
    key = key << (3 * n3) | spread3(X[0]) << 2 | spread3(X[1]) << 1 | spread3(X[2]);
  }
  return (unsigned)(key >> (n1 + 2 * n2 + 3 * n3 - 8 * passes));
}

// Adds one tile's digit counts to the digit table (digit-major inside the instance, so that
// one exclusive scan of the whole table gives every tile's first rank of every digit) and to
// the chunk sums the scan starts from.
__device__ __forceinline__ void put_digits(const TileMap& tm, int b, const int* h, int* __restrict__ digits,
                                           int* __restrict__ chunk) {
  const long long t0 = tm.tile_off[b], nt = tm.tile_off[b + 1] - t0;
  const int d = threadIdx.x;                      // 256 threads, one digit each
  const long long at = 256 * t0 + d * nt + (blockIdx.x - t0);
  digits[at] = h[d];
  if (h[d]) atomicAdd(&chunk[at / kChunk], h[d]);
}

__global__ void __launch_bounds__(256) k_keys(TileMap tm, const InstDev* __restrict__ P, const StateDev* __restrict__ st,
                                              TreeDev* __restrict__ tree, int passes, const double* __restrict__ x,
                                              const double* __restrict__ y, const double* __restrict__ z,
                                              uint2* __restrict__ kv, int* __restrict__ digits,
                                              int* __restrict__ chunk) {
  __shared__ TreeDev T;
  __shared__ KeyShape K;
  __shared__ int h[256];
  int b;
  long long lo, hi;
  if (!stile_range(tm, blockIdx.x, b, lo, hi)) return;
  const int model = P[b].model;
  h[threadIdx.x] = 0;
  if (threadIdx.x == 0) {
    make_frame(P[b], st[P[b].unit0], T);
    K = key_shape(st[P[b].unit0], T, P[b].n, passes);
    if (blockIdx.x == tm.tile_off[b]) {
      TreeDev& G = tree[b];         // the levels' fields stay as set once
      for (int a = 0; a < 3; ++a) G.lo[a] = T.lo[a];
      G.q = T.q; G.inv_q = T.inv_q; G.periodic = T.periodic; G.bits = T.bits;
      for (int a = 0; a < 2; ++a) { G.box[a] = T.box[a]; G.boxq[a] = T.boxq[a]; G.maxq[a] = T.maxq[a]; }
    }
  }
  __syncthreads();
  for (long long i = lo + threadIdx.x; i < hi; i += blockDim.x) {
    double X, Y, Z;
    model_pos(model, x[i], y[i], z[i], X, Y, Z);
    unsigned key = passes > 3 ? ~0u : 0xFFFFFFu;
    if (isfinite(X) && isfinite(Y) && isfinite(Z))
      key = sort_key(model, T, K, passes, to_unit(T, 0, X), to_unit(T, 1, Y), to_unit(T, 2, Z));
    kv[i] = make_uint2(key, (unsigned)i);
    atomicAdd(&h[key & 255u], 1);
  }
  __syncthreads();
  put_digits(tm, b, h, digits, chunk);
}

// ---------------------------------------------------------------- radix sort
__global__ void __launch_bounds__(256) k_radix_hist(TileMap tm, int shift, const uint2* __restrict__ kv,
                                                    int* __restrict__ digits, int* __restrict__ chunk) {
  __shared__ int h[256];
  int b;
  long long lo, hi;
  if (!stile_range(tm, blockIdx.x, b, lo, hi)) return;
  h[threadIdx.x] = 0;
  __syncthreads();
  for (long long i = lo + threadIdx.x; i < hi; i += blockDim.x) atomicAdd(&h[(kv[i].x >> shift) & 255u], 1);
  __syncthreads();
  put_digits(tm, b, h, digits, chunk);
}

__device__ __forceinline__ int block_excl_scan256(int v, int* sh, int& total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) sh[w] = inc;
  __syncthreads();
  int before = 0;
  total = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int s = sh[k];
    if (k < w) before += s;
    total += s;
  }
  __syncthreads();
  return before + inc - v;
}

// Exclusive scan of the digit table, a chunk per block: the chunks before it are summed first.
__global__ void __launch_bounds__(256) k_radix_scan(int n, const int* __restrict__ chunk, int* __restrict__ digits) {
  __shared__ int sh[8];
  int acc = 0, before, total;
  for (int k = threadIdx.x; k < (int)blockIdx.x; k += 256) acc += chunk[k];
  block_excl_scan256(acc, sh, before);
  constexpr int kPer = kChunk / 256;
  const int base = blockIdx.x * kChunk + threadIdx.x * kPer;
  int v[kPer], sum = 0;
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    v[k] = base + k < n ? digits[base + k] : 0;
    sum += v[k];
  }
  int e = before + block_excl_scan256(sum, sh, total);
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    if (base + k < n) digits[base + k] = e;
    e += v[k];
  }
}

// One digit's stable scatter: every warp ranks its 256 consecutive pairs 32 at a time by
// __match_any_sync, the tile is reordered in shared memory and written run by run.  The last
// pass writes the caller indices alone.
__global__ void __launch_bounds__(256) k_radix_scatter(TileMap tm, int shift, const uint2* __restrict__ kv,
                                                       const int* __restrict__ digits, uint2* __restrict__ out,
                                                       int* __restrict__ perm) {
  constexpr int kWarps = 8, kItems = kSortTile / 256;
  __shared__ int wh[kWarps][256];
  __shared__ int first[256], goff[256];
  __shared__ uint2 buf[kSortTile];
  __shared__ int sh[8];
  int b;
  long long lo, hi;
  if (!stile_range(tm, blockIdx.x, b, lo, hi)) return;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int cnt = (int)(hi - lo);
#pragma unroll
  for (int k = 0; k < kWarps; ++k) wh[k][threadIdx.x] = 0;
  __syncthreads();
  uint2 p[kItems];
  int rank[kItems];
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    const int t = w * (kItems * 32) + i * 32 + lane;
    p[i] = t < cnt ? kv[lo + t] : make_uint2(0u, 0u);
  }
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    const bool ok = w * (kItems * 32) + i * 32 + lane < cnt;
    const int d = ok ? (int)((p[i].x >> shift) & 255u) : 256;
    const unsigned peers = __match_any_sync(0xffffffffu, d);
    const int lead = __ffs(peers) - 1;
    int old = 0;
    if (ok && lane == lead) {
      old = wh[w][d];
      wh[w][d] = old + __popc(peers);
    }
    rank[i] = __shfl_sync(0xffffffffu, old, lead) + __popc(peers & ((1u << lane) - 1u));
    __syncwarp();
  }
  __syncthreads();
  {
    const int d = threadIdx.x;
    int run = 0;
#pragma unroll
    for (int k = 0; k < kWarps; ++k) {
      const int t = wh[k][d];
      wh[k][d] = run;
      run += t;
    }
    int total;
    const int e = block_excl_scan256(run, sh, total);
    first[d] = e;
    const long long t0 = tm.tile_off[b], nt = tm.tile_off[b + 1] - t0;
    goff[d] = digits[256 * t0 + d * nt + (blockIdx.x - t0)] - e;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    if (w * (kItems * 32) + i * 32 + lane < cnt) {
      const int d = (int)((p[i].x >> shift) & 255u);
      buf[first[d] + wh[w][d] + rank[i]] = p[i];
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < cnt; t += 256) {
    const uint2 v = buf[t];
    const int to = goff[(v.x >> shift) & 255u] + t;
    if (perm) perm[to] = (int)v.y;
    else out[to] = v;
  }
}

// ---------------------------------------------------------------- scatter + snapshot
// Frozen partner properties of one particle at rank r (Sect. 2.5.3): s, m, N = M/m, 1/m,
// the represented mass, and the mixed form's FP32 copy (N scaled by 2^-64).
template <bool kMixed>
__device__ __forceinline__ void put_snapshot(const InstDev& p, long long r, double si, double Mi,
                                             Snap64* __restrict__ snap64, float4* __restrict__ snap32,
                                             double* __restrict__ Mr) {
  const double m = grain_mass(p, si);
  const double im = 1.0 / m;
  const double N = Mi * im;
  Snap64 sn;
  sn.s = si; sn.m = m; sn.N = N; sn.inv_m = im;
  snap64[r] = sn;
  Mr[r] = Mi;
  if (kMixed) snap32[r] = make_float4((float)si, (float)m, (float)(N * 0x1p-64), (float)im);
}

// The gas disk's (R, Z) of a particle from its search coordinates (model_pos): a patch sits
// at R = R_0 + x; the 2D radial-polar and 1D models search (R, Z, 0) and (R, 0, 0); the 3D
// and radial-azimuthal models hold (x, y, z) and (x, y, 0).
__device__ __forceinline__ void gas_coords(const InstDev& p, double X, double Y, double Z, double& R, double& Zg) {
  if (p.geometry == GD_GEOM_PATCH) R = p.r0 + X;
  else if (p.model == GD_MODEL_RZ || p.model == GD_MODEL_R) R = X;
  else R = sqrt(X * X + Y * Y);
  Zg = p.model == GD_MODEL_RZ ? Y : Z;
}

// The snapshot alone, at unchanged ranks (positions did not move since the last build); the
// mixed form's FP32 (R, Z, M) stay, its fine bin follows the new size.
template <bool kMixed>
__global__ void k_snapshot(TileMap tm, const InstDev* __restrict__ P, const double* __restrict__ s,
                           const double* __restrict__ M, const int* __restrict__ rank_of,
                           Snap64* __restrict__ snap64, float4* __restrict__ snap32, double* __restrict__ Mr,
                           float4* __restrict__ gx) {
  int b;
  long long lo, hi;
  if (!tile_range(tm, blockIdx.x, b, lo, hi)) return;
  const InstDev p = P[b];
  for (long long i = lo + threadIdx.x; i < hi; i += blockDim.x) {
    const int r = rank_of[i];
    put_snapshot<kMixed>(p, r, s[i], M[i], snap64, snap32, Mr);
    if (kMixed) reinterpret_cast<float*>(gx + r)[3] = __int_as_float(fine_bin(s[i]));
  }
}

// Spatial groups: the round's particles (the list act) broadcast -- their live sizes become
// the sizes partners read (sb, caller order) -- and their snapshot entries follow; the other
// particles' entries keep their last broadcast.
template <bool kMixed>
__global__ void k_broadcast_snapshot(const unsigned long long* __restrict__ total, const int* __restrict__ act,
                                     const long long* __restrict__ off, int n_inst, const InstDev* __restrict__ P,
                                     const int* __restrict__ perm, const double* __restrict__ s,
                                     double* __restrict__ sb, const double* __restrict__ M,
                                     Snap64* __restrict__ snap64, float4* __restrict__ snap32,
                                     double* __restrict__ Mr, float4* __restrict__ gx) {
  const long long n = (long long)*total;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x) {
    const int r = act[t];
    const int ci = perm[r];
    const double si = s[ci];
    sb[ci] = si;
    put_snapshot<kMixed>(P[inst_of(off, n_inst, r)], r, si, M[ci], snap64, snap32, Mr);
    if (kMixed) reinterpret_cast<float*>(gx + r)[3] = __int_as_float(fine_bin(si));
  }
}

// ---------------------------------------------------------------- rank-space copies and leaves
// A warp per leaf (32 consecutive ranks of one instance): lane = rank, the caller's arrays
// gathered, every rank-space array written coalesced, and the leaf's box.  Bound by the gather:
// doubles read at random cost a 32-byte sector each, 570 B per particle through DRAM for about 160.
// (The scatter it replaces, lane = caller index, stored at random ranks in partial sectors: fewer
// bytes, 467, but 0.93 ms for 2^22 particles against 0.40.)
template <bool kMixed, bool kLists>
__global__ void __launch_bounds__(256) k_gather(int n_leaves, int n_inst, const int* __restrict__ leaf_off,
                                                const long long* __restrict__ off, const InstDev* __restrict__ P,
                                                const TreeDev* __restrict__ tree, const double* __restrict__ x,
                                                const double* __restrict__ y, const double* __restrict__ z,
                                                const double* __restrict__ s, const double* __restrict__ M,
                                                const int* __restrict__ perm, int* __restrict__ rank_of,
                                                Pos64* __restrict__ pos64, int4* __restrict__ posq,
                                                Snap64* __restrict__ snap64, float4* __restrict__ snap32,
                                                double* __restrict__ Mr, float4* __restrict__ gx,
                                                float4* __restrict__ na, float2* __restrict__ nb, StateDev* st) {
  const int lane = threadIdx.x & 31;
  const int leaf = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (leaf >= n_leaves) return;
  const int b = lev_inst(leaf_off, n_inst, leaf);
  const long long r = off[b] + (long long)(leaf - leaf_off[b]) * kLeaf + lane;
  const InstDev& p = P[b];
  const TreeDev& T = tree[b];
  if (leaf == leaf_off[b] && lane < 3) {           // the bounds are spent: reset for the next build
    st[p.unit0].bmin[lane] = ~0ull;
    st[p.unit0].bmax[lane] = 0ull;
  }
  bool fin = false;
  int u[3] = {0, 0, 0};
  if (r < off[b + 1]) {
    const int i = perm[r];
    double xi, yi, zi;
    model_pos(p.model, x[i], y[i], z[i], xi, yi, zi);
    Pos64 q;
    q.x = xi; q.y = yi; q.z = zi; q.j = i;
    pos64[r] = q;
    if (!kLists) {                                  // kLists: gd_neighbors_fixed, positions alone
      const double si = s[i], Mi = M[i];
      rank_of[i] = (int)r;
      put_snapshot<kMixed>(p, r, si, Mi, snap64, snap32, Mr);
      if (kMixed) {
        double R, Zg;
        gas_coords(p, xi, yi, zi, R, Zg);
        gx[r] = make_float4((float)R, (float)Zg, (float)Mi, __int_as_float(fine_bin(si)));
      }
    }
    fin = isfinite(xi) && isfinite(yi) && isfinite(zi);
    if (fin) { u[0] = to_unit(T, 0, xi); u[1] = to_unit(T, 1, yi); u[2] = to_unit(T, 2, zi); }
    posq[r] = make_int4(u[0], u[1], u[2], fin ? i : ~i);
  }
  int mn[3], mx[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    mn[a] = __reduce_min_sync(0xffffffffu, fin ? u[a] : INT_MAX);
    mx[a] = __reduce_max_sync(0xffffffffu, fin ? u[a] : -1);
  }
  if (lane == 0) {
    const float inf = __int_as_float(0x7F800000);
    const bool e = mx[0] < 0;                       // no finite particle: a box nothing meets
    na[leaf] = make_float4(e ? inf : __int2float_rd(mn[0]), e ? inf : __int2float_rd(mn[1]),
                           e ? inf : __int2float_rd(mn[2]), e ? -inf : __int2float_ru(mx[0]));
    nb[leaf] = make_float2(e ? -inf : __int2float_ru(mx[1]), e ? -inf : __int2float_ru(mx[2]));
  }
}

// One upper level: a warp per node, lane = child.
__global__ void __launch_bounds__(256) k_levels(int lev, int n_inst, const int* __restrict__ lev_tab,
                                                const TreeDev* __restrict__ tree, float4* __restrict__ na,
                                                float2* __restrict__ nb) {
  const int lane = threadIdx.x & 31;
  const int* tab = lev_tab + (long long)lev * (n_inst + 1);
  const int node = tab[0] + blockIdx.x * 8 + (threadIdx.x >> 5);
  if (node >= tab[n_inst]) return;
  const int b = lev_inst(tab, n_inst, node);
  const TreeDev& T = tree[b];
  const int c = (node - tab[b]) * kLeaf + lane;
  const float inf = __int_as_float(0x7F800000);
  float4 A = make_float4(inf, inf, inf, -inf);
  float2 B = make_float2(-inf, -inf);
  if (c < T.lev_n[lev - 1]) { A = na[T.lev_off[lev - 1] + c]; B = nb[T.lev_off[lev - 1] + c]; }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    A.x = fminf(A.x, __shfl_xor_sync(0xffffffffu, A.x, o));
    A.y = fminf(A.y, __shfl_xor_sync(0xffffffffu, A.y, o));
    A.z = fminf(A.z, __shfl_xor_sync(0xffffffffu, A.z, o));
    A.w = fmaxf(A.w, __shfl_xor_sync(0xffffffffu, A.w, o));
    B.x = fmaxf(B.x, __shfl_xor_sync(0xffffffffu, B.x, o));
    B.y = fmaxf(B.y, __shfl_xor_sync(0xffffffffu, B.y, o));
  }
  if (lane == 0) { na[node] = A; nb[node] = B; }
}

}  // namespace gd

// ---------------------------------------------------------------- launcher
namespace gd {

int num_tiles(gd_ctx* c) { return c->n_tiles; }

std::vector<long long> tile_table(const std::vector<long long>& off, const std::vector<int>& tile) {
  std::vector<long long> t(off.size(), 0);
  for (size_t b = 0; b + 1 < off.size(); ++b) t[b + 1] = t[b] + (off[b + 1] - off[b] + tile[b] - 1) / tile[b];
  return t;
}

static long long ceil_div(long long a, long long b) { return (a + b - 1) / b; }

// Sizes of the sort and of the tree from the offsets off[n_inst + 1]: the number of passes (see
// sort_key), the sort tiles (stile_off[n_inst + 1]) and digit-table chunks, and the node ranges of
// every level (lev[kMaxLev * (n_inst + 1)], kept by the context), level by level with the instances
// concatenated inside a level.  Allocates nothing: gd_neighbors_fixed plans each of its calls.
void tree_plan(gd_ctx* c, const long long* off, int* lev, long long* stile_off) {
  const int n = c->n_inst;
  long long nmax = 0;
  stile_off[0] = 0;
  for (int b = 0; b < n; ++b) {
    nmax = std::max(nmax, off[b + 1] - off[b]);
    stile_off[b + 1] = stile_off[b] + ceil_div(off[b + 1] - off[b], kSortTile);
  }
  c->n_stiles = (int)stile_off[n];
  c->n_chunks = (int)ceil_div(256LL * c->n_stiles, kChunk);
  c->sort_passes = nmax <= (1LL << 18) ? 3 : 4;
  c->lev = lev;
  c->max_lev = 1;
  int at = 0;
  for (int l = 0; l < kMaxLev; ++l) {
    int* tab = lev + (size_t)l * (n + 1);
    for (int b = 0; b < n; ++b) {
      long long cnt = ceil_div(off[b + 1] - off[b], kLeaf);
      for (int k = 0; k < l; ++k) cnt = cnt > kLeaf ? ceil_div(cnt, kLeaf) : 0;
      tab[b] = at;
      at += (int)cnt;
      if (cnt > 0) c->max_lev = l + 1;
    }
    tab[n] = at;
    if (l == 0) c->n_leaves = at;
  }
  c->n_nodes = at;
}

// The sizes partners read: the live sizes, or with spatial groups each particle's size as its
// group last broadcast it.
static const double* partner_sizes(gd_ctx* c) { return c->grouped ? c->d_sb : c->s; }

// Partner snapshot refresh at unchanged ranks (gd_collide's later intervals).
cudaError_t launch_snapshot(gd_ctx* c) {
  time_begin(c, 0);
  const int nt = num_tiles(c);
  const double* s = partner_sizes(c);
  if (c->precision == GD_MIXED)
    k_snapshot<true><<<nt, 256, 0, c->stream>>>(tile_map(c), c->d_inst, s, c->M, c->d_rank_of, c->d_snap64,
                                                c->d_snap32, c->d_Mr, c->d_gx);
  else
    k_snapshot<false><<<nt, 256, 0, c->stream>>>(tile_map(c), c->d_inst, s, c->M, c->d_rank_of, c->d_snap64,
                                                 c->d_snap32, c->d_Mr, c->d_gx);
  time_end(c);
  c->launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_broadcast_snapshot(gd_ctx* c) {
  time_begin(c, 0);
  const unsigned long long* total = c->d_counters + 10;
  const int grid = c->num_sms * 8;
  if (c->precision == GD_MIXED)
    k_broadcast_snapshot<true><<<grid, 256, 0, c->stream>>>(total, c->d_act, c->d_off, c->n_inst, c->d_inst,
                                                            c->d_perm, c->s, c->d_sb, c->M, c->d_snap64,
                                                            c->d_snap32, c->d_Mr, c->d_gx);
  else
    k_broadcast_snapshot<false><<<grid, 256, 0, c->stream>>>(total, c->d_act, c->d_off, c->n_inst, c->d_inst,
                                                             c->d_perm, c->s, c->d_sb, c->M, c->d_snap64,
                                                             c->d_snap32, c->d_Mr, c->d_gx);
  time_end(c);
  c->launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_stats(gd_ctx* c, double* d_sums) {
  time_begin(c, 6);
  double* part = d_sums + 3 * (long long)c->n_inst;
  k_stats_tile<<<c->n_tiles, 256, 0, c->stream>>>(tile_map(c), c->d_inst, c->s, c->M, part);
  k_stats_inst<<<c->n_inst, 256, 0, c->stream>>>(c->d_tile_off, part, d_sums);
  time_end(c);
  return cudaGetLastError();
}

cudaError_t launch_tree(gd_ctx* c) {
  TileMap tm;
  tm.off = c->d_off;
  tm.n_inst = c->n_inst;
  tm.tile = nullptr;                                // (kSortTile: stile_range)
  tm.tile_off = c->d_stile_off;
  const int nt = c->n_stiles;
  cudaStream_t st = c->stream;
  time_begin(c, 0);
  cudaMemsetAsync(c->d_chunk, 0, sizeof(int) * (size_t)c->sort_passes * c->n_chunks, st);
  k_bounds<<<nt, 256, 0, st>>>(tm, c->d_inst, c->x, c->y, c->z, c->d_state);
  if (c->check_cells) {
    k_check_cells<<<1, 256, 0, st>>>(c->d_inst, c->d_state, c->n_inst, c->cell_factor, c->cell_xsplit, c->cell_cap);
    c->launches += 1;
  }
  k_keys<<<nt, 256, 0, st>>>(tm, c->d_inst, c->d_state, c->d_tree, c->sort_passes, c->x, c->y, c->z, c->d_kv[0],
                             c->d_digits, c->d_chunk);
  for (int p = 0; p < c->sort_passes; ++p) {
    const uint2* src = c->d_kv[p & 1];
    int* chunk = c->d_chunk + (size_t)p * c->n_chunks;
    if (p > 0) k_radix_hist<<<nt, 256, 0, st>>>(tm, 8 * p, src, c->d_digits, chunk);
    k_radix_scan<<<c->n_chunks, 256, 0, st>>>(256 * nt, chunk, c->d_digits);
    k_radix_scatter<<<nt, 256, 0, st>>>(tm, 8 * p, src, c->d_digits, c->d_kv[(p & 1) ^ 1],
                                        p + 1 == c->sort_passes ? c->d_perm : nullptr);
  }
  const double* s = partner_sizes(c);
  const int nb = (c->n_leaves + 7) / 8;
  auto* gather = c->lists_only ? k_gather<false, true> : c->precision == GD_MIXED ? k_gather<true, false>
                                                                                  : k_gather<false, false>;
  gather<<<nb, 256, 0, st>>>(c->n_leaves, c->n_inst, c->d_lev, c->d_off, c->d_inst, c->d_tree, c->x, c->y, c->z, s,
                             c->M, c->d_perm, c->d_rank_of, c->d_pos64, c->d_posq, c->d_snap64, c->d_snap32, c->d_Mr,
                             c->d_gx, c->d_node_a, c->d_node_b, c->d_state);
  for (int l = 1; l < c->max_lev; ++l) {
    const int* tab = c->lev + (size_t)l * (c->n_inst + 1);
    const int nodes = tab[c->n_inst] - tab[0];
    k_levels<<<(nodes + 7) / 8, 256, 0, st>>>(l, c->n_inst, c->d_lev, c->d_tree, c->d_node_a, c->d_node_b);
  }
  time_end(c);
  c->launches += 2 + 3 * c->sort_passes - 1 + 1 + (c->max_lev - 1);
  return cudaGetLastError();
}

}  // namespace gd
