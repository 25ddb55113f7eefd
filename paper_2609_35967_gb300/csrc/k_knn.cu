// k_knn.cu -- K nearest neighbours over the Hilbert-ordered tree (Sect. 2.5.1).
//
// A warp takes one leaf: 32 queries that are consecutive on the curve, lane = query.  Their
// balls overlap almost wholly, so the warp walks the tree once for all of them, stages the
// candidates near the leaf's box in shared memory and every lane tests the same candidate at
// the same time, read by broadcast: no lane waits for another's rows, and a test is a handful
// of FP32 instructions (two candidates per packed instruction).
//
//  find   : the leaves whose box comes within the largest radius of the queries' box, level by
//           level, lane = child, four nodes at a time;
//  visit  : four of these leaves' particles are loaded at a time (lane = particle), those within
//           the radius of the queries' box are queued in shared memory;
//  test   : every lane tests the same queued candidate at the same time, read by broadcast: FP32
//           D in units of the instance's quantum, two candidates per packed instruction, a hit
//           appended to the lane's list under a predicate;
//  decide : |sqrt(D) - d| <= 10u sqrt(D) + E (u = 2^-24) separates certain members from a band
//           ranked exactly in FP64 by (d^2, caller index), d^2 = (dx dx + dy dy) + dz dz (no
//           FMA, minimum image).  The lists are the exact FP64 ones in both forms;
//  output : d_i = sqrt of the (K-1)-th d^2, V_i with the flat-boundary caps, and the row: the
//           particle itself, then its members by ascending caller index.
//
// k_knn<., ., true>  (particles that did not move): the radius is the previous build's d_i and a
//           hair, so the K-1 members and rarely more are hit.  Leaves where that fails for many
//           queries (no earlier build, or the caller changed the positions) are listed for
// k_knn<., ., false> (moved particles, first builds and those leaves): the hits go to a buffer of
//           two to three times the members as words (upper bits of D, place), and the K-1
//           smallest are chosen.  A query with too few or too many hits walks again with a
//           rescaled radius; one that stays undecided is listed for
// k_knn_exact: a warp per query, branch and bound over the tree with FP64 keys (d^2, caller
//           index) in a list held across the warp's lanes; exact for any ties.
//
// Bound by instruction issue and the latency of dependent steps, not by HBM: 456 warp
// instructions per particle at K = 32 (a uniform cell grid walked by each lane alone took 654,
// with its lanes waiting for one another), 55% of the issue slots at 16 warps an SM (fixed latencies
// 2.3, loads 1.7 and shared memory 1.1 stalled warps per issue), about 510 candidates tested per leaf
// of 32 queries.  Builds of a 2^22-particle disk, K = 32: static 5.0 -> 3.6 ms, first
// 36.6 -> 16 ms; after a push 10.8 -> 6.5 ms (2^20: 2.6 -> 1.6); K = 48 after a push 14.7 -> 8.3
// ms.  gd_neighbors_fixed of 50,001 particles, K = 32: 3.6 -> 1.1 ms.  The code is kept
// small on purpose (loops not unrolled, the reduced models' volume out of line): unrolled, it
// missed the instruction cache and the same builds took half again as long.
#include <climits>

#include "gd_ctx.h"
#include "gd_physics.cuh"

namespace gd {

constexpr int kExtra = 4;         // static: hits beyond the members that are sorted out
constexpr int kBand = 8;          // band entries resolved in FP64 per query
constexpr int kPad = 33;          // words per entry row of a warp's buffer (32 lanes + 1)
constexpr int kQueue = 160;       // candidates staged: what is left over and four leaves
constexpr uint32_t kPlaceMask = 8191u;
constexpr int kSlack = 8;
constexpr int kSlots = 256;       // leaves one walk may reach (8 + 5 bits of a candidate's place)
constexpr int kFront = 64;        // nodes of an upper level one walk may reach
constexpr int kShiftBit = 26;     // an instance's leaves fit below (2^31 particles)
constexpr int kMaxWarps = 20;     // warps an SM holds at most, the registers shared among them
                                  // (16: 4% slower, 24: 5% slower, both by spills or idle slots)
constexpr int kTries = 6;
constexpr float kMovedFac = 1.04f;  // after a push: 1.03 to 1.08 within 5% of one another (2^20 disk)
constexpr float kLeafShare = 0.24f;  // first radius: see k_knn
constexpr int kOver = 4;          // a lane with more than kOver times its buffer's entries ends its walk
constexpr float kSplit = 40.0f;   // see k_knn
constexpr float kRel = 10.0f * 5.9604645e-8f;
constexpr unsigned kAll = 0xffffffffu;

struct KnnArgs {
  long long N;
  int K, n_inst, n_leaves;
  const long long* off;
  const int* leaf_off;            // [n_inst + 1] first leaf of each instance
  const InstDev* P;
  const TreeDev* tree;
  const float4* na;               // node boxes
  const float2* nb;
  const int4* posq;
  const Pos64* pos64;
  const int* rank_of;
  int* nbr;
  double* dist;
  double* V;
  float* pref32;                  // mixed form: FP32 rate prefactor (NULL in the FP64 form)
  double* dprev;                  // caller order: d_i of the last build (0: unknown)
  StateDev* st;
  int* leaves;                    // leaves (and parts of them) with undecided queries (their dist is -1)
  unsigned long long* leaves_n;
  int listed;                     // 1: only the listed leaves and their undecided queries
  int* redo;                      // queries for k_knn_exact
  unsigned long long* redo_n;
  int fixed;                      // gd_neighbors_fixed: rows in the caller's order and indices, dist (caller
                                  // order, or null) the only other result
  int parts;                      // warps a leaf's queries are spread over (1, 2 or 4)
  int packed;                     // caller indices leave room for a buffer entry in a sort key
};

__device__ double sample_volume_reduced(const InstDev& P, double d, double x, double y);

__device__ __forceinline__ double sample_volume(const InstDev& P, double d, double x, double y) {
  if (P.kernel_mode != GD_KERNEL_PHYSICAL) return 1.0;
  if (P.model != GD_MODEL_3D) return sample_volume_reduced(P, d, x, y);
  double V = (4.0 * kPi / 3.0) * d * d * d;
  if (P.geometry == GD_GEOM_DISK) {
    const double R2 = x * x + y * y;
    const double a = P.R_in + d, bo = P.R_out - d;
    // clear of both edges by a relative 1e-12, far above the rounding of R2 and of the
    // squares: no cap applies and R is not needed
    if (R2 > a * a * (1.0 + 1e-12) && bo > 0.0 && R2 < bo * bo * (1.0 - 1e-12)) return V;
    double R = sqrt(R2);
    double h = R - P.R_in;
    if (h > 0.0 && h < d) V -= kPi * (d - h) * (d - h) * (2.0 * d + h) / 3.0;
    h = P.R_out - R;
    if (h > 0.0 && h < d) V -= kPi * (d - h) * (d - h) * (2.0 * d + h) / 3.0;
  }
  return V;
}

// Reduced models (Sect. 2.5.1), (x, y) the query's coordinates in its model: the sampled
// area (a disk of radius d less the circular segments beyond a radial edge taken as a
// straight line; the 1D annulus [R - d, R + d] clipped at the edges) times 2 pi R (2D
// radial-polar: a toroidal volume) or times the vertical length sqrt(2 pi (H_i^2 + H_j^2))
// of the Gaussian average with H_i = H_j = H_g(R_i) (vertically integrated models).
// Out of line: the gas disk's powers and the arc cosines are 70 KB of code.
__device__ __noinline__ double sample_volume_reduced(const InstDev& P, double d, double x, double y) {
  double R;
  if (P.geometry == GD_GEOM_PATCH) R = P.r0 + x;
  else if (P.model == GD_MODEL_RPHI) R = __dsqrt_rn(__dadd_rn(__dmul_rn(x, x), __dmul_rn(y, y)));
  else R = x;
  double A;
  if (P.model == GD_MODEL_R) {
    const double lo = R - d > P.R_in ? R - d : P.R_in;
    const double hi = R + d < P.R_out ? R + d : P.R_out;
    A = kPi * (hi * hi - lo * lo);
  } else {
    A = kPi * d * d;
    if (P.geometry == GD_GEOM_DISK) {
      double h = R - P.R_in;
      if (h > 0.0 && h < d) A -= d * d * acos(h / d) - h * sqrt(d * d - h * h);
      h = P.R_out - R;
      if (h > 0.0 && h < d) A -= d * d * acos(h / d) - h * sqrt(d * d - h * h);
    }
  }
  if (P.model == GD_MODEL_RZ) return A * 2.0 * kPi * R;
  const Gas g = gas_RZ(P, R, 0.0);
  return A * sqrt(2.0 * kPi * (g.H * g.H + g.H * g.H));
}

// Minimum-image FP64 d^2 of rank r from the query: the oracle's expression.
__device__ __forceinline__ double d2_fp64(const Pos64* __restrict__ pos64, int r, double qx, double qy,
                                          double qz, double bx, double by, long long& j) {
  const double2* pp = reinterpret_cast<const double2*>(pos64 + r);
  double2 a = __ldg(pp), b = __ldg(pp + 1);
  double dx = a.x - qx, dy = a.y - qy, dz = b.x - qz;
  if (bx > 0.0) {
    if (dx > 0.5 * bx) dx -= bx; else if (dx < -0.5 * bx) dx += bx;
    if (dy > 0.5 * by) dy -= by; else if (dy < -0.5 * by) dy += by;
  }
  j = __double_as_longlong(b.y);
  return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

// Result of one query: d_i, V_i, the rate prefactor and the next build's radius.
__device__ __forceinline__ void put_result(const KnnArgs& A, const InstDev& P, long long q, int ci, double d2max,
                                           double x, double y) {
  const double d = sqrt(d2max);
  if (A.fixed) {
    if (A.dist) A.dist[ci] = d;
    return;
  }
  A.dist[q] = d;
  const double Vq = sample_volume(P, d, x, y);
  A.V[q] = Vq;
  if (A.pref32) A.pref32[q] = (float)rate_prefactor(P, Vq, A.K, true);
  A.dprev[ci] = d;
}

// A query without K-1 others (or a place): the row stays valid (the particle against itself) with
// an infinite measure, so the particle gets no rate, and the status reports it.  (Fixed: -1.)
__device__ __forceinline__ void no_list(const KnnArgs& A, const InstDev& P, long long q, int ci) {
  if (A.fixed) {
    for (int k = 0; k < A.K; ++k) A.nbr[(long long)ci * A.K + k] = -1;
    if (A.dist) A.dist[ci] = -1.0;
    return;
  }
  for (int k = 0; k < A.K; ++k) A.nbr[q * (long long)A.K + k] = (int)q;
  A.dist[q] = 0.0;
  A.V[q] = __longlong_as_double(0x7FF0000000000000ll);
  if (A.pref32) A.pref32[q] = 0.0f;
  A.dprev[ci] = 0.0;
  set_status(&A.st[P.unit0], GD_ST_KNN);
}

// Squared distance between two intervals' or a point's and a box's nearest points, per axis.
__device__ __forceinline__ float gap(float alo, float ahi, float blo, float bhi) {
  return fmaxf(fmaxf(alo - bhi, blo - ahi), 0.0f);
}

__device__ __forceinline__ float grow(float rho, int found, int L, int cap) {
  // few found: the count says little, so grow by at least a quarter
  const float g = cbrtf(0.5f * (float)(L + cap) / (float)(found > 0 ? found : 1));
  return rho * fminf(fmaxf(g, 4 * found >= L ? 1.01f : 1.25f), 2.0f);
}

// Two FP32 values in one register pair and their packed arithmetic (each half rounded like the
// scalar instruction).
__device__ __forceinline__ unsigned long long pack2(float a, float b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(unsigned long long v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// Candidates of a walk, relative to the queries' box; place: the candidate's leaf (its entry in
// tab) and lane.
struct Queue {
  float x[kQueue + 32], y[kQueue + 32], z[kQueue + 32];   // past kQueue: what is not kept
  unsigned place[kQueue + 32];
};

// The walk's state common to the warp, and this lane's query.
struct Walk {
  float hx, hy, hz;               // half extents of the active queries' box around ref
  float rm2;                      // squared radius of the walk (box to node, box to particle)
  float qx, qy, qz, rhof2;        // this lane: query relative to ref, squared radius (< 0: idle)
  unsigned at;                    // shared address of the lane's next hit
  unsigned past;                  // hits not kept
};

__device__ __forceinline__ unsigned shared_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

// Appends a place or word to the lane's hits when D <= r2; the address moves on for every hit.
template <bool kStatic>
__device__ __forceinline__ void append(float D, float r2, unsigned v, unsigned& at) {
  if (kStatic)
    asm volatile("{\n .reg .pred p;\n setp.le.f32 p, %1, %2;\n @p st.shared.u16 [%0], %3;\n @p add.u32 %0, %0, 68;\n}"
                 : "+r"(at) : "f"(D), "f"(r2), "r"(v) : "memory");
  else
    asm volatile("{\n .reg .pred p;\n setp.le.f32 p, %1, %2;\n @p st.shared.u32 [%0], %3;\n @p add.u32 %0, %0, 132;\n}"
                 : "+r"(at) : "f"(D), "f"(r2), "r"(v) : "memory");
}

// 32 candidates of the queue from b on against every lane's ball.  A hit is appended at once,
// under a predicate: static, its place; otherwise a word of the upper bits of D and the place.
// (Hits kept as bits and visited afterwards took 8000 instructions per leaf of 500 candidates
// against 4500: a leaf's candidates are near one another, so a few lanes have most of the hits
// among 32 of them and the others wait.)
// Past full the lane's hits are only counted (static: its walk ends): the buffers have kSlack
// rows more than they may keep, and the address is held back every kSlack candidates.
template <bool kStatic>
__device__ __forceinline__ void test32(const Queue* Q, int b, Walk& W, unsigned full) {
  constexpr unsigned kStep = kStatic ? 68 : 4 * kPad;
  const unsigned long long nx = pack2(-W.qx, -W.qx), ny = pack2(-W.qy, -W.qy), nz = pack2(-W.qz, -W.qz);
  auto hit = [&](float D, unsigned place) {
    append<kStatic>(D, W.rhof2, kStatic ? place : (__float_as_uint(D) & ~kPlaceMask) | place, W.at);
  };
#pragma unroll 1
  for (int k = b; k < b + 32; k += 8) {
#pragma unroll
    for (int h = k; h < k + 8; h += 4) {
      const uint4 P = *reinterpret_cast<const uint4*>(Q->place + h);
      const ulonglong2 X = *reinterpret_cast<const ulonglong2*>(Q->x + h);
      const ulonglong2 Y = *reinterpret_cast<const ulonglong2*>(Q->y + h);
      const ulonglong2 Z = *reinterpret_cast<const ulonglong2*>(Q->z + h);
      float d0, d1, d2, d3;
      unsigned long long dx = add2(X.x, nx), dy = add2(Y.x, ny), dz = add2(Z.x, nz);
      unpack2(fma2(dz, dz, fma2(dy, dy, mul2(dx, dx))), d0, d1);
      dx = add2(X.y, nx); dy = add2(Y.y, ny); dz = add2(Z.y, nz);
      unpack2(fma2(dz, dz, fma2(dy, dy, mul2(dx, dx))), d2, d3);
      hit(d0, P.x);
      hit(d1, P.y);
      hit(d2, P.z);
      hit(d3, P.w);
    }
    if (W.at > full) {
      if (kStatic) W.rhof2 = -1.0f;
      else W.past += (W.at - full) / kStep;
      W.at = kStatic ? full + kStep : full;
    }
  }
}

// The leaves whose box comes within the walk's radius of the queries' box (g: lo and hi, in
// units), for one shift (code), added to tab: level by level, four nodes' children loaded
// together, since every load waits several hundred cycles.  Returns the new count, or -1 when a
// level does not fit.
__device__ __forceinline__ int find_leaves(const KnnArgs& A, const TreeDev& T, const float (&g)[6], float rm2,
                                           int code, int* tab, int cnt, int* front, int lane) {
  auto near = [&](int l, int first) -> bool {
    const int c = first + lane;
    if (first < 0 || c >= T.lev_n[l]) return false;
    const float4 a = __ldg(A.na + T.lev_off[l] + c);
    const float2 b = __ldg(A.nb + T.lev_off[l] + c);
    const float gx = gap(a.x, a.w, g[0], g[3]), gy = gap(a.y, b.x, g[1], g[4]), gz = gap(a.z, b.y, g[2], g[5]);
    return gx * gx + gy * gy + gz * gz <= rm2;
  };
  const unsigned below = (1u << lane) - 1u;
  const int top = T.nlev - 1;
  int nf;
  {
    const bool h = near(top, 0);
    const unsigned m = __ballot_sync(kAll, h);
    nf = __popc(m);
    if (top == 0) {
      if (cnt + nf > kSlots) return -1;
      if (h) tab[cnt + __popc(m & below)] = lane | code;
      return cnt + nf;
    }
    if (h) front[__popc(m & below)] = lane;
  }
#pragma unroll 1
  for (int l = top - 1; l >= 0; --l) {
    __syncwarp();
    const int* from = front + ((top - 1 - l) & 1) * kFront;
    int* to = l == 0 ? tab : front + ((top - l) & 1) * kFront;
    const int room = l == 0 ? kSlots : kFront;
    int n = l == 0 ? cnt : 0;
    const int tag = l == 0 ? code : 0;
#pragma unroll 1
    for (int k = 0; k < nf; k += 4) {
      int f[4];
      bool h[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) f[u] = k + u < nf ? from[k + u] * kLeaf : -1;
#pragma unroll
      for (int u = 0; u < 4; ++u) h[u] = near(l, f[u]);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const unsigned m = __ballot_sync(kAll, h[u]);
        const int at = n + __popc(m & below);
        n += __popc(m);
        if (h[u] && at < room) to[at] = (f[u] + lane) | tag;
      }
    }
    if (n > room) return -1;
    nf = n;
  }
  return nf;
}

// The leaves of tab: their particles within the walk's radius of the queries' box are queued and
// tested, four leaves' particles loaded together.
template <bool kStatic>
__device__ __forceinline__ void visit(const KnnArgs& A, const TreeDev& T, Queue* Q, const int* tab,
                                      int cnt, long long r0, int n, const int3 ref, bool per, Walk& W,
                                      unsigned full, unsigned over, int lane) {
  const int4* __restrict__ pq = A.posq + r0;
  constexpr int kLow = (1 << kShiftBit) - 1;
  int qn = 0;
#pragma unroll 1
  for (int s = 0; s < cnt; s += 4) {
    int4 c[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = s + u < cnt ? tab[s + u] : -1;
      const int i = (e & kLow) * kLeaf + lane;
      c[u] = make_int4(0, 0, 0, -1);
      if (e >= 0 && i < n) c[u] = __ldg(pq + i);
      if (per && e >= 0) {
        const int sc = e >> kShiftBit;
        c[u].x += (sc % 3 - 1) * T.boxq[0];
        c[u].y += (sc / 3 - 1) * T.boxq[1];
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float x = (float)(c[u].x - ref.x), y = (float)(c[u].y - ref.y), z = (float)(c[u].z - ref.z);
      const float gx = fmaxf(fabsf(x) - W.hx, 0.f), gy = fmaxf(fabsf(y) - W.hy, 0.f), gz = fmaxf(fabsf(z) - W.hz, 0.f);
      const bool keep = c[u].w >= 0 && gx * gx + gy * gy + gz * gz <= W.rm2;
      const unsigned m = __ballot_sync(kAll, keep);
      const int at = keep ? qn + __popc(m & ((1u << lane) - 1u)) : kQueue + lane;
      Q->x[at] = x;
      Q->y[at] = y;
      Q->z[at] = z;
      Q->place[at] = (unsigned)((s + u) * 32 + lane);
      qn += __popc(m);
    }
    const bool last = s + 4 >= cnt;
    if (last && (qn & 31)) {
      // the rest, padded with candidates no ball holds
      const int to = (qn + 31) & ~31;
      if (qn + lane < to) { Q->x[qn + lane] = 3e18f; Q->y[qn + lane] = 0.0f; Q->z[qn + lane] = 0.0f; }
      qn = to;
    }
    __syncwarp();
    int b = 0;
#pragma unroll 1
    for (; b + 32 <= qn; b += 32) test32<kStatic>(Q, b, W, full);
    __syncwarp();
    if (b) {
      qn -= b;
      float x = 0.f, y = 0.f, z = 0.f;
      unsigned p = 0;
      if (lane < qn) { x = Q->x[b + lane]; y = Q->y[b + lane]; z = Q->z[b + lane]; p = Q->place[b + lane]; }
      __syncwarp();
      if (lane < qn) { Q->x[lane] = x; Q->y[lane] = y; Q->z[lane] = z; Q->place[lane] = p; }
      // far too many hits: the lane's walk ends
      if (!kStatic && W.past > over) W.rhof2 = -1.0f;
      if (!__any_sync(kAll, W.rhof2 >= 0.0f)) return;
    }
  }
}

// Bound of the error of an FP32 distance apart from the relative 10u: a unit per axis from the
// quantisation (half of one more from the rounded periodic extent) and 2.5u of the relative
// coordinates, which reach the half extents plus the radius.
__device__ __forceinline__ float error_bound(bool per, float reach) {
  return 1.75f * ((per ? 1.6f : 1.1f) + 2.5f * 5.9604645e-8f * (reach * 1.001f + 64.0f));
}

// Rank of a candidate from its place.
__device__ __forceinline__ int rank_of_place(const int* tab, int place, int r0) {
  return r0 + (tab[place >> 5] & ((1 << kShiftBit) - 1)) * kLeaf + (place & 31);
}

// Static: around the D of the (K-1)-th (dk), keys below lo are certain members and keys above
// hi none; inside: every particle as near is hit by the ball of radius rho.
struct Margins {
  float lo, hi;
  bool inside;
};
__device__ __forceinline__ Margins margins(float dk, float rho, float E) {
  const float sq = sqrtf(dk);
  const float hi_tau = (sq * (1.0f + kRel) * 1.000001f + E) * 1.000001f;
  const float lo_tau = (sq * (1.0f - kRel) * 0.999999f - E) * 0.999999f;
  const float tlo = fmaxf((lo_tau - E) / (1.0f + kRel), 0.0f), thi = (hi_tau + E) / (1.0f - kRel);
  return Margins{tlo * tlo * 0.999999f, thi * thi * 1.000001f, hi_tau <= rho};
}

// The L-th smallest of a lane's n distinct words.  Counts go like D^(3/2): a threshold with L
// to L + 3 words is interpolated on D, then the largest four below it are ordered.
__device__ __forceinline__ uint32_t lth_word(const uint32_t* words, int n, int L, float dmax, int lane) {
  uint32_t t = 0xFFFFFFFFu;
  int c = n;
  if (n - L > 3) {
    uint32_t lo = 0u, hi = 0xFFFFFFFFu;       // counts clo and chi of the words below them
    int clo = 0, chi = n;
    float l3 = 0.0f, h3 = dmax * sqrtf(dmax); // their D^(3/2)
#pragma unroll 1
    for (int it = 0; it < 40 && chi - L > 3; ++it) {
      const float f = ((float)L + 1.5f - (float)clo) / (float)(chi - clo);
      float g = cbrtf(l3 + f * (h3 - l3));
      g = g * g;
      uint32_t x = __float_as_uint(g);
      if (it >= 8 || x <= lo || x >= hi) x = lo + (hi - lo) / 2u;
      int k = 0;
      for (int e = 0; e < n; ++e) k += words[e * kPad + lane] < x ? 1 : 0;
      const float fx = __uint_as_float(min(x, 0x7F000000u));
      if (k >= L) { hi = x; chi = k; h3 = fx * sqrtf(fx); } else { lo = x; clo = k; l3 = fx * sqrtf(fx); }
    }
    t = hi;
    c = chi;
  }
  uint32_t m0 = 0, m1 = 0, m2 = 0, m3 = 0;
  for (int e = 0; e < n; ++e) {
    uint32_t v = words[e * kPad + lane];
    if (v >= t) v = 0;
    uint32_t u = max(m0, v); v = min(m0, v); m0 = u;
    u = max(m1, v); v = min(m1, v); m1 = u;
    u = max(m2, v); v = min(m2, v); m2 = u;
    m3 = max(m3, v);
  }
  const int left = c - L;
  return left == 0 ? m0 : left == 1 ? m1 : left == 2 ? m2 : m3;
}

// Members of one query from its n words (L <= n <= CAP, its own among them), compacted to the
// front as ranks; d2max the (K-1)-th d^2.  A word's D lies between its upper bits and the next
// value of them; with the FP32 error bound that gives the band of words that FP64 decides.
// 1: done, 0: undecided, -1: the ball must grow.
__device__ __forceinline__ int members(const KnnArgs& A, const TreeDev& T, uint32_t* words, const int* tab,
                                       int r0, int self, int n, int L, float rho, float E,
                                       float rhof2, double x, double y, double z, double& d2max, int lane) {
  constexpr uint32_t low = kPlaceMask;
  // the query itself is the smallest: L + 1 words from the bottom
  const uint32_t wl = lth_word(words, n, L + 1, rhof2, lane);
  const float hi = sqrtf(__uint_as_float(wl | low)) * (1.0f + 2.0f * kRel) + E;      // of the L-th distance
  const float lo = sqrtf(__uint_as_float(wl & ~low)) * (1.0f - 2.0f * kRel) - E;
  if (!(hi * 1.000001f <= rho)) return -1;
  const float a = fmaxf((lo - E) * (1.0f - 2.0f * kRel), 0.0f), b = (hi + E) * (1.0f + 2.0f * kRel);
  const uint32_t Tlo = __float_as_uint(a * a * 0.999999f), Thi = __float_as_uint(b * b * 1.000001f);
  int p_lo = 0, nb = 0;
  int br[kBand];
#pragma unroll 2
  for (int e = 0; e < n; ++e) {
    const uint32_t w = words[e * kPad + lane];
    if ((w & ~low) > Thi) continue;
    const int r = rank_of_place(tab, (int)(w & low), r0);
    if (r == self) continue;
    if ((w | low) < Tlo) {
      words[(p_lo++) * kPad + lane] = (uint32_t)r;
    } else {
      if (nb == kBand) return 0;
      br[nb++] = r;
    }
  }
  const int want = L - p_lo;
  if (want < 1 || want > nb) return 0;
  // exact FP64 keys of the band, the `want` smallest by (d^2, caller index), compared as bit
  // patterns (non-negative doubles order like them)
  unsigned long long bd[kBand];
  long long bj[kBand];
#pragma unroll 1
  for (int t = 0; t < nb; ++t)
    bd[t] = (unsigned long long)__double_as_longlong(d2_fp64(A.pos64, br[t], x, y, z, T.box[0], T.box[1], bj[t]));
  unsigned long long kmax = 0;
  int wr = p_lo;
#pragma unroll 1
  for (int t = 0; t < nb; ++t) {
    int rank = 0;
#pragma unroll 1
    for (int u = 0; u < nb; ++u)
      if (bd[u] < bd[t] || (bd[u] == bd[t] && bj[u] < bj[t])) rank++;
    if (rank < want) {
      words[(wr++) * kPad + lane] = (uint32_t)br[t];
      kmax = kmax > bd[t] ? kmax : bd[t];
    }
  }
  d2max = __longlong_as_double((long long)kmax);
  return 1;
}

// Ascending sort of N keys held in registers (bitonic network, fully unrolled).
template <int N>
__device__ __forceinline__ void bitonic(uint32_t (&c)[N]) {
#pragma unroll
  for (int k = 2; k <= N; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
#pragma unroll
      for (int i = 0; i < N; ++i) {
        const int l = i ^ j;
        if (l > i) {
          const uint32_t a = c[i], b = c[l];
          const uint32_t lo = a < b ? a : b, hi = a < b ? b : a;
          if ((i & k) == 0) { c[i] = lo; c[l] = hi; } else { c[i] = hi; c[l] = lo; }
        }
      }
    }
  }
}

// LMAX: K at most.  Shared memory of a warp: the hits (static: places; otherwise CAP words), the
// leaf table, and a scratch that holds the queue and the upper levels' nodes during a walk and
// the sort keys (a word a member; the ranks then) and, for K > 32, their order (bytes) at
// the output.
template <int LMAX, int CAP, bool kStatic> struct KnnShape {
  static constexpr int al(int v) { return (v + 15) / 16 * 16; }
  static constexpr int cap = kStatic ? LMAX + kExtra : CAP;    // hits kept, the query's own among them
  static constexpr int hits = al((cap + kSlack) * (kStatic ? 34 * 2 : kPad * 4));
  static constexpr int queue = al((int)sizeof(Queue));
  static constexpr bool regs = LMAX <= 32;                     // the sort in registers
  // the sort keys: behind the members in the words when there is room
  static constexpr bool behind = !kStatic && CAP >= 2 * (LMAX - 1);
  static constexpr int keys = behind ? 0 : al(LMAX * kPad * 4);
  static constexpr int out = regs ? keys : keys + al(LMAX * kPad);
  static constexpr int walk = queue + 2 * kFront * 4;
  static constexpr int scratch = walk > out ? walk : out;
  static constexpr int bytes = hits + scratch + kSlots * 4;
  static constexpr int wpb = 2 * bytes <= 56 * 1024 ? 2 : 1;   // warps per block
  // blocks an SM's shared memory takes (1 KB of it per block is the system's), for the registers
  static constexpr int fit = 227 * 1024 / (wpb * bytes + 1024);
  static constexpr int blocks = fit < 1 ? 1 : fit * wpb < kMaxWarps ? fit : kMaxWarps / wpb;
};

template <int LMAX, int CAP, bool kStatic>
__global__ void __launch_bounds__(32 * KnnShape<LMAX, CAP, kStatic>::wpb, KnnShape<LMAX, CAP, kStatic>::blocks) k_knn(KnnArgs A) {
  using Sh = KnnShape<LMAX, CAP, kStatic>;
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31;
  unsigned char* mine = smem + (size_t)(threadIdx.x >> 5) * Sh::bytes;
  unsigned short* ids = reinterpret_cast<unsigned short*>(mine);
  uint32_t* words = reinterpret_cast<uint32_t*>(mine);
  unsigned char* scratch = mine + Sh::hits;
  Queue* Q = reinterpret_cast<Queue*>(scratch);
  int* front = reinterpret_cast<int*>(scratch + Sh::queue);
  int* tab = reinterpret_cast<int*>(scratch + Sh::scratch);
  const int L = A.K - 1;
  const int total = A.listed ? (int)*A.leaves_n : A.n_leaves * A.parts;
  // no block-wide barrier below: the warps of a block go their own ways
#pragma unroll 1
  for (int it = blockIdx.x * Sh::wpb + (threadIdx.x >> 5); it < total; it += gridDim.x * Sh::wpb) {
  const int item = A.listed ? A.leaves[it] : it;
  const int leaf = item / A.parts;
  const int b = lev_inst(A.leaf_off, A.n_inst, leaf);
  const TreeDev& T = A.tree[b];
  const InstDev& P = A.P[b];
  const long long r0 = A.off[b];
  const int n = (int)(A.off[b + 1] - r0);
  const int own = leaf - A.leaf_off[b];
  const int il = own * kLeaf + lane;
  const bool have = il < n;
  const long long q = r0 + (have ? il : 0);
  const int4 me = have ? __ldg(A.posq + q) : make_int4(0, 0, 0, -1);
  // this warp's queries: all of the leaf's, or a half or quarter of them
  const bool mine_q = have && (A.parts == 1 || lane / (kLeaf / A.parts) == item % A.parts);
  const bool valid = me.w >= 0;
  const bool per = T.periodic != 0;
  const float half = per ? 0.5f * (float)min(T.boxq[0], T.boxq[1]) : 0.0f;
  bool pend = valid && mine_q && (!A.listed || A.dist[q] < 0.0);
  // ---- first radius
  float rho = 0.0f;
  {
    const double dp = pend && !A.fixed ? A.dprev[me.w] : 0.0;
    float d = (float)(dp * T.inv_q);
    const bool known = dp > 0.0 && dp < 1e300 && d < 1e18f;
    if (!known) d = 0.0f;
    if (kStatic) {
      // a hair over the exact distance: the margins of members_static (E is about 2 units and
      // 1e-6 d) and no more, so that a particle beyond the members is rarely hit
      rho = d * 1.000008f + 8.0f;
      if (!known) { rho = 0.0f; pend = false; }
    } else {
      // moved: over one step most neighbourhoods keep their members nearly, so the last distance
      // and a little is tried first (the counts of a decorrelated neighbourhood scatter by a
      // sixth: half of its queries then walk again, wider)
      rho = known ? kMovedFac * d : 0.0f;
      const bool open = pend && !(rho > 4.0f);
      if (__any_sync(kAll, open)) {
        // unknown: the distance to the eighth nearest of the particles of this leaf and the two
        // beside it on the curve, which hold most of the particles so near, scaled by the
        // wanted count
        float near[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) near[k] = 3e38f;
#pragma unroll 1
        for (int w = -1; w <= 1; ++w) {
          const int iw = il + w * kLeaf;
          int4 c = me;
          if (w != 0) c = iw >= 0 && iw < n ? __ldg(A.posq + r0 + iw) : make_int4(0, 0, 0, -1);
#pragma unroll 1
          for (int src = 0; src < 32; ++src) {
            const int x = __shfl_sync(kAll, c.x, src), y = __shfl_sync(kAll, c.y, src), z = __shfl_sync(kAll, c.z, src);
            const bool there = __shfl_sync(kAll, c.w, src) >= 0 && !(w == 0 && src == lane);
            const float dx = (float)(x - me.x), dy = (float)(y - me.y), dz = (float)(z - me.z);
            float v = there ? dx * dx + dy * dy + dz * dz : 3e38f;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              const float m = fminf(near[k], v);
              v = fmaxf(near[k], v);
              near[k] = m;
            }
          }
        }
        float d2 = 0.0f;
        int m = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k)
          if (near[k] < 3e38f) { d2 = near[k]; m = k + 1; }
        // (its noise and its dependence on the place in the leaf evened out by the leaf's mean)
        const float d8 = sqrtf(d2);
        const int no = __popc(__ballot_sync(kAll, open));
        const float mean = warp_sumf(open ? d8 : 0.0f) / (float)max(no, 1);
        const float r = d8 < 2.0f * mean && mean < 2.0f * d8 ? 0.25f * d8 + 0.75f * mean : d8;
        if (open) rho = fmaxf(r * cbrtf(kLeafShare * (float)(L + CAP) / (float)max(m, 1)), 8.0f);
      }
    }
  }
  // ---- walks
  bool done = false, near_tie = false;
  float r_lo = 0.0f, r_hi = 0.0f;                  // radii known to hold too few / too many
  double X = 0.0, Y = 0.0, Z = 0.0;
  if (have) {
    const double2* pp = reinterpret_cast<const double2*>(A.pos64 + q);
    const double2 a0 = __ldg(pp), a1 = __ldg(pp + 1);
    X = a0.x; Y = a0.y; Z = a1.x;
  }
#pragma unroll 1
  for (int att = 0; att < (kStatic ? 1 : kTries); ++att) {
    // a ball reaching across half a periodic extent meets a particle and its image: exact redo
    if (pend && per && rho * 1.0001f + 64.0f >= half) {
      if (!kStatic && att == 0) rho = 0.98f * half - 128.0f;   // an estimate: try the largest
      if (rho * 1.0001f + 64.0f >= half || !(rho > 0.0f)) pend = false;
    }
    // One walk for all pending queries, or several: a walk visits the particles within the
    // largest radius of the queries' box, so a leaf that straddles a density gradient (a large
    // box or radius beside a small one) is split in halves along the curve until the volume so
    // visited is below kSplit times the smallest ball's.
    int largest = 32;                                // queries of a walk at most
#pragma unroll 1
    for (unsigned todo = __ballot_sync(kAll, pend); todo;) {
      const int first = __ffs(todo) - 1;
      bool act;
      int gx0, gx1, gy0, gy1, gz0, gz1;
      float rmax;
      int size = largest;
#pragma unroll 1
      for (;; size >>= 1) {
        act = ((todo >> lane) & 1u) && (lane & -size) == (first & -size);
        gx0 = __reduce_min_sync(kAll, act ? me.x : INT_MAX);
        gx1 = __reduce_max_sync(kAll, act ? me.x : INT_MIN);
        gy0 = __reduce_min_sync(kAll, act ? me.y : INT_MAX);
        gy1 = __reduce_max_sync(kAll, act ? me.y : INT_MIN);
        gz0 = __reduce_min_sync(kAll, act ? me.z : INT_MAX);
        gz1 = __reduce_max_sync(kAll, act ? me.z : INT_MIN);
        rmax = __uint_as_float(__reduce_max_sync(kAll, __float_as_uint(act ? rho : 0.0f)));
        const float rmin = __uint_as_float(__reduce_min_sync(kAll, __float_as_uint(act ? rho : 3e38f)));
        const float vol = (0.5f * (float)(gx1 - gx0) + rmax) * (0.5f * (float)(gy1 - gy0) + rmax) *
                          (0.5f * (float)(gz1 - gz0) + rmax);
        if (size == 1 || vol <= kSplit * rmin * rmin * rmin) break;
      }
      Walk W;
      const int3 ref = make_int3(gx0 + (gx1 - gx0) / 2, gy0 + (gy1 - gy0) / 2, gz0 + (gz1 - gz0) / 2);
      W.hx = __int2float_ru(gx1 - ref.x);            // the larger half
      W.hy = __int2float_ru(gy1 - ref.y);
      W.hz = __int2float_ru(gz1 - ref.z);
      const float E = error_bound(per, fmaxf(W.hx, fmaxf(W.hy, W.hz)) + rmax);
      const float rf = (rho * (1.0f + 2.0f * kRel) + 2.0f * E) * 1.000001f;
      const float rw = (rmax * (1.0f + 4.0f * kRel) + 4.0f * E) * 1.00001f;
      const float rhof2 = rf * rf * 1.000001f;
      W.rhof2 = act ? rhof2 : -1.0f;
      W.rm2 = rw * rw * 1.00001f;
      W.qx = (float)(me.x - ref.x);
      W.qy = (float)(me.y - ref.y);
      W.qz = (float)(me.z - ref.z);
      constexpr unsigned kStep = kStatic ? 68 : 4 * kPad;
      const unsigned base = kStatic ? shared_addr(ids + lane) : shared_addr(words + lane);
      W.at = base;
      W.past = 0;
      // shifts of the candidates by -1, 0 or 1 periodic extents that can reach the queries
      int ix0 = 0, ix1 = 0, iy0 = 0, iy1 = 0;
      if (per) {
        const int rr = (int)rw + 8;
        if (gx0 - rr < T.maxq[0] - T.boxq[0]) ix0 = -1;
        if (gx1 + rr > T.boxq[0]) ix1 = 1;
        if (gy0 - rr < T.maxq[1] - T.boxq[1]) iy0 = -1;
        if (gy1 + rr > T.boxq[1]) iy1 = 1;
      }
      int cnt = 0;
#pragma unroll 1
      for (int iy = iy0; iy <= iy1 && cnt >= 0; ++iy)
#pragma unroll 1
        for (int ix = ix0; ix <= ix1 && cnt >= 0; ++ix) {
          const int sx = ix * T.boxq[0], sy = iy * T.boxq[1];
          const float g[6] = {__int2float_rd(gx0 - sx), __int2float_rd(gy0 - sy), __int2float_rd(gz0),
                              __int2float_ru(gx1 - sx), __int2float_ru(gy1 - sy), __int2float_ru(gz1)};
          __syncwarp();
          cnt = find_leaves(A, T, g, W.rm2, (iy * 3 + ix + 4) << kShiftBit, tab, cnt, front, lane);
        }
      __syncwarp();
      if (cnt < 0 && size > 1) { largest = size >> 1; continue; }   // its leaves do not fit: fewer queries
      todo &= ~__ballot_sync(kAll, act);
      const bool fits = cnt >= 0;
      if (fits) {
        visit<kStatic>(A, T, Q, tab, cnt, r0, n, ref, per, W, base + Sh::cap * kStep, (kOver - 1) * CAP, lane);
      }
      const int hits = (int)((W.at - base) / kStep + W.past);
      __syncwarp();
      // ---- this walk's queries
      bool ok = false;
      double d2max = 0.0;
      constexpr int kEB = LMAX <= 32 ? 6 : LMAX <= 64 ? 7 : LMAX <= 128 ? 8 : 9;   // hits are below cap
      const bool packed = A.packed != 0;
      // a hit's particle, and its D from the quantised coordinates (static)
      auto rank_at = [&](int e) -> int {
        return kStatic ? rank_of_place(tab, ids[e * 34 + lane], (int)r0) : (int)words[e * kPad + lane];
      };
      auto dist_to = [&](const int4 c) -> float {
        int dx = c.x - me.x, dy = c.y - me.y;
        if (per) {                                   // the hit is the nearest image
          const int bqx = T.boxq[0], bqy = T.boxq[1];
          if (2 * abs(dx) > bqx) dx -= dx > 0 ? bqx : -bqx;
          if (2 * abs(dy) > bqy) dy -= dy > 0 ? bqy : -bqy;
        }
        const float fx = (float)dx, fy = (float)dy, fz = (float)(c.z - me.z);
        return fmaf(fz, fz, fmaf(fy, fy, fx * fx));
      };
      // sort keys; the code of this part is kept small (loops over shared memory), since what does
      // not fit the instruction cache costs more than the loads
      uint32_t* keys = Sh::behind ? words + L * kPad : reinterpret_cast<uint32_t*>(scratch);
      const int ne = kStatic ? A.K : L;              // entries to sort (static: the query's own too)
      if (kStatic) {
        // the members' sort keys and their two largest D, from the particles themselves (the
        // coordinates and the caller index come in one load)
        if (act && hits == A.K) {
          float m0 = -1.0f, m1 = -1.0f;
          int e0 = 0;
          auto key_of = [&](int e) -> uint32_t {
            const int4 c = __ldg(A.posq + rank_at(e));
            const float D = dist_to(c);
            m1 = fmaxf(m1, fminf(m0, D));
            if (D > m0) { m0 = D; e0 = e; }
            if (c.w == me.w) return 0xFFFFFFFFu;     // the query itself: past the members
            return packed ? ((uint32_t)c.w << kEB) | (uint32_t)e : (uint32_t)c.w;
          };
#pragma unroll 4
          for (int e = 0; e < A.K; ++e) keys[e * kPad + lane] = key_of(e);
          const Margins g = margins(m0, rho, E);
          ok = g.inside && m1 < g.lo;
          if (ok) {
            long long j;
            d2max = d2_fp64(A.pos64, rank_at(e0), X, Y, Z, T.box[0], T.box[1], j);
          }
        }
        if (act && !ok && hits >= A.K && hits < A.K + kExtra) {
          // a few hits too many, or the largest too near one another (a query in a few
          // hundred): the largest in order give the K-1-th, and its band is ranked in FP64
          float m[kExtra + 1];
#pragma unroll
          for (int k = 0; k <= kExtra; ++k) m[k] = -1.0f;
#pragma unroll 1
          for (int e = 0; e < hits; ++e) {
            float v = dist_to(__ldg(A.posq + rank_at(e)));
#pragma unroll
            for (int k = 0; k <= kExtra; ++k) { const float u = fmaxf(m[k], v); v = fminf(m[k], v); m[k] = u; }
          }
          float dk = m[0];
#pragma unroll
          for (int k = 1; k < kExtra; ++k)
            if (k == hits - A.K) dk = m[k];
          const Margins g = margins(dk, rho, E);
          if (g.inside) {
            int w = 0, nb = 0;                       // certain entries (the query's own too), band
            int br[kBand];
            bool over = false;
#pragma unroll 1
            for (int e = 0; e < hits; ++e) {
              const unsigned short place = ids[e * 34 + lane];
              const float D = dist_to(__ldg(A.posq + rank_of_place(tab, place, (int)r0)));
              if (D < g.lo) {
                ids[(w++) * 34 + lane] = place;
              } else if (D <= g.hi) {
                if (nb < kBand) br[nb++] = place; else over = true;
              }
            }
            const int want = A.K - w;
            if (!over && want >= 1 && want <= nb) {
              unsigned long long bd[kBand], kmax = 0;
              long long bj[kBand];
#pragma unroll 1
              for (int k = 0; k < nb; ++k)
                bd[k] = (unsigned long long)__double_as_longlong(
                    d2_fp64(A.pos64, rank_of_place(tab, br[k], (int)r0), X, Y, Z, T.box[0], T.box[1], bj[k]));
#pragma unroll 1
              for (int k = 0; k < nb; ++k) {
                int rank = 0;
#pragma unroll 1
                for (int u = 0; u < nb; ++u)
                  if (bd[u] < bd[k] || (bd[u] == bd[k] && bj[u] < bj[k])) rank++;
                if (rank < want) {
                  ids[(w++) * 34 + lane] = (unsigned short)br[k];
                  kmax = kmax > bd[k] ? kmax : bd[k];
                }
              }
              d2max = __longlong_as_double((long long)kmax);
              ok = true;
#pragma unroll 1
              for (int e = 0; e < A.K; ++e) {
                const uint32_t c = (uint32_t)__ldg(&A.posq[rank_at(e)].w);
                keys[e * kPad + lane] = c == (uint32_t)me.w ? 0xFFFFFFFFu : packed ? (c << kEB) | (uint32_t)e : c;
              }
            }
          }
        }
        if (act && !ok) {
          pend = false;
          if (!fits) near_tie = true;
          // ties within the error bounds go straight to the exact search
          if (hits >= A.K && hits < A.K + kExtra) near_tie = true;
        }
      } else if (act) {
        if (!fits) {
          pend = false;                              // the walk's leaves do not fit: exact search
        } else if (hits <= L) {
          r_lo = rho;
          rho = r_hi > 0.0f ? sqrtf(r_lo * r_hi) : grow(rho, hits, L, CAP);
        } else if (hits > CAP) {
          r_hi = rho;
          rho = r_lo > 0.0f ? sqrtf(r_lo * r_hi)
                            : rho * (hits > kOver * CAP ? 0.5f : cbrtf(0.5f * (float)(L + CAP) / (float)hits));
        } else {
          const int got = members(A, T, words, tab, (int)r0, (int)q, hits, L, rho, E, rhof2, X, Y, Z,
                                            d2max, lane);
          ok = got > 0;
          if (got < 0) { r_lo = rho; rho *= 1.05f; r_hi = 0.0f; }
          if (got == 0) pend = false;
        }
      }
      if (ok) { pend = false; done = true; }
      const unsigned okm = __ballot_sync(kAll, ok);
      if (okm) {
        // the members in ascending caller index: sort keys are the caller index with, when the
        // indices leave room, the member's entry in the low bits
        auto sort_key = [&](int e) -> uint32_t {
          const uint32_t c = (uint32_t)__ldg(&A.posq[rank_at(e)].w);
          return packed ? (c << kEB) | (uint32_t)e : c;
        };
        auto rank_of_key = [&](uint32_t k) -> int {
          return packed ? rank_at((int)(k & ((1u << kEB) - 1u))) : __ldg(&A.rank_of[k]);
        };
        int* rows = A.nbr + (r0 + (long long)own * kLeaf) * A.K;      // the leaf's first row
        if constexpr (Sh::regs) {
          // Sorted in registers; the ranks then go through shared memory and out row by row: a
          // row is one 128-byte store for K = 32, where each lane storing its own row touched
          // 32 sectors per element.
          uint32_t* out = keys;
          if (ok) {
            if (!kStatic) {
#pragma unroll 4
              for (int e = 0; e < L; ++e) keys[e * kPad + lane] = sort_key(e);
            }
            uint32_t cs[32];
#pragma unroll
            for (int e = 0; e < 32; ++e) cs[e] = e < ne ? keys[e * kPad + lane] : 0xFFFFFFFFu;
            bitonic<32>(cs);
#pragma unroll
            for (int e = 0; e < 32 - 1; ++e)
              if (e < L) keys[e * kPad + lane] = cs[e];
#pragma unroll 4
            for (int e = 0; e < L; ++e) {
              const uint32_t k = keys[e * kPad + lane];
              out[e * kPad + lane] = A.fixed ? (packed ? k >> kEB : k) : (uint32_t)rank_of_key(k);
            }
          }
          __syncwarp();
#pragma unroll 1
          for (unsigned m = okm; m; m &= m - 1u) {
            const int l = __ffs(m) - 1;
            const int wl = __shfl_sync(kAll, me.w, l);
            int* row = A.fixed ? A.nbr + (long long)wl * A.K : rows + l * A.K;
            const int first = A.fixed ? wl : (int)(r0 + own * kLeaf + l);
            for (int k = lane; k < A.K; k += 32) row[k] = k == 0 ? first : (int)out[(k - 1) * kPad + l];
          }
          __syncwarp();
        } else {
          // runs of 32 sort keys ordered in registers, then merged: the order of the entries
          // (packed) or the caller indices themselves
          unsigned char* order = scratch + Sh::keys;
          constexpr int NR = (LMAX + 31) / 32;
          if (ok) {
#pragma unroll 1
            for (int h = 0; h < NR && 32 * h < ne; ++h) {
              uint32_t run[32];
#pragma unroll
              for (int e = 0; e < 32; ++e) {
                const int i = 32 * h + e;
                run[e] = i < ne ? (kStatic ? keys[i * kPad + lane] : sort_key(i)) : 0xFFFFFFFFu;
              }
              bitonic<32>(run);
#pragma unroll
              for (int e = 0; e < 32; ++e)
                if (32 * h + e < ne) keys[(32 * h + e) * kPad + lane] = run[e];
            }
            uint32_t hd[NR];      // each run's next key (0xFFFFFFFF when it is used up)
            int ps[NR];
#pragma unroll
            for (int c = 0; c < NR; ++c) {
              ps[c] = 32 * c;
              hd[c] = ps[c] < ne ? keys[ps[c] * kPad + lane] : 0xFFFFFFFFu;
            }
#pragma unroll 1
            for (int k = 0; k < L; ++k) {
              uint32_t key = hd[0];
              int bi = 0;
#pragma unroll
              for (int c = 1; c < NR; ++c)
                if (hd[c] < key) { key = hd[c]; bi = c; }
#pragma unroll
              for (int c = 0; c < NR; ++c) {
                if (c == bi) {
                  ++ps[c];
                  const int end = 32 * c + 32 < ne ? 32 * c + 32 : ne;
                  hd[c] = ps[c] < end ? keys[ps[c] * kPad + lane] : 0xFFFFFFFFu;
                }
              }
              if (packed) order[k * kPad + lane] = (unsigned char)(key & ((1u << kEB) - 1u));
              else rows[(long long)lane * A.K + 1 + k] = __ldg(&A.rank_of[key]);
            }
            if (!packed) rows[(long long)lane * A.K] = (int)q;
          }
          __syncwarp();
          if (packed)
#pragma unroll 1
            for (unsigned m = okm; m; m &= m - 1u) {
              const int l = __ffs(m) - 1;
              const int wl = __shfl_sync(kAll, me.w, l);
              int* row = A.fixed ? A.nbr + (long long)wl * A.K : rows + (long long)l * A.K;
              for (int k = lane; k < A.K; k += 32) {
                int r = (int)(r0 + own * kLeaf + l);
                if (k > 0) {
                  const int e = order[(k - 1) * kPad + l];
                  r = kStatic ? rank_of_place(tab, ids[e * 34 + l], (int)r0) : (int)words[e * kPad + l];
                }
                row[k] = A.fixed ? __ldg(&A.posq[r].w) : r;
              }
            }
          __syncwarp();
        }
        if (ok) put_result(A, P, q, me.w, d2max, X, Y);
      }
    }
    if (!__any_sync(kAll, pend)) break;
  }
  // ---- undecided queries
  if (kStatic) {
    // ties and stragglers to the exact search; a leaf with many undecided queries (the caller
    // moved the particles, or there is no earlier build) to the general kernel
    bool left = valid && mine_q && !done && !near_tie;
    const bool few = __popc(__ballot_sync(kAll, left)) * A.parts <= 8;
    if (near_tie || (left && few)) A.redo[atomicAdd(A.redo_n, 1ull)] = (int)q;
    left = left && !few;
    if (left) A.dist[q] = -1.0;
    if (__any_sync(kAll, left) && lane == 0) A.leaves[atomicAdd(A.leaves_n, 1ull)] = item;
  } else if (valid && mine_q && !done && (!A.listed || A.dist[q] < 0.0)) {
    A.redo[atomicAdd(A.redo_n, 1ull)] = (int)q;
  }
  if (mine_q && !valid && !A.listed) {
    // a coordinate that is not finite
    no_list(A, P, q, ~me.w);
  }
  }
}

// ---------------------------------------------------------------- exact queries
// The list across a warp: entry t * 32 + lane in ascending (key, caller index).
template <int KPL>
struct WarpList {
  unsigned long long k[KPL];      // bits of d^2
  int j[KPL], r[KPL];             // caller index and rank
};

// Inserts one entry (the same in every lane) that is smaller than the list's last.
template <int KPL>
__device__ __forceinline__ void insert(WarpList<KPL>& S, unsigned long long nk, int nj, int nr, int lane) {
  int pos = 0;
#pragma unroll
  for (int t = 0; t < KPL; ++t) pos += __popc(__ballot_sync(kAll, S.k[t] < nk || (S.k[t] == nk && S.j[t] < nj)));
#pragma unroll
  for (int t = KPL - 1; t >= 0; --t) {
    unsigned long long uk = __shfl_up_sync(kAll, S.k[t], 1);
    int uj = __shfl_up_sync(kAll, S.j[t], 1), ur = __shfl_up_sync(kAll, S.r[t], 1);
    const int tp = t > 0 ? t - 1 : 0;
    const unsigned long long ck = __shfl_sync(kAll, S.k[tp], 31);
    const int cj = __shfl_sync(kAll, S.j[tp], 31), cr = __shfl_sync(kAll, S.r[tp], 31);
    if (lane == 0 && t > 0) { uk = ck; uj = cj; ur = cr; }
    const int at = t * 32 + lane;
    if (at > pos) { S.k[t] = uk; S.j[t] = uj; S.r[t] = ur; }
    else if (at == pos) { S.k[t] = nk; S.j[t] = nj; S.r[t] = nr; }
  }
}

// Ascending sort of 32 KPL keys, entry t * 32 + lane (bitonic).
template <int KPL>
__device__ __forceinline__ void warp_sort(unsigned long long (&v)[KPL], int lane) {
  for (int k = 2; k <= 32 * KPL; k <<= 1)
    for (int s = k >> 1; s > 0; s >>= 1) {
      if (s >= 32) {
#pragma unroll
        for (int t = 0; t < KPL; ++t) {
#pragma unroll
          for (int u = t + 1; u < KPL; ++u) {
            if ((t ^ u) != (s >> 5)) continue;
            const bool up = ((t * 32 + lane) & k) == 0;
            if (up ? v[t] > v[u] : v[t] < v[u]) { const unsigned long long a = v[t]; v[t] = v[u]; v[u] = a; }
          }
        }
      } else {
#pragma unroll
        for (int t = 0; t < KPL; ++t) {
          const unsigned long long o = __shfl_xor_sync(kAll, v[t], s);
          const bool up = ((t * 32 + lane) & k) == 0, low = (lane & s) == 0;
          if (low == up ? o < v[t] : o > v[t]) v[t] = o;
        }
      }
    }
}

template <int KPL>
__global__ void __launch_bounds__(128) k_knn_exact(KnnArgs A) {
  __shared__ int stacks[4][2 * kMaxLev];
  const int lane = threadIdx.x & 31;
  int* stack = stacks[threadIdx.x >> 5];
  const int L = A.K - 1;
  const long long total = (long long)*A.redo_n;
  const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long t = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < total; t += nw) {
    const int q = A.redo[t];
    const int b = inst_of(A.off, A.n_inst, q);
    const TreeDev& T = A.tree[b];
    const InstDev& P = A.P[b];
    const long long r0 = A.off[b];
    const int n = (int)(A.off[b + 1] - r0);
    const int4 me = __ldg(A.posq + q);
    const Pos64 c = A.pos64[q];
    const double bx = T.box[0], by = T.box[1];
    WarpList<KPL> S;
#pragma unroll
    for (int u = 0; u < KPL; ++u) { S.k[u] = ~0ull; S.j[u] = INT_MAX; S.r[u] = q; }
    unsigned long long wk = ~0ull;                 // the (K-1)-th entry so far
    int wj = INT_MAX;
    float rm2 = __int_as_float(0x7F800000);
    auto leaf_in = [&](int leaf) {
      const int i = leaf * kLeaf + lane;
      unsigned long long ck = ~0ull;
      int cj = INT_MAX, cr = -1;
      if (i < n && r0 + i != q) {
        const int w = __ldg(&A.posq[r0 + i].w);
        if (w >= 0) {
          long long jj;
          ck = (unsigned long long)__double_as_longlong(d2_fp64(A.pos64, (int)(r0 + i), c.x, c.y, c.z, bx, by, jj));
          cj = w;
          cr = (int)(r0 + i);
        }
      }
      unsigned m = __ballot_sync(kAll, ck < wk || (ck == wk && cj < wj));
      if (!m) return;
      while (m) {
        const int src = __ffs(m) - 1;
        m &= m - 1u;
        const unsigned long long nk = __shfl_sync(kAll, ck, src);
        const int nj = __shfl_sync(kAll, cj, src), nr = __shfl_sync(kAll, cr, src);
        if (!(nk < wk || (nk == wk && nj < wj))) continue;
        insert<KPL>(S, nk, nj, nr, lane);
        unsigned long long kv = S.k[0];
        int jv = S.j[0];
#pragma unroll
        for (int u = 1; u < KPL; ++u)
          if (u == ((L - 1) >> 5)) { kv = S.k[u]; jv = S.j[u]; }
        wk = __shfl_sync(kAll, kv, (L - 1) & 31);
        wj = __shfl_sync(kAll, jv, (L - 1) & 31);
      }
      if (wk != ~0ull) {
        // in units, with room for the truncation of both positions and the box's rounding
        const float u = __double2float_ru(sqrt(__longlong_as_double((long long)wk)) * T.inv_q) * 1.00001f + 8.0f;
        rm2 = u * u * 1.00001f;
      }
    };
    // the leaves around the query on the curve first: they bound the rest
    const int own = (int)(q - r0) / kLeaf, e = (L + 31) / 64 + 1, last = T.lev_n[0] - 1;
    const int la = max(0, own - e), lb = min(last, own + e);
    for (int leaf = la; leaf <= lb; ++leaf) leaf_in(leaf);
    const float qxl = __int2float_rd(me.x), qxh = __int2float_ru(me.x), qyl = __int2float_rd(me.y),
                qyh = __int2float_ru(me.y), qzl = __int2float_rd(me.z), qzh = __int2float_ru(me.z);
    const float pbx = (float)T.boxq[0], pby = (float)T.boxq[1];
    auto children = [&](int l, int first) -> unsigned {
      const int k = first + lane;
      bool hit = false;
      if (k < T.lev_n[l]) {
        const float4 a = __ldg(A.na + T.lev_off[l] + k);
        const float2 d = __ldg(A.nb + T.lev_off[l] + k);
        float gx = gap(a.x, a.w, qxl, qxh), gy = gap(a.y, d.x, qyl, qyh);
        const float gz = gap(a.z, d.y, qzl, qzh);
        if (T.periodic) {
          gx = fminf(gx, fminf(gap(a.x, a.w, qxl - pbx, qxh - pbx), gap(a.x, a.w, qxl + pbx, qxh + pbx)));
          gy = fminf(gy, fminf(gap(a.y, d.x, qyl - pby, qyh - pby), gap(a.y, d.x, qyl + pby, qyh + pby)));
          gx = fmaxf(gx - 256.0f, 0.0f);           // the extents' rounding
          gy = fmaxf(gy - 256.0f, 0.0f);
        }
        hit = gx * gx + gy * gy + gz * gz <= rm2;
      }
      return __ballot_sync(kAll, hit);
    };
    const int top = T.nlev - 1;
    int l = top, first = 0;
    unsigned m = children(l, 0);
    for (;;) {
      while (m == 0 && l < top) {
        ++l;
        m = (unsigned)stack[2 * l];
        first = stack[2 * l + 1];
      }
      if (m == 0) break;
      const int k = first + __ffs(m) - 1;
      m &= m - 1u;
      if (l == 0) {
        if (k < la || k > lb) leaf_in(k);
      } else {
        __syncwarp();
        if (lane == 0) { stack[2 * l] = (int)m; stack[2 * l + 1] = first; }
        __syncwarp();
        --l;
        first = k * kLeaf;
        m = children(l, first);
      }
    }
    if (wk != ~0ull) {
      int* row = A.nbr + (A.fixed ? me.w : q) * (long long)A.K;
      unsigned long long v[KPL];
#pragma unroll
      for (int u = 0; u < KPL; ++u)
        v[u] = u * 32 + lane < L ? ((unsigned long long)(unsigned)S.j[u] << 32) | (unsigned)S.r[u] : ~0ull;
      warp_sort<KPL>(v, lane);
#pragma unroll
      for (int u = 0; u < KPL; ++u)
        if (u * 32 + lane < L) row[1 + u * 32 + lane] = A.fixed ? (int)(v[u] >> 32) : (int)(unsigned)v[u];
      if (lane == 0) {
        row[0] = A.fixed ? me.w : q;
        put_result(A, P, q, me.w, __longlong_as_double((long long)wk), c.x, c.y);
        if (A.pref32) atomicAdd((unsigned long long*)&A.st[P.unit0].knn_redo, 1ull);
      }
    } else if (lane == 0) {
      no_list(A, P, q, me.w);
    }
  }
}

// ---------------------------------------------------------------- launchers
template <int LMAX, int CAP, bool kStatic>
static cudaError_t launch_knn_t(gd_ctx* c, KnnArgs& A) {
  using Sh = KnnShape<LMAX, CAP, kStatic>;
  constexpr int kEB = LMAX <= 32 ? 6 : LMAX <= 64 ? 7 : LMAX <= 128 ? 8 : 9;
  A.packed = A.N <= (1LL << (32 - kEB)) ? 1 : 0;
  // few leaves: their queries over more warps (a warp's time is a long chain of dependent steps;
  // a quarter of the queries has a smaller box, fewer candidates and shorter loops)
  A.parts = 1;
  while (A.parts < 4 && A.n_leaves * A.parts * 2LL <= 32LL * c->num_sms) A.parts *= 2;
  int blocks = (int)((A.n_leaves * (long long)A.parts + Sh::wpb - 1) / Sh::wpb);
  if (A.listed) blocks = blocks < 8 * c->num_sms ? blocks : 8 * c->num_sms;
  k_knn<LMAX, CAP, kStatic><<<blocks, 32 * Sh::wpb, Sh::wpb * Sh::bytes, c->stream>>>(A);
  return cudaGetLastError();
}

template <int LMAX, int CAP>
static cudaError_t prepare_t() {
  cudaError_t e = cudaFuncSetAttribute(k_knn<LMAX, CAP, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       KnnShape<LMAX, CAP, true>::wpb * KnnShape<LMAX, CAP, true>::bytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_knn<LMAX, CAP, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             KnnShape<LMAX, CAP, false>::wpb * KnnShape<LMAX, CAP, false>::bytes);
  return e;
}

// Shared-memory opt-in of the neighbour kernels this context launches (once, before any launch
// or graph capture).
cudaError_t knn_prepare(gd_ctx* c) {
  if (c->K <= 32) return prepare_t<32, 96>();
  if (c->K <= 48) return prepare_t<48, 104>();
  if (c->K <= 64) return prepare_t<64, 112>();
  if (c->K <= 128) return prepare_t<128, 208>();
  return prepare_t<256, 320>();
}

template <bool kStatic>
static cudaError_t launch_k(gd_ctx* c, KnnArgs& A) {
  if (A.K <= 32) return launch_knn_t<32, 96, kStatic>(c, A);
  if (A.K <= 48) return launch_knn_t<48, 104, kStatic>(c, A);
  if (A.K <= 64) return launch_knn_t<64, 112, kStatic>(c, A);
  if (A.K <= 128) return launch_knn_t<128, 208, kStatic>(c, A);
  return launch_knn_t<256, 320, kStatic>(c, A);
}

cudaError_t launch_knn(gd_ctx* c) {
  KnnArgs A;
  A.N = c->N;
  A.K = c->K;
  A.n_inst = c->n_inst;
  A.n_leaves = c->n_leaves;
  A.off = c->d_off;
  A.leaf_off = c->d_lev;
  A.P = c->d_inst;
  A.tree = c->d_tree;
  A.na = c->d_node_a;
  A.nb = c->d_node_b;
  A.posq = c->d_posq;
  A.pos64 = c->d_pos64;
  A.rank_of = c->d_rank_of;
  A.fixed = c->lists_only ? 1 : 0;
  A.nbr = c->lists_only ? c->fix_nbr : c->d_nbr;
  A.dist = c->lists_only ? c->fix_d : c->d_dist;
  A.V = c->d_V;
  A.pref32 = c->d_pref32;
  A.dprev = c->d_dprev;
  A.st = c->d_state;
  A.leaves = c->d_heavy;          // free until the sampler
  A.leaves_n = c->d_counters + 2;
  A.redo = c->d_redo;
  A.redo_n = c->d_counters + 1;
  A.listed = 0;
  A.parts = 1;
  A.packed = 0;
  const bool moved = c->moved;
  c->moved = false;
  time_begin(c, 1);
  cudaError_t e = cudaMemsetAsync(c->d_counters + 1, 0, 2 * sizeof(unsigned long long), c->stream);
  if (e == cudaSuccess && !moved) {
    e = launch_k<true>(c, A);
    A.listed = 1;
    c->launches += 1;
  }
  if (e == cudaSuccess) e = launch_k<false>(c, A);
  if (e == cudaSuccess) {
    const int blocks = c->num_sms * 4, L = A.K - 1;
    if (L <= 32) k_knn_exact<1><<<blocks, 128, 0, c->stream>>>(A);
    else if (L <= 64) k_knn_exact<2><<<blocks, 128, 0, c->stream>>>(A);
    else if (L <= 128) k_knn_exact<4><<<blocks, 128, 0, c->stream>>>(A);
    else k_knn_exact<8><<<blocks, 128, 0, c->stream>>>(A);
    e = cudaGetLastError();
  }
  c->launches += 2;
  time_end(c);
  return e;
}

}  // namespace gd
