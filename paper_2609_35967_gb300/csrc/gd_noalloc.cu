// gd_noalloc.cu -- gd_neighbors_fixed: the neighbour search of one instance with its
// scratch in a fixed device array, for callers that cannot allocate device memory.
//
// Some callers cannot call cudaMalloc: a host program that has already reserved the
// device's memory for its own pool (a new allocation would fail or fragment it), or a
// latency-bound loop that cannot afford cudaMalloc's implicit device synchronisation.
// This entry point allocates nothing, on the device or the host.  Its scratch (the order, the tree and the
// positions along it) lives in one file-scope __device__ array of GD_FIXED_SCRATCH_BYTES
// bytes, which every GPU that loads the library holds until the process exits.
// The search is the library's own (k_tree.cu, k_knn.cu) on pointers into that array: a warp per
// query over cell rows, which it replaces, took 3.6 ms for 50,001 particles and K = 32, this
// 1.1 ms (0.9 in the search, whose radius starts from an estimate in every call).
//
// The result is the same as gd_build_neighbors' nbr_out / d_out for a one-instance
// FP64 context: slot 0 the particle itself, then the K-1 nearest others by (d^2, index)
// in ascending index order; d = distance to the farthest of them.
#include <algorithm>
#include <climits>
#include <cmath>
#include <mutex>

#include "gd_ctx.h"

namespace gdfix {

using gd::kLeaf;
using gd::kMaxLev;

constexpr long long kMaxN = GD_FIXED_MAX_PARTICLES;
constexpr int kMaxK = GD_FIXED_MAX_K;

constexpr size_t a256(size_t v) { return (v + 255) / 256 * 256; }
constexpr int kSTile = 2048;                                  // particles per sort tile (k_tree.cu)
constexpr int kTilesMax = (int)(kMaxN / kSTile);
constexpr int kNodesMax = (int)(kMaxN / kLeaf + kMaxN / (kLeaf * kLeaf) + 2 + kMaxLev);

// What a call sets up on the device: the tables of one instance.
struct Tables {
  gd::InstDev inst;
  gd::StateDev state;
  gd::TreeDev tree;
  long long off[2], stile_off[2];
  int lev[2 * kMaxLev];
};

constexpr size_t kOffTables = 0;
constexpr size_t kOffCounters = a256(sizeof(Tables));
constexpr size_t kOffChunk = kOffCounters + a256(16 * sizeof(unsigned long long));
constexpr size_t kOffDigits = kOffChunk + a256(sizeof(int) * 4 * (kTilesMax / 8 + 1));
constexpr size_t kOffNodeA = kOffDigits + a256(sizeof(int) * 256 * kTilesMax);
constexpr size_t kOffNodeB = kOffNodeA + a256(sizeof(float4) * kNodesMax);
constexpr size_t kOffKv = kOffNodeB + a256(sizeof(float2) * kNodesMax);        // two buffers; the
constexpr size_t kOffPosq = kOffKv + a256(2 * sizeof(uint2) * kMaxN);           // order and the redo
constexpr size_t kOffPos64 = kOffPosq + a256(sizeof(int4) * kMaxN);             // list reuse them
constexpr size_t kBytes = kOffPos64 + a256(sizeof(gd::Pos64) * kMaxN);
static_assert(kBytes <= GD_FIXED_SCRATCH_BYTES, "the layout must fit GD_FIXED_SCRATCH_BYTES");

// The fixed scratch.  Host code must not use this name as an address: it is a host-side
// stand-in.  The device address comes from cudaGetSymbolAddress (see scratch_address).
static __device__ __align__(256) unsigned char g_scratch[GD_FIXED_SCRATCH_BYTES];

__global__ void fk_setup(Tables* to, const __grid_constant__ Tables from) { *to = from; }

// Device address of the fixed array, looked up once per device (with that device current)
// and kept for the life of the process: a cudaDeviceReset, which replaces the device's
// primary context, leaves the kept address stale, so the library is not used across one.
static std::mutex g_mu;
static void* g_addr[256];
static int g_sms[256];

static gd_status scratch_address(unsigned char** out, int* sms) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 256) return GD_ERR_CUDA;
  std::lock_guard<std::mutex> lk(g_mu);
  if (!g_addr[dev]) {
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_scratch) != cudaSuccess || !ptr) return GD_ERR_CUDA;
    if (cudaDeviceGetAttribute(&g_sms[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return GD_ERR_CUDA;
    for (int K : {32, 48, 64}) {                     // the search kernels' shared memory, once
      gd_ctx c;
      c.K = K;
      if (gd::knn_prepare(&c) != cudaSuccess) return GD_ERR_CUDA;
    }
    g_addr[dev] = ptr;
  }
  *out = static_cast<unsigned char*>(g_addr[dev]);
  *sms = g_sms[dev];
  return GD_OK;
}

}  // namespace gdfix

extern "C" gd_status gd_neighbors_fixed(const double* x, const double* y, const double* z, int64_t n,
                                        int32_t K, const gd_instance_params* params, int32_t* nbr_out,
                                        double* d_out, void* stream) {
  using namespace gdfix;
  if (!x || !y || !z || !params || !nbr_out) return GD_ERR_ARG;
  if (K < 2 || K > kMaxK || n < K) return GD_ERR_ARG;
  if (n > kMaxN) return GD_ERR_CAPACITY;
  if (params->geometry != GD_GEOM_PATCH && params->geometry != GD_GEOM_DISK) return GD_ERR_ARG;
  if (params->geometry == GD_GEOM_PATCH && !(params->box_x > 0.0 && params->box_y > 0.0)) return GD_ERR_ARG;
  if (params->model != GD_MODEL_3D) return GD_ERR_ARG;   // 3D positions only
  unsigned char* base = nullptr;
  int sms = 0;
  const gd_status st = scratch_address(&base, &sms);
  if (st != GD_OK) return st;
  // a context of one FP64 instance over the scratch, for the launchers alone
  gd_ctx c;
  c.n_inst = 1;
  c.K = K;
  c.precision = GD_FP64;
  c.N = n;
  c.stream = static_cast<cudaStream_t>(stream);
  c.num_sms = sms;
  c.x = const_cast<double*>(x);
  c.y = const_cast<double*>(y);
  c.z = const_cast<double*>(z);
  c.lists_only = true;
  c.fix_nbr = nbr_out;
  c.fix_d = d_out;
  Tables T = {};
  T.off[1] = n;
  gd::tree_plan(&c, T.off, T.lev, T.stile_off);
  T.inst.geometry = params->geometry;
  T.inst.model = GD_MODEL_3D;
  T.inst.kernel_mode = GD_KERNEL_PHYSICAL;
  T.inst.box_x = params->box_x;
  T.inst.box_y = params->box_y;
  T.inst.n = n;
  T.inst.n_sg = 1;
  for (int a = 0; a < 3; ++a) { T.state.bmin[a] = ~0ull; T.state.bmax[a] = 0ull; }
  for (int l = 0; l < c.max_lev; ++l) {
    T.tree.lev_off[l] = T.lev[2 * l];
    T.tree.lev_n[l] = T.lev[2 * l + 1] - T.lev[2 * l];
    if (T.tree.lev_n[l] > 0) T.tree.nlev = l + 1;
  }
  Tables* dT = reinterpret_cast<Tables*>(base + kOffTables);
  c.d_inst = &dT->inst;
  c.d_state = &dT->state;
  c.d_tree = &dT->tree;
  c.d_off = dT->off;
  c.d_stile_off = dT->stile_off;
  c.d_lev = dT->lev;
  c.d_counters = reinterpret_cast<unsigned long long*>(base + kOffCounters);
  c.d_chunk = reinterpret_cast<int*>(base + kOffChunk);
  c.d_digits = reinterpret_cast<int*>(base + kOffDigits);
  c.d_node_a = reinterpret_cast<float4*>(base + kOffNodeA);
  c.d_node_b = reinterpret_cast<float2*>(base + kOffNodeB);
  c.d_kv[0] = reinterpret_cast<uint2*>(base + kOffKv);
  c.d_kv[1] = c.d_kv[0] + kMaxN;
  // three passes: the last reads kv[0] and writes the order, which takes kv[1]'s place; the
  // redo list takes kv[0]'s after it
  c.d_perm = reinterpret_cast<int*>(c.d_kv[1]);
  c.d_redo = reinterpret_cast<int*>(c.d_kv[0]);
  c.d_posq = reinterpret_cast<int4*>(base + kOffPosq);
  c.d_pos64 = reinterpret_cast<gd::Pos64*>(base + kOffPos64);
  fk_setup<<<1, 1, 0, c.stream>>>(dT, T);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = gd::launch_tree(&c);
  if (e == cudaSuccess) e = gd::launch_knn(&c);
  return e == cudaSuccess ? GD_OK : GD_ERR_CUDA;
}
