// upload.cu -- a mesh handle's device arrays from the caller's: validation,
// node_map offsets and the element lists per type (the element loop of Alg.
// "sequential assembly" runs them type by type), all on the device.
//
// The element arrays used to come back to the host, where loops checked them
// and built the per-type lists.  Three kernels do that now: a check that also
// counts each type per tile of elements, a scan of the counts (type-major, so
// that an element's position among all elements of its type is one offset plus
// its rank in the tile), and a pass that writes the lists.  The counts of the
// types before an element give its node_map offset too.  Two allocations hold
// every array of the handle (cudaMalloc and cudaFree cost more than the kernels
// on small meshes): one sized by nodes and elements, and one, sized by the
// check, for the connectivity and, with several types, their lists.  Upload and
// pattern of 412,500 mixed elements from device arrays, one GB300: 18.1 -> 1.44
// ms (with the row builder of pattern.cu).
#include <algorithm>
#include <cstring>
#include <string>

#include "fea_internal.cuh"

namespace fea {

constexpr int kUpThreads = 256;
constexpr int kUpRounds = 4;
constexpr int kUpTile = kUpThreads * kUpRounds;  // elements per tile

struct UploadInfo {
  unsigned long long bad_elem;  // smallest 2 e + (0: unknown type, 1: wrong node count), or ~0
  unsigned long long bad_conn;  // smallest t with conn[t] out of range, or ~0
  int64_t off0, len;            // conn_offsets[0], conn_offsets[E]
  unsigned types;               // bit t: elements of type t
  int64_t base[kNumTypes + 1];  // elements of the types before t
};

__device__ __forceinline__ int up_nodes(int t) { return t < 3 ? t + 4 : 8; }
static_assert(kNodesOf[0] == 4 && kNodesOf[1] == 5 && kNodesOf[2] == 6 && kNodesOf[3] == 8, "node counts per type");

// per tile: elements of each type (tile_cnt[t * tiles + tile]); invalid elements
__global__ void __launch_bounds__(kUpThreads) k_upload_count(const uint8_t* types, const int64_t* off, int64_t E,
                                                             int64_t* tile_cnt, UploadInfo* info) {
  __shared__ int cnt[kNumTypes];
  if (threadIdx.x < kNumTypes) cnt[threadIdx.x] = 0;
  __syncthreads();
  for (int r = 0; r < kUpRounds; ++r) {
    const int64_t e = (int64_t)blockIdx.x * kUpTile + r * kUpThreads + threadIdx.x;
    int t = -1;
    if (e < E) {
      t = types[e];
      const unsigned long long id = 2ull * (unsigned long long)e;
      if (t >= kNumTypes) {
        atomicMin(&info->bad_elem, id);
        t = -1;
      } else if (off[e + 1] - off[e] != up_nodes(t)) {
        atomicMin(&info->bad_elem, id + 1);
      }
    }
#pragma unroll
    for (int k = 0; k < kNumTypes; ++k) {
      const unsigned m = __ballot_sync(0xffffffffu, t == k);
      if ((threadIdx.x & 31) == 0 && m) atomicAdd(&cnt[k], __popc(m));
    }
  }
  __syncthreads();
  if (threadIdx.x < kNumTypes) {
    tile_cnt[(int64_t)threadIdx.x * gridDim.x + blockIdx.x] = cnt[threadIdx.x];
    if (cnt[threadIdx.x]) atomicOr(&info->types, 1u << threadIdx.x);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    info->off0 = off[0];
    info->len = off[E];
  }
}

__global__ void __launch_bounds__(256) k_conn_check(const int32_t* conn, int64_t L, int32_t N, UploadInfo* info) {
  const int64_t t = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (t < L && (uint32_t)conn[t] >= (uint32_t)N) atomicMin(&info->bad_conn, (unsigned long long)t);
}

// tile_off: the exclusive scan of tile_cnt.  Every element's node_map offset,
// and its place in the lists of its type: original id, node_map offset and
// connectivity, type after type (a mesh of one type needs none of the lists).
__global__ void __launch_bounds__(kUpThreads) k_upload_lists(const uint8_t* types, const int64_t* off,
                                                             const int32_t* conn, int64_t E, const int64_t* tile_off,
                                                             int64_t* map_off, int32_t* ids, int64_t* mapoff,
                                                             int32_t* packed, UploadInfo* info) {
  __shared__ int warp_cnt[kNumTypes][kUpThreads / 32];
  __shared__ int64_t base[kNumTypes + 1], run[kNumTypes], pack0[kNumTypes];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    int64_t p = 0;
    for (int k = 0; k <= kNumTypes; ++k) {
      base[k] = k < kNumTypes ? tile_off[(int64_t)k * gridDim.x] : E;
      if (blockIdx.x == 0) info->base[k] = base[k];
    }
    for (int k = 0; k < kNumTypes; ++k) {
      run[k] = tile_off[(int64_t)k * gridDim.x + blockIdx.x] - base[k];
      pack0[k] = p;
      p += up_nodes(k) * (base[k + 1] - base[k]);
    }
  }
  __syncthreads();
  bool uniform = false;
  for (int k = 0; k < kNumTypes; ++k) uniform |= base[k + 1] - base[k] == E;
  for (int r = 0; r < kUpRounds; ++r) {
    const int64_t e = (int64_t)blockIdx.x * kUpTile + r * kUpThreads + threadIdx.x;
    const int t = e < E ? (int)types[e] : -1;
    int before[kNumTypes];  // of each type, in the warp before this lane
#pragma unroll
    for (int k = 0; k < kNumTypes; ++k) {
      const unsigned m = __ballot_sync(0xffffffffu, t == k);
      before[k] = __popc(m & ((1u << lane) - 1u));
      if (lane == 0) warp_cnt[k][warp] = __popc(m);
    }
    __syncthreads();
    if (e < E) {
      int64_t mo = 0, rank = 0;
#pragma unroll
      for (int k = 0; k < kNumTypes; ++k) {
        int64_t c = run[k] + before[k];
        for (int w = 0; w < warp; ++w) c += warp_cnt[k][w];
        mo += c * (up_nodes(k) * up_nodes(k));
        if (k == t) rank = c;
      }
      map_off[e] = mo;
      const int nn = up_nodes(t);
      if (!uniform) {
        ids[base[t] + rank] = (int32_t)e;
        mapoff[base[t] + rank] = mo;
        int32_t* p = packed + pack0[t] + rank * nn;
        const int32_t* c = conn + off[e];
        for (int a = 0; a < nn; ++a) p[a] = c[a];
      }
      if (e == E - 1) map_off[E] = mo + nn * nn;
    }
    __syncthreads();
    if (threadIdx.x < kNumTypes)
      for (int w = 0; w < kUpThreads / 32; ++w) run[threadIdx.x] += warp_cnt[threadIdx.x][w];
    __syncthreads();
  }
}

int upload_mesh(const fea_mesh_desc* d, cudaStream_t s, fea_mesh** out) {
  if (!d || !out) return fail(FEA_ERR_ARG, "fea_mesh_upload: null argument");
  *out = nullptr;
  if (d->n_nodes <= 0 || d->n_elems <= 0) return fail(FEA_ERR_ARG, "fea_mesh_upload: empty mesh");
  if (d->n_nodes >= (1ll << 31) || d->n_elems >= (1ll << 31))
    return fail(FEA_ERR_INDEX_OVERFLOW, "fea_mesh_upload: n_nodes and n_elems must be < 2^31");
  if (!d->coords || !d->types || !d->conn_offsets || !d->conn)
    return fail(FEA_ERR_ARG, "fea_mesh_upload: null array");
  const int64_t N = d->n_nodes, E = d->n_elems;

  fea_mesh* m = new fea_mesh();
  auto leave = [&](int rc) {
    free_mesh(m);
    return rc;
  };
#define FEA_UP(call)                                        \
  do {                                                      \
    cudaError_t _e = (call);                                \
    if (_e != cudaSuccess) return leave(cuda_fail(_e, #call)); \
  } while (0)
  FEA_UP(cudaGetDevice(&m->device));
  m->n_nodes = N;
  m->n_elems = E;
  const int64_t tiles = (E + kUpTile - 1) / kUpTile;
  size_t bytes = 0;
  auto place = [&](size_t n) {
    const size_t at = bytes;
    bytes += (n + 255) & ~(size_t)255;
    return at;
  };
  auto alloc = [&](unsigned char** p) -> int {
    if (cudaMalloc((void**)p, bytes) == cudaSuccess) return FEA_OK;
    cudaGetLastError();
    *p = nullptr;
    return fail(FEA_ERR_OOM, "fea_mesh_upload: cudaMalloc of " + std::to_string(bytes) + " bytes failed");
  };
  const size_t a_coords = place(3 * N * 8), a_off = place((E + 1) * 8), a_moff = place((E + 1) * 8),
               a_types = place(E), a_status = place(sizeof(DevStatus)),
               a_info = place(sizeof(UploadInfo)), a_tiles = place(kNumTypes * tiles * 8);
  int rc = alloc(&m->arena);
  if (rc) return leave(rc);
  unsigned char* base = m->arena;
  m->coords = reinterpret_cast<double*>(base + a_coords);
  m->conn_off = reinterpret_cast<int64_t*>(base + a_off);
  m->map_off = reinterpret_cast<int64_t*>(base + a_moff);
  m->status = reinterpret_cast<DevStatus*>(base + a_status);
  UploadInfo* info = reinterpret_cast<UploadInfo*>(base + a_info);
  int64_t* tile_cnt = reinterpret_cast<int64_t*>(base + a_tiles);
  uint8_t* types = base + a_types;

  const cudaMemcpyKind kind = d->on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
  FEA_UP(cudaMemcpyAsync(m->conn_off, d->conn_offsets, (E + 1) * 8, kind, s));
  FEA_UP(cudaMemcpyAsync(types, d->types, E, kind, s));
  const DevStatus zero = {0, 0, ~0ull};
  UploadInfo got;
  std::memset(&got, 0, sizeof(got));
  got.bad_elem = got.bad_conn = ~0ull;
  FEA_UP(cudaMemcpyAsync(m->status, &zero, sizeof(zero), cudaMemcpyHostToDevice, s));
  FEA_UP(cudaMemcpyAsync(info, &got, sizeof(got), cudaMemcpyHostToDevice, s));
  k_upload_count<<<(unsigned)tiles, kUpThreads, 0, s>>>(types, m->conn_off, E, tile_cnt, info);
  FEA_UP(cudaGetLastError());
  // the length of conn is only known, and conn only read, once every offset is right
  FEA_UP(cudaMemcpyAsync(&got, info, sizeof(got), cudaMemcpyDeviceToHost, s));
  FEA_UP(cudaStreamSynchronize(s));
  if (got.off0 != 0) return leave(fail(FEA_ERR_ARG, "fea_mesh_upload: conn_offsets[0] != 0"));
  if (got.bad_elem != ~0ull) {
    const std::string e = std::to_string(got.bad_elem >> 1);
    return leave((got.bad_elem & 1)
                     ? fail(FEA_ERR_ARG, "fea_mesh_upload: conn_offsets does not match the node count of element " + e)
                     : fail(FEA_ERR_ARG, "fea_mesh_upload: unknown element type at element " + e));
  }
  const int64_t L = got.len;
  m->conn_len = L;
  bytes = 0;
  // the lists per type only where there are several types
  const bool lists = (got.types & (got.types - 1)) != 0;
  const size_t a_conn = place(L * 4), a_gmoff = place(lists ? E * 8 : 0), a_ids = place(lists ? E * 4 : 0),
               a_packed = place(lists ? L * 4 : 0);
  rc = alloc(&m->arena_conn);
  if (rc) return leave(rc);
  base = m->arena_conn;
  m->conn = reinterpret_cast<int32_t*>(base + a_conn);
  int32_t* packed = reinterpret_cast<int32_t*>(base + a_packed);
  int32_t* ids = reinterpret_cast<int32_t*>(base + a_ids);
  int64_t* gmoff = reinterpret_cast<int64_t*>(base + a_gmoff);
  FEA_UP(cudaMemcpyAsync(m->coords, d->coords, 3 * N * 8, kind, s));
  FEA_UP(cudaMemcpyAsync(m->conn, d->conn, L * 4, kind, s));
  k_conn_check<<<grid_for(L, 256), 256, 0, s>>>(m->conn, L, (int32_t)N, info);
  scan_tile_sums(tile_cnt, kNumTypes * tiles, s);
  k_upload_lists<<<(unsigned)tiles, kUpThreads, 0, s>>>(types, m->conn_off, m->conn, E, tile_cnt, m->map_off, ids,
                                                        gmoff, packed, info);
  FEA_UP(cudaGetLastError());
  FEA_UP(cudaMemcpyAsync(&got, info, sizeof(got), cudaMemcpyDeviceToHost, s));
  FEA_UP(cudaStreamSynchronize(s));
#undef FEA_UP
  if (got.bad_conn != ~0ull)
    return leave(fail(FEA_ERR_ARG, "fea_mesh_upload: node id out of range at conn[" + std::to_string(got.bad_conn) + "]"));

  int64_t pack0 = 0;
  for (int t = 0; t < kNumTypes; ++t) {
    TypeGroup& g = m->group[t];
    g.n = got.base[t + 1] - got.base[t];
    m->map_len += g.n * kNodesOf[t] * kNodesOf[t];
    if (g.n == E) {
      m->uniform = true;
      m->uniform_type = t;
      g.conn = m->conn;
    } else if (g.n) {
      g.conn = packed + pack0;
      g.ids = ids + got.base[t];
      g.mapoff = gmoff + got.base[t];
    }
    pack0 += g.n * kNodesOf[t];
  }
  rc = init_rule_constants();  // synchronous copy, so never inside a stream capture
  if (rc) return leave(rc);
  *out = m;
  return FEA_OK;
}

}  // namespace fea
