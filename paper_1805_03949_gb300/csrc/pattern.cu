// pattern.cu -- the integer CSR pattern / element-to-nonzero map builder.
//
// The sparsity pattern of the assembled system is the node graph of the mesh
// (the local square matrices of Sec. 3.1 of the MPI+X assembly paper): nodes i
// and j couple iff some element holds both, the diagonal included.  It is
// built without a global sort:
//   1. node -> (element, local index) incidence lists (count, scan, fill);
//   2. one warp per node puts the nodes of its incident elements into a hash
//      table in shared memory, which leaves the distinct ones: their number is
//      the row length; a scan of the lengths gives the row pointers, and a
//      second pass ranks the distinct ones (rank = number of smaller ids) into
//      the sorted row;
//   3. the element-to-nonzero map: one warp per node looks its incident
//      elements' nodes up in the finished row;
//   4. the scalar pattern for ndof interleaved dofs per node is expanded from
//      the node pattern.
// Everything is integer work and deterministic: the atomics of step 1 only
// decide the order of the incidence lists, which no output depends on, and
// those of step 2 the order in which the distinct nodes are found, which the
// ranking removes.
#include <algorithm>
#include <cstdio>
#include <mutex>
#include <string>

#include "fea_internal.cuh"

namespace fea {

constexpr int kMaxCand = 1024;  // (element, node) incidences gathered per node

// ---------------------------------------------------------------------------
// exclusive scan int32 -> int64, out[n] = total (three passes)
// ---------------------------------------------------------------------------
constexpr int kScanBlock = 1024;
constexpr int kScanItems = 4;  // items per thread
constexpr int kScanTile = kScanBlock * kScanItems;

__device__ __forceinline__ int64_t block_excl_scan(int64_t v, int64_t* total) {
  __shared__ int64_t warp_sums[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int64_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int64_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_sums[warp] = x;
  __syncthreads();
  if (warp == 0) {
    int64_t w = (lane < (int)(blockDim.x >> 5)) ? warp_sums[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int64_t y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    warp_sums[lane] = w;  // inclusive
  }
  __syncthreads();
  int64_t base = warp ? warp_sums[warp - 1] : 0;
  if (total) *total = warp_sums[(blockDim.x >> 5) - 1];
  int64_t r = base + x - v;
  __syncthreads();
  return r;
}

__global__ void k_scan_reduce(const int32_t* in, int64_t n, int64_t* tile_sums) {
  int64_t base = (int64_t)blockIdx.x * kScanTile;
  int64_t s = 0;
  for (int k = 0; k < kScanItems; ++k) {
    int64_t i = base + (int64_t)k * kScanBlock + threadIdx.x;
    if (i < n) s += in[i];
  }
  int64_t tot;
  block_excl_scan(s, &tot);
  if (threadIdx.x == 0) tile_sums[blockIdx.x] = tot;
}

__global__ void k_scan_tiles(int64_t* tile_sums, int64_t ntiles) {
  // single CTA: exclusive scan of the tile sums in place, chunk by chunk
  __shared__ int64_t carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int64_t c = 0; c < ntiles; c += kScanBlock) {
    int64_t i = c + threadIdx.x;
    int64_t v = i < ntiles ? tile_sums[i] : 0;
    int64_t tot;
    int64_t ex = block_excl_scan(v, &tot);
    if (i < ntiles) tile_sums[i] = carry + ex;
    __syncthreads();
    if (threadIdx.x == 0) carry += tot;
    __syncthreads();
  }
}

__global__ void k_scan_apply(const int32_t* in, int64_t n, const int64_t* tile_offsets, int64_t* out) {
  // each thread owns kScanItems consecutive items of the tile
  int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
  int32_t v[kScanItems];
  int64_t s = 0;
  for (int k = 0; k < kScanItems; ++k) {
    v[k] = (base + k < n) ? in[base + k] : 0;
    s += v[k];
  }
  int64_t tot;
  int64_t ex = block_excl_scan(s, &tot) + tile_offsets[blockIdx.x];
  for (int k = 0; k < kScanItems; ++k) {
    if (base + k < n) out[base + k] = ex;
    ex += v[k];
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == blockDim.x - 1) out[n] = tile_offsets[blockIdx.x] + tot;
}

void scan_tile_sums(int64_t* tile_sums, int64_t n, cudaStream_t s) {
  k_scan_tiles<<<1, kScanBlock, 0, s>>>(tile_sums, n);
}

// tiles: scratch of scan_tiles(n) values
static int64_t scan_tiles(int64_t n) { return std::max<int64_t>((n + kScanTile - 1) / kScanTile, 1); }

static int exclusive_scan_i32(const int32_t* in, int64_t n, int64_t* out, int64_t* tiles, cudaStream_t s) {
  const int64_t ntiles = scan_tiles(n);
  k_scan_reduce<<<(unsigned)ntiles, kScanBlock, 0, s>>>(in, n, tiles);
  k_scan_tiles<<<1, kScanBlock, 0, s>>>(tiles, ntiles);
  k_scan_apply<<<(unsigned)ntiles, kScanBlock, 0, s>>>(in, n, tiles, out);
  FEA_CUDA(cudaGetLastError());
  return FEA_OK;
}

// ---------------------------------------------------------------------------
// node -> incidence lists
// ---------------------------------------------------------------------------
__global__ void k_inc_count(const int32_t* conn, int64_t len, int32_t* cnt) {
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < len) atomicAdd(&cnt[conn[t]], 1);
}

// cnt[node] counts down from the number of incidences to 0
__global__ void k_inc_fill(const int64_t* conn_off, const int32_t* conn, int64_t n_elems, const int64_t* inc_off,
                           int32_t* cnt, int64_t* inc) {
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n_elems) return;
  const int64_t o = conn_off[e];
  const int nn = (int)(conn_off[e + 1] - o);
  for (int a = 0; a < nn; ++a) {
    const int32_t node = conn[o + a];
    inc[inc_off[node] + atomicSub(&cnt[node], 1) - 1] = e * 16 + a;
  }
}

// ---------------------------------------------------------------------------
// rows: one warp per node
// ---------------------------------------------------------------------------
// The incident elements of a node in slots of 8 lanes: lane s reads node s % 8
// of incidence s / 8 (lanes past the element's nodes rest), so a warp reads
// four elements' nodes at once.  uniform_nn > 0: every element has that many nodes.
struct RowMesh {
  const int64_t* inc_off;
  const int64_t* inc;
  const int64_t* conn_off;
  const int32_t* conn;
  const int64_t* map_off;
  int uniform_nn;
};

__device__ __forceinline__ int32_t row_candidate(const RowMesh& M, int64_t i0, int64_t i1, int64_t first, int lane,
                                                 int64_t* dst) {
  const int64_t t = i0 + first + (lane >> 3);
  const int b = lane & 7;
  if (t >= i1) return -1;
  const int64_t v = M.inc[t], e = v >> 4;
  const int64_t o = M.uniform_nn ? e * M.uniform_nn : M.conn_off[e];
  const int nn = M.uniform_nn ? M.uniform_nn : (int)(M.conn_off[e + 1] - o);
  if (b >= nn) return -1;
  if (dst) *dst = (M.uniform_nn ? e * nn * nn : M.map_off[e]) + (v & 15) * nn + b;
  return M.conn[o + b];
}

// Distinct nodes of node i's incident elements, by the warp, into list (in no
// order); their number, or -1 past kMaxCand incidences.  tab: H slots, a power
// of two no smaller than 8 times the incidences or than kMaxCand.
__device__ __forceinline__ int row_distinct(const RowMesh& M, int64_t i0, int64_t i1, int32_t* tab, int H,
                                            int32_t* list) {
  const int lane = threadIdx.x & 31;
  for (int h = lane; h < H; h += 32) tab[h] = -1;
  __syncwarp();
  const int shift = 32 - (31 - __clz(H));
  int D = 0, C = 0;
  for (int64_t f = 0; i0 + f < i1; f += 4) {
    const int32_t key = row_candidate(M, i0, i1, f, lane, nullptr);
    C += __popc(__ballot_sync(0xffffffffu, key >= 0));
    if (C > kMaxCand) return -1;
    bool fresh = false;
    if (key >= 0) {
      uint32_t h = ((uint32_t)key * 2654435769u) >> shift;  // Fibonacci hashing (Knuth, TAOCP 3, 6.4)
      for (;;) {
        const int32_t seen = *(volatile int32_t*)&tab[h];
        if (seen == key) break;
        if (seen < 0) {
          const int32_t was = atomicCAS(&tab[h], -1, key);
          if (was < 0) fresh = true;
          if (was < 0 || was == key) break;
        }
        h = (h + 1) & (uint32_t)(H - 1);
      }
    }
    const unsigned m = __ballot_sync(0xffffffffu, fresh);
    if (fresh && list) list[D + __popc(m & ((1u << lane) - 1u))] = key;
    D += __popc(m);
  }
  __syncwarp();
  return D;
}

// FILL false: deg[i] = number of distinct neighbours of node i; true: the
// sorted row i of col_node.  H: hash slots per warp.  Nodes with more than
// H / 8 incidences are left to the launch with the larger table: the first
// launch (todo != nullptr) appends them to todo[1 ..], *todo their number; the
// second (nodes != nullptr) takes them from there.
template <int H, bool FILL>
__global__ void __launch_bounds__(128) k_rows(RowMesh M, int64_t n_nodes, int32_t* deg, const int64_t* rp,
                                              int32_t* col_node, int32_t* todo, const int32_t* nodes,
                                              DevStatus* st) {
  constexpr int kList = H < kMaxCand ? H : kMaxCand;
  __shared__ int32_t s_tab[4][H];
  __shared__ __align__(16) int32_t s_list[FILL ? 4 : 1][FILL ? kList : 4];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t n = nodes ? nodes[0] : n_nodes;
  for (int64_t k = (int64_t)blockIdx.x * 4 + warp; k < n; k += (int64_t)gridDim.x * 4) {
    const int64_t i = nodes ? nodes[1 + k] : k;
    const int64_t i0 = M.inc_off[i], i1 = M.inc_off[i + 1];
    if (!nodes && i1 - i0 > H / 8) {
      if (lane == 0) todo[1 + atomicAdd(todo, 1)] = (int32_t)i;
      continue;
    }
    int h = 32;
    while (h < H && h < 8 * (i1 - i0)) h *= 2;
    int32_t* list = FILL ? s_list[warp] : nullptr;
    const int D = row_distinct(M, i0, i1, s_tab[warp], h, list);
    if (D < 0) {
      if (lane == 0) {
        latch_error(st, FEA_ERR_UNSUPPORTED, (unsigned long long)i);
        if (!FILL) deg[i] = 0;
      }
      continue;
    }
    if constexpr (!FILL) {
      if (lane == 0) deg[i] = D;
    } else {
      if (lane < 4 && D + lane < ((D + 3) & ~3)) list[D + lane] = INT32_MAX;
      __syncwarp();
      const int4* l4 = reinterpret_cast<const int4*>(list);
      for (int u = lane; u < D; u += 32) {
        const int32_t key = list[u];
        int r = 0;
        for (int w = 0; w < (D + 3) / 4; ++w) {
          const int4 v = l4[w];
          r += (v.x < key) + (v.y < key) + (v.z < key) + (v.w < key);
        }
        col_node[rp[i] + r] = key;
      }
      __syncwarp();
    }
  }
}
constexpr int kRowSlots = 512;            // first launch: nodes of up to 64 elements
constexpr int kRowSlotsMax = 2 * kMaxCand;  // second: as many as kMaxCand allows (an element has at least 4 nodes)

// Every row pass: the nodes of few elements, then the others.  A node of more
// than kMaxCand / 4 elements is past the limit whatever they are.
template <bool FILL>
static int launch_rows(const fea_mesh* m, const RowMesh& M, int32_t* deg, int32_t* todo, cudaStream_t s) {
  FEA_CUDA(cudaMemsetAsync(todo, 0, sizeof(int32_t), s));
  k_rows<kRowSlots, FILL><<<grid_for(m->n_nodes, 4), 128, 0, s>>>(M, m->n_nodes, deg, m->rp_node, m->col_node, todo,
                                                                  nullptr, m->status);
  k_rows<kRowSlotsMax, FILL><<<1024, 128, 0, s>>>(M, m->n_nodes, deg, m->rp_node, m->col_node, nullptr, todo,
                                                  m->status);
  FEA_CUDA(cudaGetLastError());
  return FEA_OK;
}

// node_map: the place of every incident element's nodes in the finished row
__global__ void __launch_bounds__(256) k_node_map(RowMesh M, int64_t n_nodes, const int64_t* rp,
                                                  const int32_t* col_node, int32_t* node_map) {
  const int lane = threadIdx.x & 31;
  const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (i >= n_nodes) return;
  const int64_t i0 = M.inc_off[i], i1 = M.inc_off[i + 1], r0 = rp[i];
  const int32_t* row = col_node + r0;
  const int deg = (int)(rp[i + 1] - r0);
  for (int64_t f = 0; i0 + f < i1; f += 4) {
    int64_t dst = 0;
    const int32_t key = row_candidate(M, i0, i1, f, lane, &dst);
    if (key < 0) continue;
    int lo = 0, hi = deg;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (__ldg(row + mid) < key)
        lo = mid + 1;
      else
        hi = mid;
    }
    node_map[dst] = lo;
  }
}

// ---------------------------------------------------------------------------
// scalar expansion for 3 dofs per node: one warp per node, whose three rows
// hold the same columns one after the other
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_expand3(int64_t n_nodes, const int64_t* rp, const int32_t* col_node,
                                                 int64_t* row_ptr, int32_t* col_idx) {
  const int lane = threadIdx.x & 31;
  const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (i >= n_nodes) return;
  const int64_t r0 = rp[i], base = 9 * r0;
  const int len = 3 * (int)(rp[i + 1] - r0);
  if (lane < 3) row_ptr[3 * i + lane] = base + (int64_t)lane * len;
  if (i == n_nodes - 1 && lane == 0) row_ptr[3 * n_nodes] = base + 3 * (int64_t)len;
  if (!col_idx) return;
  int32_t* out = col_idx + base;
  for (int t = lane; t < len; t += 32) {
    const int k = t / 3;
    const int32_t c = 3 * __ldg(col_node + r0 + k) + (t - 3 * k);
    out[t] = c;
    out[len + t] = c;
    out[2 * (int64_t)len + t] = c;
  }
}

__global__ void k_copy_i64(const int64_t* src, int64_t* dst, int64_t n) {
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) dst[t] = src[t];
}

static int read_status(fea_mesh* m, cudaStream_t s, int* code, unsigned long long* info) {
  DevStatus st;
  FEA_CUDA(cudaMemcpyAsync(&st, m->status, sizeof(st), cudaMemcpyDeviceToHost, s));
  FEA_CUDA(cudaStreamSynchronize(s));
  *code = st.code;
  *info = st.info;
  return FEA_OK;
}

static RowMesh row_mesh(const fea_mesh* m) {
  return {m->inc_off, m->inc, m->conn_off, m->conn, m->map_off, m->uniform ? kNodesOf[m->uniform_type] : 0};
}

static void drop_graph(fea_mesh* m) {
  cudaFree(m->graph);
  cudaFree(m->col_node);
  m->graph = nullptr;
  m->inc_off = m->inc = m->rp_node = nullptr;
  m->col_node = nullptr;
}

static int node_graph(fea_mesh* m, cudaStream_t s) {
  const int64_t N = m->n_nodes, E = m->n_elems, L = m->conn_len;
  // one allocation: incidence offsets and lists, row pointers, the scans'
  // scratch, and two int32 work arrays (counts, then row lengths; the nodes of
  // many elements)
  size_t bytes = 0;
  auto place = [&](size_t n) {
    const size_t at = bytes;
    bytes += (n + 255) & ~(size_t)255;
    return at;
  };
  const size_t a_off = place((size_t)(N + 1) * 8), a_inc = place((size_t)L * 8), a_rp = place((size_t)(N + 1) * 8),
               a_tiles = place((size_t)scan_tiles(N) * 8), a_cnt = place((size_t)N * 4),
               a_todo = place((size_t)(N + 1) * 4);
  FEA_CUDA(cudaMalloc((void**)&m->graph, bytes));
  m->inc_off = reinterpret_cast<int64_t*>(m->graph + a_off);
  m->inc = reinterpret_cast<int64_t*>(m->graph + a_inc);
  m->rp_node = reinterpret_cast<int64_t*>(m->graph + a_rp);
  int64_t* tiles = reinterpret_cast<int64_t*>(m->graph + a_tiles);
  int32_t* cnt = reinterpret_cast<int32_t*>(m->graph + a_cnt);
  int32_t* todo = reinterpret_cast<int32_t*>(m->graph + a_todo);
  FEA_CUDA(cudaMemsetAsync(cnt, 0, N * sizeof(int32_t), s));
  k_inc_count<<<grid_for(L, 256), 256, 0, s>>>(m->conn, L, cnt);
  int rc = exclusive_scan_i32(cnt, N, m->inc_off, tiles, s);
  if (rc) return rc;
  k_inc_fill<<<grid_for(E, 256), 256, 0, s>>>(m->conn_off, m->conn, E, m->inc_off, cnt, m->inc);
  const RowMesh M = row_mesh(m);
  rc = launch_rows<false>(m, M, cnt, todo, s);
  if (rc) return rc;
  rc = exclusive_scan_i32(cnt, N, m->rp_node, tiles, s);
  if (rc) return rc;
  FEA_CUDA(cudaMemcpyAsync(&m->nnz_node, m->rp_node + N, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  int code = 0;
  unsigned long long info = 0;
  rc = read_status(m, s, &code, &info);
  if (rc) return rc;
  if (code) {
    DevStatus zero = {0, 0, ~0ull};
    cudaMemcpy(m->status, &zero, sizeof(zero), cudaMemcpyHostToDevice);
    return fail(code, "pattern: node " + std::to_string(info) + " gathers more than " + std::to_string(kMaxCand) +
                          " (element, node) incidences");
  }
  FEA_CUDA(cudaMalloc(&m->col_node, (m->nnz_node ? m->nnz_node : 1) * sizeof(int32_t)));
  rc = launch_rows<true>(m, M, nullptr, todo, s);
  if (rc) return rc;
  FEA_CUDA(cudaStreamSynchronize(s));
  return FEA_OK;
}

int build_node_graph(fea_mesh* m, cudaStream_t s) {
  const int rc = node_graph(m, s);
  if (rc) drop_graph(m);
  return rc;
}

int write_csr_pattern(fea_mesh* m, int ndof, int64_t* row_ptr, int32_t* col_idx, int32_t* node_map,
                      cudaStream_t s) {
  const int64_t N = m->n_nodes;
  if (node_map)
    k_node_map<<<grid_for(N * 32, 256), 256, 0, s>>>(row_mesh(m), N, m->rp_node, m->col_node, node_map);
  if (ndof == 1) {
    k_copy_i64<<<grid_for(N + 1, 256), 256, 0, s>>>(m->rp_node, row_ptr, N + 1);
    if (col_idx)
      FEA_CUDA(cudaMemcpyAsync(col_idx, m->col_node, m->nnz_node * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
  } else {
    k_expand3<<<grid_for(N * 32, 256), 256, 0, s>>>(N, m->rp_node, m->col_node, row_ptr, col_idx);
  }
  FEA_CUDA(cudaGetLastError());
  return FEA_OK;
}

// ---------------------------------------------------------------------------
// Row pointers from row lengths without any device allocation.
//
// The scan above takes its per-tile partial sums from the mesh handle's
// allocation.  Callers that hand all device memory to their own pool up
// front, or that must not let a library allocate on their behalf, use
// fea_row_ptr_from_counts_noalloc instead: the tile sums live in the
// file-scope array below, which every GPU that loads the library holds until
// the process exits.
// ---------------------------------------------------------------------------
constexpr int64_t kNoAllocMaxTiles = 16384;                      // 128 KB of tile sums
constexpr int64_t kNoAllocMaxCounts = kNoAllocMaxTiles * kScanTile;  // 67,108,864 rows
constexpr int kNoAllocMaxDevices = 64;

static __device__ __align__(256) int64_t g_noalloc_tiles[kNoAllocMaxTiles];

static std::mutex g_noalloc_mutex;
static int64_t* g_noalloc_ptr[kNoAllocMaxDevices];  // device address of g_noalloc_tiles, per device

// Device address of the scratch array on the current device: taken once per
// device, with that device current, on the first call there.
static int noalloc_scratch(int64_t** out) {
  int dev = 0;
  FEA_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kNoAllocMaxDevices)
    return fail(FEA_ERR_UNSUPPORTED, "fea_row_ptr_from_counts_noalloc: device index " + std::to_string(dev) +
                                         " beyond the supported " + std::to_string(kNoAllocMaxDevices));
  std::lock_guard<std::mutex> lock(g_noalloc_mutex);
  if (!g_noalloc_ptr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_tiles);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_noalloc_tiles)");
    g_noalloc_ptr[dev] = (int64_t*)p;
  }
  *out = g_noalloc_ptr[dev];
  return FEA_OK;
}

}  // namespace fea

extern "C" int fea_row_ptr_from_counts_noalloc(const int32_t* counts, int64_t n, int64_t* row_ptr, void* stream) {
  using namespace fea;
  if (n < 0 || !row_ptr || (n > 0 && !counts))
    return fail(FEA_ERR_ARG, "fea_row_ptr_from_counts_noalloc: null pointer or negative length");
  if (n > kNoAllocMaxCounts)
    return fail(FEA_ERR_UNSUPPORTED, "fea_row_ptr_from_counts_noalloc: " + std::to_string(n) +
                                         " rows exceed the fixed scratch limit of " +
                                         std::to_string(kNoAllocMaxCounts));
  int64_t* tiles = nullptr;
  int rc = noalloc_scratch(&tiles);
  if (rc != FEA_OK) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  int64_t ntiles = (n + kScanTile - 1) / kScanTile;
  if (ntiles < 1) ntiles = 1;
  // every tile sum read below is written first by k_scan_reduce, so the
  // scratch left by an earlier call needs no clearing
  k_scan_reduce<<<(unsigned)ntiles, kScanBlock, 0, s>>>(counts, n, tiles);
  k_scan_tiles<<<1, kScanBlock, 0, s>>>(tiles, ntiles);
  k_scan_apply<<<(unsigned)ntiles, kScanBlock, 0, s>>>(counts, n, tiles, row_ptr);
  FEA_CUDA(cudaGetLastError());
  return FEA_OK;
}
