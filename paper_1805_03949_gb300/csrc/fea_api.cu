// fea_api.cu -- the C-ABI entry points: errors, mesh handles, pattern calls,
// assemble, check.
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "fea_internal.cuh"

namespace fea {

static thread_local std::string g_err;

void set_error(const std::string& msg) { g_err = msg; }

int fail(int code, const std::string& msg) {
  g_err = msg;
  return code;
}

int cuda_fail(cudaError_t e, const char* what) {
  g_err = std::string("CUDA error in ") + what + ": " + cudaGetErrorString(e);
  return FEA_ERR_CUDA;
}

void free_mesh(fea_mesh* m) {
  if (!m) return;
  cudaFree(m->arena);
  cudaFree(m->arena_conn);
  cudaFree(m->graph);
  cudaFree(m->col_node);
  drop_rows_plans(m);
  cudaFree(m->geo[0]);
  cudaFree(m->geo[1]);
  fea::free_sched(m);
  free_color_plan(m);
  free_multidep_plan(m);
  if (m->blocks) {
    free_rows_plan(m->blocks);
    delete m->blocks;
  }
  delete m;
}

}  // namespace fea

using namespace fea;

extern "C" {

const char* fea_last_error(void) { return fea::g_err.c_str(); }

int fea_abi_version(void) { return FEA_ABI_VERSION; }

int fea_mesh_upload(const fea_mesh_desc* desc, void* stream, fea_mesh** out) {
  return upload_mesh(desc, (cudaStream_t)stream, out);
}

int fea_mesh_set_coords(fea_mesh* m, const double* coords, int on_device, void* stream) {
  if (!m || !coords) return fail(FEA_ERR_ARG, "fea_mesh_set_coords: null argument");
  FEA_CUDA(cudaMemcpyAsync(m->coords, coords, 3 * m->n_nodes * sizeof(double),
                           on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, (cudaStream_t)stream));
  return FEA_OK;
}

int fea_mesh_destroy(fea_mesh* mesh) {
  if (!mesh) return fail(FEA_ERR_ARG, "fea_mesh_destroy: null handle");
  cudaDeviceSynchronize();
  free_mesh(mesh);
  return FEA_OK;
}

int fea_mesh_info(const fea_mesh* m, int64_t* n_nodes, int64_t* n_elems, int64_t* map_len) {
  if (!m) return fail(FEA_ERR_ARG, "fea_mesh_info: null handle");
  if (n_nodes) *n_nodes = m->n_nodes;
  if (n_elems) *n_elems = m->n_elems;
  if (map_len) *map_len = m->map_len;
  return FEA_OK;
}

int fea_pattern_size(fea_mesh* m, int ndof, int64_t* nnz, void* stream) {
  if (!m || !nnz) return fail(FEA_ERR_ARG, "fea_pattern_size: null argument");
  if (ndof != 1 && ndof != 3) return fail(FEA_ERR_ARG, "fea_pattern_size: ndof must be 1 or 3");
  if ((int64_t)ndof * m->n_nodes >= (1ll << 31))
    return fail(FEA_ERR_INDEX_OVERFLOW, "fea_pattern_size: ndof * n_nodes must be < 2^31 (int32 columns)");
  cudaStream_t s = (cudaStream_t)stream;
  if (!m->rp_node) {
    int rc = build_node_graph(m, s);
    if (rc != FEA_OK) return rc;
  }
  m->pattern_ndof = ndof;
  m->pattern_built = false;
  *nnz = (int64_t)ndof * ndof * m->nnz_node;
  return FEA_OK;
}

int fea_build_csr_pattern(fea_mesh* m, int ndof, int64_t* row_ptr, int32_t* col_idx, int32_t* node_map,
                          void* stream) {
  if (!m || !row_ptr) return fail(FEA_ERR_ARG, "fea_build_csr_pattern: null argument");
  if (!m->rp_node || m->pattern_ndof != ndof)
    return fail(FEA_ERR_ARG, "fea_build_csr_pattern: call fea_pattern_size with the same ndof first");
  int rc = write_csr_pattern(m, ndof, row_ptr, col_idx, node_map, (cudaStream_t)stream);
  if (rc == FEA_OK && node_map) m->pattern_built = true;
  return rc;
}

int fea_assemble(const fea_operator* op, fea_mesh* m, const int64_t* row_ptr, const int32_t* node_map,
                 double* A, double* b, void* stream) {
  // rows of complete entry blocks are written with 16-byte stores
  if (((uintptr_t)A & 15u) != 0 || ((uintptr_t)b & 7u) != 0)
    return fail(FEA_ERR_ARG, "fea_assemble: A_vals_d must be 16-byte aligned and b_d 8-byte aligned");
  return fea::assemble(op, m, row_ptr, node_map, A, b, (cudaStream_t)stream);
}

int fea_mesh_set_rows_block(fea_mesh* m, int block_nodes) {
  if (!m) return fail(FEA_ERR_ARG, "fea_mesh_set_rows_block: null handle");
  if (block_nodes < 1 || block_nodes > 512) return fail(FEA_ERR_ARG, "fea_mesh_set_rows_block: block size in [1, 512]");
  if (block_nodes != m->rows_block_nodes) {
    cudaDeviceSynchronize();
    drop_rows_plans(m);
  }
  m->rows_block_nodes = block_nodes;
  return FEA_OK;
}

int fea_mesh_set_block_elems(fea_mesh* m, int block_elems) {
  if (!m) return fail(FEA_ERR_ARG, "fea_mesh_set_block_elems: null handle");
  if (block_elems < 1 || block_elems > kRowsStageHalo)
    return fail(FEA_ERR_ARG, "fea_mesh_set_block_elems: elements per block in [1, " + std::to_string(kRowsStageHalo) + "]");
  if (block_elems != m->block_elems && m->blocks) {
    cudaDeviceSynchronize();
    free_rows_plan(m->blocks);
    delete m->blocks;
    m->blocks = nullptr;
  }
  m->block_elems = block_elems;
  return FEA_OK;
}

int fea_rows_plan_info(const fea_mesh* m, int64_t info[8]) {
  if (!m || !info) return fail(FEA_ERR_ARG, "fea_rows_plan_info: null argument");
  for (int k = 0; k < 8; ++k) info[k] = 0;
  const fea::RowsPlan* pp = m->rows[1] ? m->rows[1] : m->rows[0];
  if (!pp) return FEA_OK;
  const fea::RowsPlan& P = *pp;
  info[0] = P.n_blocks;
  info[1] = P.block_nodes;
  info[2] = P.max_local;
  info[3] = P.max_helem;
  info[4] = P.n_tasks;
  info[5] = P.n_contrib;
  info[6] = P.n_helem_total;
  info[7] = (int64_t)P.bytes;
  return FEA_OK;
}

int fea_color_info(const fea_mesh* m, int32_t* colors_h, int* n_colors) {
  if (!m || !n_colors) return fail(FEA_ERR_ARG, "fea_color_info: null argument");
  if (!m->color) return fail(FEA_ERR_ARG, "fea_color_info: no coloring yet (run a FEA_SCATTER_COLOR assembly)");
  *n_colors = m->color->n_colors;
  if (colors_h) std::memcpy(colors_h, m->color->colors_host.data(), m->n_elems * sizeof(int32_t));
  return FEA_OK;
}

int fea_assemble_launches(const fea_operator* op, const fea_mesh* m, int* n_kernels) {
  return fea::assemble_launches(op, m, n_kernels);
}

int fea_check(fea_mesh* m, void* stream) {
  if (!m) return fail(FEA_ERR_ARG, "fea_check: null handle");
  cudaStream_t s = (cudaStream_t)stream;
  FEA_CUDA(cudaStreamSynchronize(s));
  FEA_CUDA(cudaGetLastError());
  DevStatus st;
  FEA_CUDA(cudaMemcpy(&st, m->status, sizeof(st), cudaMemcpyDeviceToHost));
  if (st.code == 0) return FEA_OK;
  DevStatus zero = {0, 0, ~0ull};
  FEA_CUDA(cudaMemcpy(m->status, &zero, sizeof(zero), cudaMemcpyHostToDevice));
  switch (st.code) {
    case FEA_ERR_INVERTED_ELEMENT:
      return fail(st.code, "inverted element: det J <= 0 at a quadrature point of element " + std::to_string(st.info));
    case FEA_ERR_UNSUPPORTED:
      return fail(st.code, "node " + std::to_string(st.info) +
                               " gathers more than 1024 (element, node) incidences (pattern builder limit)");
    default:
      return fail(st.code, "device error " + std::to_string(st.code) + " (id " + std::to_string(st.info) + ")");
  }
}

}  // extern "C"
