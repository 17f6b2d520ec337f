// One block column of the FP64 factorization on its own, for the tests: an m x bw panel (column-major, bw <= 64, the
// covariance's lower part) through the kernels that factor its diagonal tile, invert it and solve the rows below.
#include <cstring>
#include <vector>

#include "trsm64.cuh"

namespace {
struct Buffers {   // frees what it allocated
  std::vector<void*> p;
  cudaError_t e = cudaSuccess;
  template <class V>
  V* make(size_t n, const V* src = nullptr) {
    void* d = nullptr;
    if (e == cudaSuccess) e = cudaMalloc(&d, (n + 1) * sizeof(V));
    if (e != cudaSuccess) return nullptr;
    p.push_back(d);
    e = src ? cudaMemcpy(d, src, n * sizeof(V), cudaMemcpyHostToDevice) : cudaMemset(d, 0, (n + 1) * sizeof(V));
    return (V*)d;
  }
  ~Buffers() {
    for (void* d : p) cudaFree(d);
  }
};
}  // namespace

// panel: in the covariance, out L. dinv: 64 x 64, the inverse of the diagonal block, row-major. diag: the m rows' variances.
// status[0]: smallest failing column (INT32_MAX: none), status[1]: nonzero if a wait ran out. Returns a cudaError_t.
extern "C" __attribute__((visibility("default"))) int fp64_panel(double* panel, int m, int bw, const double* diag, double* dinv, int32_t* status) {
  if (m < 1 || m > 4096 || bw < 1 || bw > 64 || bw > m) return -1;
  const int nt = (m - bw + TRSM_ROWS - 1) / TRSM_ROWS;
  std::vector<int32_t> rows(m), rho(m);
  for (int i = 0; i < m; i++) {
    rows[i] = i;
    uint64_t u;
    std::memcpy(&u, &diag[i], 8);
    rho[i] = (((int)((u >> 52) & 0x7ff) - 1023 + 2) >> 1) - 1;   // as k_row_scale
  }
  const int32_t w = bw, r = m - bw, zero = 0, none = INT32_MAX;
  const int64_t z64 = 0, pre[2] = {0, nt};
  Buffers b;
  DevPlan dp{};
  dp.w = b.make(1, &w);
  dp.r = b.make(1, &r);
  dp.loff = b.make(1, &z64);
  dp.doff = b.make(1, &z64);
  dp.frow_off = b.make(1, &z64);
  dp.frows = b.make(m, rows.data());
  dp.sn_first = b.make(1, &zero);
  double* P = b.make((size_t)m * bw, (const double*)panel);
  double* D = b.make<double>(64 * 64);
  uint8_t* tile = b.make<uint8_t>(p64::TILE_BYTES);
  __half* op = b.make<__half>((size_t)f64d::NS * m * 64);
  int32_t *fronts = b.make(1, &zero), *slot = b.make(1, &zero), *d_rho = b.make(m, (const int32_t*)rho.data());
  int64_t* d_pre = b.make(2, pre);
  int32_t *notpd = b.make(1, &none), *err = b.make<int32_t>(1);
  CUtensorMap map;
  cudaDriverEntryPointQueryResult qr;
  void* fn = nullptr;
  if (b.e == cudaSuccess) b.e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &qr);
  if (b.e != cudaSuccess || !fn) return b.e ? (int)b.e : -2;
  cuuint64_t dims[4] = {64, (cuuint64_t)m, f64d::NS, 1}, strides[3] = {128, (cuuint64_t)m * 128, (cuuint64_t)f64d::NS * m * 128};
  cuuint32_t box[4] = {64, 64, 1, 1}, es[4] = {1, 1, 1, 1};
  if (((PFN_cuTensorMapEncodeTiled_v12000)fn)(&map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, op, dims, strides, box, es,
                                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return -3;
  uint8_t* d_map = b.make(sizeof(map), (const uint8_t*)&map);
  if (b.e == cudaSuccess) b.e = cudaFuncSetAttribute(k_potrf64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(p64::Smem));
  if (b.e == cudaSuccess) b.e = cudaFuncSetAttribute(k_trsm64, cudaFuncAttributeMaxDynamicSharedMemorySize, TRSM_SMEM);
  if (b.e != cudaSuccess) return (int)b.e;
  const int64_t PE = (int64_t)m * bw;
  k_potrf64<<<dim3(2, 1), p64::THREADS, sizeof(p64::Smem)>>>(fronts, 0, dp, P, PE, notpd, D, 4096, tile, p64::TILE_BYTES, err);
  if (nt > 0)
    k_trsm64<<<dim3(nt, 1), TRSM_THREADS, TRSM_SMEM>>>(fronts, d_pre, 1, 0, dp, P, PE, tile, p64::TILE_BYTES, d_rho, m, d_map, slot,
                                             notpd, err, tcg::DEFAULT_WAIT);
  b.e = cudaGetLastError();
  if (b.e == cudaSuccess) b.e = cudaMemcpy(panel, P, PE * sizeof(double), cudaMemcpyDeviceToHost);
  if (b.e == cudaSuccess) b.e = cudaMemcpy(dinv, D, 4096 * sizeof(double), cudaMemcpyDeviceToHost);
  if (b.e == cudaSuccess) b.e = cudaMemcpy(&status[0], notpd, 4, cudaMemcpyDeviceToHost);
  if (b.e == cudaSuccess) b.e = cudaMemcpy(&status[1], err, 4, cudaMemcpyDeviceToHost);
  return (int)b.e;
}
