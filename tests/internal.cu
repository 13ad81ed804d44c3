// Parts of the library by themselves, for the tests: linked with its object files.
#include "../paper_1711_02242_gb300/csrc/oz.cuh"

namespace afq {
int mcd_bounded(int64_t dim, const double* d_V, double delta, int32_t max_vectors, double* d_L, int32_t* d_piv,
                int32_t* nvec, double* residual, void* d_work, long long wait_cycles, int sms, cudaStream_t s);
}

namespace {
struct Carve {
  char* p;
  char* end;
  void* take(size_t n) {
    n = (n + 255) & ~size_t(255);
    if (p + n > end) return nullptr;
    void* r = p;
    p += n;
    return r;
  }
  bool operand(afq::OzOperand& o, size_t rows, size_t k, int batch) {
    o.nkb = (int)((k + 15) / 16);
    o.batch_stride = (long)afq::oz_bytes(rows, o.rows_per_tile, o.RT, k);
    o.batch_exp_stride = (long)rows;
    o.data = take((size_t)batch * o.batch_stride);
    o.exps = static_cast<int*>(take((size_t)batch * rows * sizeof(int)));
    return o.data && o.exps;
  }
};
}  // namespace

// Sliced contractions: every pointer is a device pointer; ws holds the slices and
// row exponents, 256-byte aligned.
// C[m][n] = 2^alpha A B^T, rows of k values.
extern "C" __attribute__((visibility("default"))) int sp_gemm(const double* A, const double* B, int m, int n, int k,
                                                               double* C, int alpha, char* ws, size_t ws_bytes,
                                                               int* status, void* stream) {
  using namespace afq;
  Carve c{ws, ws + ws_bytes};
  OzGemm g;
  g.B.RT = g.B.rows_per_tile = 64;
  if (!c.operand(g.A, m, k, 1) || !c.operand(g.B, n, k, 1)) return AFQMC_ENOSPC;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  AFQ_TRY(oz_slice_rows(A, m, k, k, g.A, st));
  AFQ_TRY(oz_slice_rows(B, n, k, k, g.B, st));
  g.m = m;
  g.n = n;
  g.C = C;
  g.ldc = n;
  g.alpha_log2 = alpha;
  g.err = status;
  return oz_gemm_store(g, st);
}

// D[z][2 M][2 M] of groups of cw walkers (see oz_slice_densities).
extern "C" __attribute__((visibility("default"))) int sp_densities(
    const double* phi, const double* thA, const double* thB, int W, int N, int M, int cw, double* D, char* ws,
    size_t ws_bytes, int* status, void* stream) {
  using namespace afq;
  const int nz = (W + cw - 1) / cw;
  if (2 * N * cw > kOzSegK) return AFQMC_EINVAL;
  Carve c{ws, ws + ws_bytes};
  OzGemm g;
  g.B.RT = g.B.rows_per_tile = 64;
  if (!c.operand(g.A, 2 * (size_t)M, 2 * (size_t)N * cw, nz) || !c.operand(g.B, 2 * (size_t)M, 2 * (size_t)N * cw, nz))
    return AFQMC_ENOSPC;
  int* planes = static_cast<int*>(c.take(sizeof(int) * (size_t)nz * cw * 2 * N));
  if (!planes) return AFQMC_ENOSPC;
  g.m = g.n = 2 * M;
  g.batch = nz;
  g.ldc = 2L * M;
  g.c_batch = 4L * M * M;
  g.C = D;
  g.err = status;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  AFQ_TRY(oz_slice_densities(phi, thA, thB, W, N, M, 0, nz, cw, planes, g.A, g.B, st));
  return oz_gemm_store(g, st);
}

// The modified Cholesky decomposition whose waits end after wait_cycles, on a
// device of `sms` SMs (0: as it is).
extern "C" __attribute__((visibility("default"))) int in_mcd(long long dim, const double* V, double delta,
                                                              int max_vectors, double* L, int* piv, int* nvec,
                                                              double* residual, void* work, long long wait_cycles,
                                                              int sms, void* stream) {
  return afq::mcd_bounded(dim, V, delta, max_vectors, L, piv, nvec, residual, work, wait_cycles, sms,
                          static_cast<cudaStream_t>(stream));
}
