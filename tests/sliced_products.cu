// The sliced contractions by themselves, for test_gpu_sliced_products.py: linked
// with the library's object files.  Every pointer is a device pointer; ws holds
// the slices and row exponents, 256-byte aligned.
#include "../paper_1711_02242_gb300/csrc/oz.cuh"

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
  int* orb = static_cast<int*>(c.take(sizeof(int) * (size_t)nz * cw * N));
  if (!orb) return AFQMC_ENOSPC;
  g.m = g.n = 2 * M;
  g.batch = nz;
  g.ldc = 2L * M;
  g.c_batch = 4L * M * M;
  g.C = D;
  g.err = status;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  AFQ_TRY(oz_slice_densities(phi, thA, thB, W, N, M, 0, nz, cw, orb, g.A, g.B, st));
  return oz_gemm_store(g, st);
}
