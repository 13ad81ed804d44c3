// Float64 contractions as exact integer products on the tensor cores: slicing
// kernels and the contraction (see oz.cuh for the number format).
#include <vector>

#include "oz.cuh"
#include "tc.cuh"
#include "tc_dev.cuh"

namespace afq {
namespace {

using namespace tc;

constexpr int kS = kOzSlices;
constexpr long long kDigitBias = 64ll * (1ll + (1ll << 7) + (1ll << 14) + (1ll << 21) + (1ll << 28) +
                                         (1ll << 35) + (1ll << 42));

// ---------------------------------------------------------------- slicing ---
// |x| as the high word of its bits without the sign: monotonic in |x|.
__device__ __forceinline__ uint32_t abs_hi(double x) { return (uint32_t)__double2hiint(x) & 0x7fffffffu; }

// Row exponent e with 2^e above every element, from the largest abs_hi.
__device__ __forceinline__ int row_exp(uint32_t hi, bool any) {
  const int ef = (int)(hi >> 20);
  if (ef == 0x7ff) return kOzNanExp;
  if (!any) return kOzZeroExp;
  return (ef > 0 ? ef : 1) - 1022;
}

// The same for one element scaled by 2^-s: a row's exponent is the largest.
__device__ __forceinline__ int elem_exp(double x, int s) {
  const uint32_t hi = abs_hi(x);
  const int ef = (int)(hi >> 20);
  if (ef == 0x7ff) return kOzNanExp;
  if ((hi | (uint32_t)__double2loint(x)) == 0u) return kOzZeroExp;
  return (ef > 0 ? ef : 1) - 1022 - s;
}

// x in units of 2^(e - 56), rounded to nearest (|X| <= 2^56).
__device__ __forceinline__ long long fixed57(double x, int e) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int ef = (int)(u >> 52) & 0x7ff;
  unsigned long long m = u & 0xfffffffffffffull;
  if (ef) m |= 1ull << 52;
  const int sh = (ef ? ef : 1) - 1019 - e;  // 3 for the largest element's binade
  unsigned long long r;
  if (sh >= 0) {
    r = m << sh;
  } else if (sh >= -54) {
    r = (m + (1ull << (-sh - 1))) >> -sh;
  } else {
    r = 0;
  }
  return (long long)u < 0 ? -(long long)r : (long long)r;
}

// Two integers |d| <= 128 as a pair of BF16 (exact).
__device__ __forceinline__ uint32_t bf16_pair(int lo, int hi) {
  const uint32_t a = __float_as_uint(__int_as_float(0x4b400000 + lo) - 12582912.0f);
  const uint32_t b = __float_as_uint(__int_as_float(0x4b400000 + hi) - 12582912.0f);
  return __byte_perm(a, b, 0x7632);
}

// Digit i (0 = leading) of X + kDigitBias.
__device__ __forceinline__ int digit(long long u, int i) {
  return i == 0 ? (int)(u >> 49) : (int)((u >> (49 - 7 * i)) & 127) - 64;
}

// Eight values of K of one row (fixed-point, biased) into the 16-byte core
// matrix rows of the eight slices.
__device__ __forceinline__ void put_chunk(char* tile_row, int slice_bytes, const long long* u) {
#pragma unroll
  for (int i = 0; i < kS; ++i) {
    uint4 w;
    w.x = bf16_pair(digit(u[0], i), digit(u[1], i));
    w.y = bf16_pair(digit(u[2], i), digit(u[3], i));
    w.z = bf16_pair(digit(u[4], i), digit(u[5], i));
    w.w = bf16_pair(digit(u[6], i), digit(u[7], i));
    *reinterpret_cast<uint4*>(tile_row + (long)i * slice_bytes) = w;
  }
}

// Byte offset of (row r of the tile, chunk c of 8 values of K) within a row tile.
__device__ __forceinline__ long chunk_off(int RT, int r, int c) {
  return (long)(c >> 1) * (kS * RT * 32) + (r >> 3) * 256 + (c & 1) * 128 + (r & 7) * 16;
}

// Eight rows per block: each warp takes the largest element of a row, then
// the block writes the rows' chunks, eight rows of a chunk (128 contiguous
// bytes per slice) by eight neighbouring lanes.  Bound by memory: 8 bytes in
// (twice, the second time from L2), 16 out per element.
__global__ void __launch_bounds__(256) k_oz_slice_rows(const double* src, long rows, int k, long ld,
                                                       OzOperand o) {
  pdl_begin();
  __shared__ int e_sh[8];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int gpt = (o.rows_per_tile + 7) >> 3;  // groups of eight rows per row tile
  const long rt = blockIdx.x / gpt;
  const int g8 = (int)(blockIdx.x - rt * gpt);
  {
    const int r = 8 * g8 + warp;
    const long gr = rt * o.rows_per_tile + r;
    uint32_t m = 0, any = 0;
    if (r < o.rows_per_tile && gr < rows) {
      const double* p = src + gr * ld;
      for (int c = lane; c < k; c += 32) {
        const double x = p[c];
        m = max(m, abs_hi(x));
        any |= abs_hi(x) | (uint32_t)__double2loint(x);
      }
    }
    m = __reduce_max_sync(0xffffffffu, m);
    any = __reduce_or_sync(0xffffffffu, any);
    const int e = row_exp(m, any != 0);
    if (lane == 0) {
      e_sh[warp] = e;
      if (r < o.rows_per_tile && gr < rows) o.exps[gr] = e;
    }
  }
  __syncthreads();
  const int r = 8 * g8 + (tid & 7);
  const long gr = rt * o.rows_per_tile + r;
  if (r >= o.rows_per_tile || gr >= rows) return;
  const int e = e_sh[tid & 7];
  const bool fine = e != kOzNanExp && e != kOzZeroExp;
  const double* p = src + gr * ld;
  char* base = reinterpret_cast<char*>(o.data) + rt * o.nkb * (long)(kS * o.RT * 32);
  for (int c = tid >> 3; c < 2 * o.nkb; c += 32) {
    long long u[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int kk = 8 * c + i;
      u[i] = kDigitBias + (fine && kk < k ? fixed57(p[kk], e) : 0ll);
    }
    put_chunk(base + chunk_off(o.RT, r, c), o.RT * 32, u);
  }
}

// V / sqrt(dt) = -Im Y + i Re Y of walker blockIdx.y, rows 8 blockIdx.x ..:
// operand rows p = [-Im Y_p | Re Y_p], segments of Mp (zero past M), from the
// packed upper triangle.  The rows' largest element first, then the slices;
// a tile's rows below the diagonal read Y columns, eight rows of a column at
// a time (64 contiguous bytes).
__global__ void __launch_bounds__(256) k_oz_slice_v(const double* Y, long ldy, int M, int Mp, OzOperand o) {
  pdl_begin();
  __shared__ uint32_t m_sh[8], any_sh[8];
  const int tid = threadIdx.x, w = blockIdx.y;
  const int gpt = (o.rows_per_tile + 7) >> 3;
  const int rt = blockIdx.x / gpt, g8 = blockIdx.x - rt * gpt;
  const int r = 8 * g8 + (tid & 7);
  const int p = rt * o.rows_per_tile + r;
  const bool act = r < o.rows_per_tile && p < M;
  const double* yr = Y + (long)w * 2 * ldy;
  const double* yi = yr + ldy;
  if (tid < 8) m_sh[tid] = any_sh[tid] = 0u;
  __syncthreads();
  uint32_t m = 0, any = 0;
  if (act)
    for (int q = tid >> 3; q < M; q += 32) {
      const int a = q <= p ? q : p, b = q <= p ? p : q;
      const long id = (long)a * M - (long)a * (a - 1) / 2 + (b - a);
      const double vr = yi[id], vi = yr[id];
      m = max(m, max(abs_hi(vr), abs_hi(vi)));
      any |= abs_hi(vr) | (uint32_t)__double2loint(vr) | abs_hi(vi) | (uint32_t)__double2loint(vi);
    }
  if (m | any) {
    atomicMax(&m_sh[tid & 7], m);
    atomicOr(&any_sh[tid & 7], any);
  }
  __syncthreads();
  if (!act) return;
  const int e = row_exp(m_sh[tid & 7], any_sh[tid & 7] != 0);
  if (tid < 8) o.exps[(long)w * o.batch_exp_stride + p] = e;
  const bool fine = e != kOzNanExp && e != kOzZeroExp;
  char* base = reinterpret_cast<char*>(o.data) + (long)w * o.batch_stride +
               (long)rt * o.nkb * (long)(kS * o.RT * 32);
  for (int c = tid >> 3; c < Mp / 8; c += 32) {
    long long ur[8], ui[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int q = 8 * c + i;
      ur[i] = ui[i] = kDigitBias;
      if (fine && q < M) {
        const int a = q <= p ? q : p, b = q <= p ? p : q;
        const long id = (long)a * M - (long)a * (a - 1) / 2 + (b - a);
        ur[i] -= fixed57(yi[id], e);
        ui[i] += fixed57(yr[id], e);
      }
    }
    put_chunk(base + chunk_off(o.RT, r, c), o.RT * 32, ur);
    put_chunk(base + chunk_off(o.RT, r, Mp / 8 + c), o.RT * 32, ui);
  }
}

// A Taylor term [2][N][M] of walker blockIdx.y as operand rows i = [Re T_i |
// -Im T_i] and N + i = [Im T_i | Re T_i] (segments of Mp), so that the rows
// [Re | Im] of V times them give Re and Im of V T.  Eight orbitals per block, a
// warp each for the largest element; then eight neighbouring lanes write the
// eight orbitals' rows of a chunk (128 contiguous bytes per slice where the
// rows share a group of eight).
__global__ void __launch_bounds__(256) k_oz_slice_term(const double* t, int N, int M, int Mp,
                                                       OzOperand o) {
  pdl_begin();
  __shared__ int e_sh[8];
  const int tid = threadIdx.x, lane = tid & 31, w = blockIdx.y;
  const double* tw = t + (long)w * 2 * N * M;
  {
    const int i = blockIdx.x * 8 + (tid >> 5);
    uint32_t m = 0, any = 0;
    if (i < N) {
      const double* tr = tw + (long)i * M;
      const double* ti = tr + (long)N * M;
      for (int p = lane; p < M; p += 32) {
        const double x = tr[p], y = ti[p];
        m = max(m, max(abs_hi(x), abs_hi(y)));
        any |= abs_hi(x) | (uint32_t)__double2loint(x) | abs_hi(y) | (uint32_t)__double2loint(y);
      }
    }
    m = __reduce_max_sync(0xffffffffu, m);
    any = __reduce_or_sync(0xffffffffu, any);
    const int e = row_exp(m, any != 0);
    if (lane == 0) {
      e_sh[tid >> 5] = e;
      if (i < N) {
        int* ex = o.exps + (long)w * o.batch_exp_stride;
        ex[i] = ex[N + i] = e;
      }
    }
  }
  __syncthreads();
  const int i = blockIdx.x * 8 + (tid & 7);
  if (i >= N) return;
  const int e = e_sh[tid & 7];
  const bool fine = e != kOzNanExp && e != kOzZeroExp;
  const double* tr = tw + (long)i * M;
  const double* ti = tr + (long)N * M;
  const int rpt = o.rows_per_tile, nc = Mp / 8;
  const long tile_stride = (long)o.nkb * (kS * o.RT * 32);
  char* base = reinterpret_cast<char*>(o.data) + (long)w * o.batch_stride;
  char* re_row = base + (i / rpt) * tile_stride;
  char* im_row = base + ((N + i) / rpt) * tile_stride;
  const int r0 = i % rpt, r1 = (N + i) % rpt;
  // the real and the imaginary part of a chunk are separate items
  for (int c2 = tid >> 3; c2 < 2 * nc; c2 += 32) {
    const bool im = c2 >= nc;
    const int c = im ? c2 - nc : c2;
    const double* src = im ? ti : tr;
    long long u[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int p = 8 * c + j;
      u[j] = fine && p < M ? fixed57(src[p], e) : 0ll;
    }
    long long up[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) up[j] = kDigitBias + u[j];
    if (!im) {
      put_chunk(re_row + chunk_off(o.RT, r0, c), o.RT * 32, up);
      put_chunk(im_row + chunk_off(o.RT, r1, nc + c), o.RT * 32, up);
    } else {
      put_chunk(im_row + chunk_off(o.RT, r1, c), o.RT * 32, up);
#pragma unroll
      for (int j = 0; j < 8; ++j) up[j] = kDigitBias - u[j];
      put_chunk(re_row + chunk_off(o.RT, r0, nc + c), o.RT * 32, up);
    }
  }
}

// Exponents of n rows of M values (as k_oz_slice_rows leaves them), four rows per
// warp so that enough loads are in flight.  Bound by memory: 20480 rows of 100
// 6.5 us (10.3 with a row per warp).
__global__ void __launch_bounds__(256) k_oz_row_exps(const double* src, long n, int M, int* exps) {
  pdl_begin();
  const long t0 = 4 * ((long)blockIdx.x * 8 + (threadIdx.x >> 5));
  const int lane = threadIdx.x & 31;
  int e[4] = {kOzZeroExp, kOzZeroExp, kOzZeroExp, kOzZeroExp};
  for (int p = lane; p < M; p += 32) {
    double x[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) x[r] = t0 + r < n ? src[(t0 + r) * M + p] : 0.0;
#pragma unroll
    for (int r = 0; r < 4; ++r) e[r] = max(e[r], elem_exp(x[r], 0));
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) e[r] = __reduce_max_sync(0xffffffffu, e[r]);
  if (lane < 4 && t0 + lane < n) exps[t0 + lane] = lane == 0 ? e[0] : lane == 1 ? e[1] : lane == 2 ? e[2] : e[3];
}

// Exponent of orbital i of a walker from those of its 2 N planes; none for an
// orbital of zeros, or one that is not finite.  Rows that run over a walker's
// orbitals are sliced with every orbital divided by 2^s and the other operand's
// row i multiplied by it: orbitals of very different norm would otherwise share
// the largest one's exponent and lose the bits that the inverse's small and large
// rows need.
__device__ __forceinline__ int orbital_exp(const int* planes, int N, int i) {
  const int e = max(planes[i], planes[N + i]);
  return e == kOzZeroExp || e == kOzNanExp ? 0 : e;
}

// Rows p = [Re Phi_p | Im Phi_p] of walker blockIdx.y, orbitals scaled by their
// exponents: K runs over the 2 N orbital planes, a lane owns a row, so both the
// reads along p and the writes (eight rows of a chunk: 128 contiguous bytes per
// slice) are contiguous.  1024 walkers, M = 100, N = 10 23 us; 512, M = 300, N = 25
// 47 us (20 and 44 with one scale for all orbitals).
__global__ void __launch_bounds__(256) k_oz_slice_cols(const double* phi, int N, int M, const int* planes,
                                                       OzOperand o) {
  pdl_begin();
  __shared__ int e_sh[8][32], s_sh[64];
  const int lane = threadIdx.x & 31, wk = threadIdx.x >> 5, w = blockIdx.y, N2 = 2 * N;
  const int p = blockIdx.x * 32 + lane;
  const double* src = phi + (long)w * N2 * M + p;
  // the first values are on their way while the exponents arrive
  double x[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) x[j] = p < M && wk + 8 * j < N2 ? src[(long)(wk + 8 * j) * M] : 0.0;
  if (threadIdx.x < N) s_sh[threadIdx.x] = orbital_exp(planes + (long)w * N2, N, threadIdx.x);
  __syncthreads();
  int e = kOzZeroExp;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int k = wk + 8 * j;
    if (k < N2) e = max(e, elem_exp(x[j], s_sh[k < N ? k : k - N]));
  }
  if (p < M)
    for (int k = wk + 64; k < N2; k += 8) e = max(e, elem_exp(src[(long)k * M], s_sh[k < N ? k : k - N]));
  e_sh[wk][lane] = e;
  __syncthreads();
  if (p >= M) return;
#pragma unroll
  for (int q = 0; q < 8; ++q) e = max(e, e_sh[q][lane]);
  const bool fine = e != kOzNanExp && e != kOzZeroExp;
  if (wk == 0) o.exps[(long)w * o.batch_exp_stride + p] = e;
  const int rt = p / o.rows_per_tile, r = p - rt * o.rows_per_tile;
  char* base = reinterpret_cast<char*>(o.data) + (long)w * o.batch_stride +
               (long)rt * o.nkb * (kS * o.RT * 32);
  for (int c = wk; c < 2 * o.nkb; c += 8) {
    long long u[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int k = 8 * c + i;
      u[i] = kDigitBias + (fine && k < N2 ? fixed57(src[(long)k * M], e + s_sh[k < N ? k : k - N]) : 0ll);
    }
    put_chunk(base + chunk_off(o.RT, r, c), o.RT * 32, u);
  }
}

// Rows of the density sums (oz_slice_densities): group blockIdx.y of cw
// walkers, whose K values (w, c, i) of a column p lie M apart; blockIdx.z: Phi
// as it is, Phi times i, thA, thB.  A lane owns a row as in k_oz_slice_cols, and
// the orbitals of Phi are scaled down and Theta's up by their exponents as there
// (planes: of the walkers from w0 on): a row runs over walkers whose orbitals' norms may differ widely.
__global__ void __launch_bounds__(256) k_oz_slice_densities(const double* phi, const double* thA,
                                                            const double* thB, int W, int N, int M, int w0,
                                                            int cw, const int* planes, OzOperand A, OzOperand B) {
  pdl_begin();
  __shared__ int e_sh[8][32], s_sh[kOzSegK / 2];  // K = 2 N cw of at most one segment
  const int lane = threadIdx.x & 31, wk = threadIdx.x >> 5, z = blockIdx.y, which = blockIdx.z;
  const int p = blockIdx.x * 32 + lane, first = w0 + z * cw, N2 = 2 * N;
  const int nk = (W - first < cw ? W - first : cw) * N2;
  const OzOperand& o = which < 2 ? A : B;
  const double* src = (which < 2 ? phi : which == 2 ? thA : thB) + (long)first * N2 * M + p;
  for (int t = threadIdx.x; t < nk / 2; t += 256) {
    const int s = orbital_exp(planes + ((long)z * cw + t / N) * N2, N, t % N);
    s_sh[t] = which < 2 ? s : -s;
  }
  __syncthreads();
  auto shift = [&](int k) { return s_sh[k / N2 * N + k % N]; };
  int e = kOzZeroExp;
  if (p < M)
#pragma unroll 4
    for (int k = wk; k < nk; k += 8) e = max(e, elem_exp(src[(long)k * M], shift(k)));
  e_sh[wk][lane] = e;
  __syncthreads();
  if (p >= M) return;
#pragma unroll
  for (int q = 0; q < 8; ++q) e = max(e, e_sh[q][lane]);
  const bool fine = e != kOzNanExp && e != kOzZeroExp;
  const int row = (which & 1) * M + p, rt = row / o.rows_per_tile, r = row - rt * o.rows_per_tile;
  if (wk == 0) o.exps[(long)z * o.batch_exp_stride + row] = e;
  char* base = reinterpret_cast<char*>(o.data) + (long)z * o.batch_stride + (long)rt * o.nkb * (kS * o.RT * 32);
  for (int c = wk; c < 2 * o.nkb; c += 8) {
    long long u[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int k = 8 * c + i;
      long long v = 0;
      if (fine && k < nk) {
        if (which == 1) {  // (re, im) <- (-im, re)
          const bool re = k % N2 < N;
          v = fixed57(src[(long)(re ? k + N : k - N) * M], e + shift(k));
          if (re) v = -v;
        } else {
          v = fixed57(src[(long)k * M], e + shift(k));
        }
      }
      u[i] = kDigitBias + v;
    }
    put_chunk(base + chunk_off(o.RT, r, c), o.RT * 32, u);
  }
}

// The inverse of (ds, w) = (blockIdx.y, blockIdx.x) as operand rows (re, j) =
// [Re S^-1_j | -Im S^-1_j] and (im, j) = [Im S^-1_j | Re S^-1_j], S^-1_j column j
// with row i scaled by the exponent of orbital i (planes: of Phi, walker by walker).
__global__ void __launch_bounds__(256) k_oz_slice_inverse(const double2* sinv, int W, int w0, int N,
                                                          const int* planes, OzOperand o) {
  pdl_begin();
  __shared__ int e_sh[64], s_sh[64];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int w = blockIdx.x, ds = blockIdx.y;
  const long batch = (long)ds * gridDim.x + w;
  const double2* S = sinv + ((long)ds * W + w0 + w) * N * N;
  int* ex = o.exps + batch * o.batch_exp_stride;
  if (threadIdx.x < N) s_sh[threadIdx.x] = -orbital_exp(planes + (long)w * 2 * N, N, threadIdx.x);
  __syncthreads();
  for (int j = warp; j < N; j += 8) {
    int e = kOzZeroExp;
    for (int i = lane; i < N; i += 32) {
      const double2 x = S[i * N + j];
      e = max(e, max(elem_exp(x.x, s_sh[i]), elem_exp(x.y, s_sh[i])));
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) {
      e_sh[j] = e;
      ex[j] = ex[N + j] = e;
    }
  }
  __syncthreads();
  const int rows8 = (2 * N + 7) / 8 * 8;
  const long tile_stride = (long)o.nkb * (kS * o.RT * 32);
  char* base = reinterpret_cast<char*>(o.data) + batch * o.batch_stride;
  for (int it = threadIdx.x; it < rows8 * 2 * o.nkb; it += 256) {
    const int row = it % rows8, c = it / rows8;
    if (row >= 2 * N) continue;
    const int im = row >= N ? 1 : 0, j = row - im * N, e = e_sh[j];
    const bool fine = e != kOzNanExp && e != kOzZeroExp;
    long long u[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int k = 8 * c + i;
      u[i] = kDigitBias;
      if (fine && k < 2 * N) {
        const int part = k >= N ? 1 : 0, q = k - part * N;
        const double2 x = S[q * N + j];
        const long long f = fixed57(im == part ? x.x : x.y, e + s_sh[q]);
        u[i] += (im == 0 && part == 1) ? -f : f;
      }
    }
    put_chunk(base + (row / o.rows_per_tile) * tile_stride + chunk_off(o.RT, row % o.rows_per_tile, c),
              o.RT * 32, u);
  }
}

// ------------------------------------------------------------ contraction ---
// (hi 2^28 + lo) 2^e as float64, rounded to nearest even once.
__device__ __forceinline__ double round_sum(long long hi, long long lo, int e) {
  long long h = hi + (lo >> 28);
  uint32_t l = (uint32_t)lo & 0xfffffffu;
  const bool neg = h < 0;
  if (neg) {  // negate the pair
    l = (0x10000000u - l) & 0xfffffffu;
    h = ~h + (l == 0 ? 1 : 0);
  }
  unsigned long long x;  // leading bit at 63
  int top;               // weight of the leading bit
  uint32_t lost = 0;
  if (h != 0) {
    const int z = __clzll(h);
    x = (unsigned long long)h << z;
    if (z >= 28) {
      x |= (unsigned long long)l << (z - 28);
    } else {
      x |= l >> (28 - z);
      lost = l & ((1u << (28 - z)) - 1u);
    }
    top = 63 - z + 28;
  } else {
    if (l == 0) return 0.0;
    const int z = __clzll((long long)l);
    x = (unsigned long long)l << z;
    top = 63 - z;
  }
  unsigned long long man = x >> 11;
  const uint32_t rest = (uint32_t)x & 2047u;
  if (rest > 1024u || (rest == 1024u && (lost != 0 || (man & 1ull)))) ++man;  // may carry to 2^53
  const int E = top + e;
  const unsigned long long sign = neg ? 1ull << 63 : 0ull;
  if (E > -1022 && E < 1023)
    return __longlong_as_double((long long)(sign | (((unsigned long long)(E + 1022) << 52) + man)));
  const double d = __longlong_as_double((long long)(sign | ((1022ull << 52) + man)));  // E = 0
  return scalbn(d, E < -4000 ? -4000 : (E > 4000 ? 4000 : E));
}

// The same for row exponents ea, eb; a row with an infinity or a NaN gives NaN
// (its exponent is above any sum of two ordinary ones).
__device__ __forceinline__ double scaled_sum(long long hi, long long lo, int e) {
  return e > kOzNanExp / 2 ? __longlong_as_double(0x7ff8000000000000ll) : round_sum(hi, lo, e - 63);
}

__device__ __forceinline__ void tmem_ld8_async(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7])
      : "r"(taddr));
}

// Contiguous global -> shared copy, completing on an mbarrier.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// Shared-memory matrix descriptor of a K-major operand in core matrices of 8
// rows x 16 bytes (no swizzle): 128 bytes between the two core matrices of a
// K step, 256 bytes between groups of eight rows.
__device__ __forceinline__ uint64_t core_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)(128 >> 4) << 16;
  d |= (uint64_t)(256 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

struct OzArgs {
  const char* A;
  const char* B;
  long a_batch, b_batch;    // bytes
  const int* ea;
  const int* eb;
  long ea_batch, eb_batch;  // rows
  int a_rpt, b_rpt;         // rows of a tile that are operand rows
  int a_bytes;              // bytes of an A tile's K block
  int RTA;
  int nkb, nseg;
  int nmt, nnt, ntiles;     // tiles = batch x nnt x nmt, mt fastest
  int a_mod;                // batch entry b reads A of entry b % a_mod
  int* err;
};

// Shared memory: a ring of STAGES K blocks (A tile of up to 128 rows, then the
// B tile), the epilogue's buffer, the barriers.  (With RTA < 128 the M = 128
// rows of a slice run into the next one's; the rows past RTA are dropped.)
template <int BN, class Epi>
struct OzSmem {
  static constexpr int STAGE = kS * 32 * (BM + BN);
  static constexpr int STAGES = Epi::kStages;
  static constexpr int EPI = STAGES * STAGE;
  static constexpr int BAR = EPI + Epi::kSmemBytes;
  static constexpr int TOTAL = BAR + 256 + 1024;
};

// Epilogue warps: four per TMEM lane quarter (two for the narrowest tile).
// With two per quarter the drain and the epilogue, a chain of dependent
// integer operations per value, took as long as 25 K blocks of MMAs.
template <int BN>
constexpr int kOzEpiWarps = BN >= 32 ? 16 : 8;
template <int BN>
constexpr int kOzThreads = 64 + 32 * kOzEpiWarps<BN>;

// What an epilogue knows about its tile and thread.
struct OzTile {
  int b, mt, nt;  // batch entry, row and column tile
  int r, c0;      // this thread's row of the tile, first of its warp's columns
  int lane, ew;
};

// An epilogue's reads for a thread's row and its warp's CW columns: the sums of
// the row exponents, whether the row is stored, earlier values (narrow tiles).
template <int CW>
struct OzPre {
  int e[CW];
  bool on;
  double old[CW <= 8 ? CW : 1];
};

// D_t .. D_{t+3} of eight columns as D_t 2^21 + D_{t+1} 2^14 + D_{t+2} 2^7 +
// D_{t+3}; the pairs stay below 2^31.
template <int BN>
__device__ __forceinline__ void drain4(uint32_t base, int t, long long* sum) {
  int p[8];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t r0[8], r1[8];
    tmem_ld8_async(base + (uint32_t)((t + 2 * h) * BN), r0);
    tmem_ld8_async(base + (uint32_t)((t + 2 * h + 1) * BN), r1);
    tmem_ld_wait();
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const int q = __float2int_rn(__uint_as_float(r0[c])) * 128 + __float2int_rn(__uint_as_float(r1[c]));
      if (h == 0)
        p[c] = q;
      else
        sum[c] += (long long)p[c] * 16384 + q;
    }
  }
}

// Persistent contraction: one CTA per SM walks 128 x BN tiles.  Warp 0 copies
// the operands' K blocks (16 values of K, all eight slices: contiguous in
// memory) into the ring; one thread of warp 1 multiplies: slice i of A against
// slices 0 .. 7 - i of B, which lie side by side as (8 - i) BN columns, into
// the accumulator columns of D_i .. D_7, so that one instruction covers several
// slice pairs and every A slice is read once per 256 columns.  36 of 64 pairs.
// The epilogue warps drain the accumulators after every kOzSegBlk blocks
// (MULTI: 64-bit sums kept in registers) and hand the sums to the epilogue.
// BN = 64 fills tensor memory with one set of accumulators; narrower tiles
// have two, so that the epilogue overlaps the next segment.
// Bound by the tensor pipe at large K: 36 x 64 columns take 1152 cycles per
// K block against 48 KB of operands from L2 (43 B per cycle).
template <int BN, class Epi, bool MULTI>
__global__ void __launch_bounds__(kOzThreads<BN>, 1)
    k_oz_gemm(const OzArgs g, const __grid_constant__ Epi epi) {
  extern __shared__ uint8_t oz_raw[];
  using S = OzSmem<BN, Epi>;
  constexpr int EW = kOzEpiWarps<BN>;
  constexpr int STAGES = S::STAGES;
  constexpr int NBUF = BN <= 32 ? 2 : 1;
  constexpr uint32_t DCOLS = kS * BN;
  constexpr uint32_t TCOLS = NBUF * DCOLS;
  constexpr int CW = 4 * BN / EW;  // columns per epilogue warp
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(oz_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + S::BAR);
  uint64_t* empty = full + STAGES;
  uint64_t* tfull = empty + STAGES;  // [2]
  uint64_t* tempty = tfull + 2;      // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty + 2);
  int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&tfull[a], 1);
      mbar_init(&tempty[a], EW);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(TCOLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;
  const int per_batch = g.nmt * g.nnt;
  constexpr int B_BYTES = kS * BN * 32;

  if (warp == 0 && lane == 0) {
    int it = 0;
    for (int t = blockIdx.x; t < g.ntiles && !*(volatile int*)abort_flag; t += gridDim.x) {
      const int b = t / per_batch, rem = t - b * per_batch, nt = rem / g.nmt, mt = rem - nt * g.nmt;
      const char* a_src = g.A + (b % g.a_mod) * g.a_batch + (long)mt * g.nkb * g.a_bytes;
      const char* b_src = g.B + b * g.b_batch + (long)nt * g.nkb * B_BYTES;
      for (int kb = 0; kb < g.nkb; ++kb, ++it) {
        const int s = it % STAGES;
        if (it >= STAGES && !mbar_wait(&empty[s], ((it / STAGES) - 1) & 1, g.err, 61)) {
          *(volatile int*)abort_flag = 1;
          break;
        }
        uint8_t* dst = smem + s * S::STAGE;
        mbar_expect_tx(&full[s], (uint32_t)(g.a_bytes + B_BYTES));
        bulk_load(dst, a_src + (long)kb * g.a_bytes, (uint32_t)g.a_bytes, &full[s]);
        bulk_load(dst + kS * 32 * BM, b_src + (long)kb * B_BYTES, (uint32_t)B_BYTES, &full[s]);
      }
    }
    // given up: no copy may still be in flight when the CTA's memory is released
    if (*(volatile int*)abort_flag)
      for (int n = it > STAGES ? it - STAGES : 0; n < it; ++n)
        mbar_wait(&full[n % STAGES], (n / STAGES) & 1, g.err, 65);
  } else if (warp == 1 && lane == 0) {
    int it = 0, j = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < g.ntiles && ok && !*(volatile int*)abort_flag; t += gridDim.x) {
      int kb = 0;
      for (int sg = 0; sg < g.nseg && ok; ++sg, ++j) {
        const int kend = (int)((long)g.nkb * (sg + 1) / g.nseg);
        const int buf = NBUF == 2 ? (j & 1) : 0;
        if (j >= NBUF && !mbar_wait(&tempty[buf], ((j / NBUF) - 1) & 1, g.err, 62)) {
          ok = false;
          break;
        }
        fence_after();
        const uint32_t d = tmem + (uint32_t)buf * DCOLS;
        for (bool first = true; kb < kend; ++kb, ++it, first = false) {
          const int s = it % STAGES;
          if (!mbar_wait(&full[s], (it / STAGES) & 1, g.err, 63)) {
            ok = false;
            break;
          }
          fence_after();
          const uint32_t a = smem_u32(smem + s * S::STAGE);
          const uint32_t bb = a + kS * 32 * BM;
#pragma unroll
          for (int i = 0; i < kS; ++i) {
            const uint64_t ad = core_desc(a + (uint32_t)(i * g.RTA * 32));
            constexpr int kMaxN = 256;
#pragma unroll
            for (int c = 0; c < (kS - i) * BN; c += kMaxN) {
              const int n = (kS - i) * BN - c < kMaxN ? (kS - i) * BN - c : kMaxN;
              mma<false>(d + (uint32_t)(i * BN + c), ad, core_desc(bb + (uint32_t)(c * 32)),
                         instr_desc(1u, (uint32_t)n), (first && i == 0) ? 0u : 1u);
            }
          }
          mma_commit(&empty[s]);
        }
        mma_commit(&tfull[buf]);
      }
    }
    if (!ok) *(volatile int*)abort_flag = 1;
  } else if (warp >= 2) {
    const int q = warp & 3;
    OzTile tl;
    tl.lane = lane;
    tl.ew = warp - 2;
    tl.r = 32 * q + lane;
    tl.c0 = CW * (tl.ew >> 2);
    int j = 0;
    for (int t = blockIdx.x; t < g.ntiles; t += gridDim.x) {
      const int b = t / per_batch, rem = t - b * per_batch, nt = rem / g.nmt, mt = rem - nt * g.nmt;
      tl.b = b;
      tl.mt = mt;
      tl.nt = nt;
      long long hi[MULTI ? CW : 8], lo[MULTI ? CW : 8];
#pragma unroll
      for (int c = 0; c < (MULTI ? CW : 8); ++c) hi[c] = lo[c] = 0;
      // what the epilogue reads from memory, in flight during the products
      OzPre<CW> pre;
      epi.pre(g, tl, pre);
      bool stop = false;
      for (int sg = 0; sg < (MULTI ? g.nseg : 1); ++sg, ++j) {
        const int buf = NBUF == 2 ? (j & 1) : 0;
        const bool bad = !mbar_wait_sleep(&tfull[buf], (j / NBUF) & 1, g.err, 64);
        fence_after();
        uint32_t out;
        asm volatile(
            "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %1, 0;\n\t"
            "bar.red.or.pred p, 1, %2, q;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(out)
            : "r"((uint32_t)(bad || *(volatile int*)abort_flag)), "n"(32 * EW)
            : "memory");
        if (out) {
          *(volatile int*)abort_flag = 1;
          stop = true;
          break;
        }
        const uint32_t base = tmem + (uint32_t)buf * DCOLS + ((uint32_t)(32 * q) << 16) + (uint32_t)tl.c0;
#pragma unroll
        for (int c0 = 0; c0 < CW; c0 += 8) {
          if constexpr (MULTI) {
            drain4<BN>(base + (uint32_t)c0, 0, hi + c0);
            drain4<BN>(base + (uint32_t)c0, 4, lo + c0);
          } else {
#pragma unroll
            for (int c = 0; c < 8; ++c) hi[c] = lo[c] = 0;
            drain4<BN>(base + (uint32_t)c0, 0, hi);
            drain4<BN>(base + (uint32_t)c0, 4, lo);
            epi.chunk(g, tl, c0, hi, lo, pre, smem + S::EPI);
            __syncwarp();  // the next TMEM loads need the whole warp
          }
        }
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&tempty[buf]);
      }
      if (stop) break;
      if constexpr (MULTI) {
#pragma unroll
        for (int c0 = 0; c0 < CW; c0 += 8) epi.chunk(g, tl, c0, hi + c0, lo + c0, pre, smem + S::EPI);
      }
      epi.template finish<EW>(g, tl, smem + S::EPI);
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 1) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TCOLS));
  }
}

// -------------------------------------------------------------- epilogues ---
// pre(): reads that do not depend on the products; chunk(): eight columns from
// the warp's column c0 on, row tl.r.
// C[m][n] = 2^alpha D: each warp passes its 32 rows x 8 columns through 2 KB
// of shared memory so that a store instruction covers four rows of 64 bytes.
struct EpiOzStore {
  static constexpr int kStages = 4;
  static constexpr int kSmemBytes = 16 * 32 * 8 * 8;
  double* C;
  long ldc, c_batch;
  int M, N, alpha;
  const double* mask;
  int mask_rows;
  template <int CW>
  __device__ __forceinline__ void pre(const OzArgs& g, const OzTile& tl, OzPre<CW>& q) const {
    const int row = tl.mt * g.a_rpt + tl.r, col = tl.nt * g.b_rpt + tl.c0;
    const int ea = (row < M ? g.ea[(long)tl.b * g.ea_batch + row] : kOzZeroExp) + alpha;
    const int* eb = g.eb + (long)tl.b * g.eb_batch;
#pragma unroll
    for (int c = 0; c < CW; ++c) q.e[c] = ea + (col + c < N ? eb[col + c] : kOzZeroExp);
  }
  template <int CW>
  __device__ __forceinline__ void chunk(const OzArgs& g, const OzTile& tl, int c0, const long long* hi,
                                        const long long* lo, const OzPre<CW>& q, uint8_t* sm) const {
    double* buf = reinterpret_cast<double*>(sm) + tl.ew * 256;
    const int lane = tl.lane, row = tl.mt * g.a_rpt + tl.r, col = tl.nt * g.b_rpt + tl.c0 + c0;
#pragma unroll
    for (int i = 0; i < 8; ++i)
      // 16-byte slots permuted by row: row-per-lane writes without conflicts
      buf[lane * 8 + ((i & 1) | (((i >> 1) ^ (lane & 3)) << 1))] = scaled_sum(hi[i], lo[i], q.e[c0 + i]);
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int rr = 4 * k + (lane >> 3), i = lane & 7;
      const int grow = row - lane + rr, gcol = col + i;
      if (tl.r - lane + rr < g.a_rpt && grow < M && gcol < N && (!mask || walker_alive(mask, grow / mask_rows)))
        C[(long)tl.b * c_batch + (long)grow * ldc + gcol] =
            buf[rr * 8 + ((i & 1) | (((i >> 1) ^ (rr & 3)) << 1))];
    }
    __syncwarp();
  }
  template <int EW>
  __device__ __forceinline__ void finish(const OzArgs&, const OzTile&, uint8_t*) const {}
};

// A Taylor term: rows p, columns (c, i) of walker b.  A lane owns a row, so
// the accesses along p are contiguous; the running sum is read ahead (narrow
// tiles) or before the values are formed.
struct EpiOzTerm {
  static constexpr int kStages = 4;
  static constexpr int kSmemBytes = 0;
  int M, N2;  // N2 = 2 N
  int first, last;
  double scale;  // sqrt(dt) / k
  const double* tin;
  double* tout;
  double* acc;
  template <int CW>
  __device__ __forceinline__ void pre(const OzArgs& g, const OzTile& tl, OzPre<CW>& q) const {
    const int p = tl.mt * g.a_rpt + tl.r, col = tl.nt * g.b_rpt + tl.c0;
    q.on = tl.r < g.a_rpt && p < M && col < N2;
    const int ea = q.on ? g.ea[(long)tl.b * g.ea_batch + p] : kOzZeroExp;
    const int* eb = g.eb + (long)tl.b * g.eb_batch + col;
#pragma unroll
    for (int c = 0; c < CW; ++c) q.e[c] = q.on && col + c < N2 ? ea + eb[c] : kOzZeroExp;
    if constexpr (CW <= 8) {
      const double* src = (first ? tin : acc) + ((long)tl.b * N2 + col) * M + p;
#pragma unroll
      for (int c = 0; c < CW; ++c) q.old[c] = q.on && col + c < N2 ? src[(long)c * M] : 0.0;
    }
  }
  template <int CW>
  __device__ __forceinline__ void chunk(const OzArgs& g, const OzTile& tl, int c0, const long long* hi,
                                        const long long* lo, const OzPre<CW>& q, uint8_t*) const {
    const int p = tl.mt * g.a_rpt + tl.r, col = tl.nt * g.b_rpt + tl.c0 + c0;
    if (!q.on || col >= N2) return;
    const long at = ((long)tl.b * N2 + col) * M + p;
    double old[8], v[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      if constexpr (CW <= 8)
        old[c] = q.old[c];
      else
        old[c] = col + c < N2 ? ((first ? tin : acc) + at)[(long)c * M] : 0.0;
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) v[c] = scaled_sum(hi[c], lo[c], q.e[c0 + c]) * scale;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      if (col + c >= N2) break;
      if (!last) tout[at + (long)c * M] = v[c];
      acc[at + (long)c * M] = old[c] + v[c];
    }
  }
  template <int EW>
  __device__ __forceinline__ void finish(const OzArgs&, const OzTile&, uint8_t*) const {}
};

// Theta rows: like a Taylor term's, batch entry b = (ds, w).
struct EpiOzTheta {
  static constexpr int kStages = 4;
  static constexpr int kSmemBytes = 0;
  OzTheta t;
  template <int CW>
  __device__ __forceinline__ void pre(const OzArgs& g, const OzTile& tl, OzPre<CW>& q) const {
    const int p = tl.mt * g.a_rpt + tl.r, col = tl.nt * g.b_rpt + tl.c0, N2 = 2 * t.N;
    const int ds = tl.b / t.nw, wl = tl.b - ds * t.nw, w = t.w0 + wl;
    // the three conditions' loads are independent
    const bool ok = t.flag ? t.flag[w] != 0 : t.ld[(long)w * t.ld_w + (long)ds * t.ld_ds] > -INFINITY;
    const bool alive = !t.wt || walker_alive(t.wt, w);
    q.on = tl.r < g.a_rpt && p < t.M && col < N2 && alive && (ok || t.zero_singular);
    const int ea = q.on ? g.ea[(long)wl * g.ea_batch + p] : kOzZeroExp;
    const int* eb = g.eb + (long)tl.b * g.eb_batch + col;
    // (a row of zeros gives zeros whatever the sums: singular walkers)
#pragma unroll
    for (int c = 0; c < CW; ++c) q.e[c] = q.on && ok && col + c < N2 ? ea + eb[c] : kSkip;
  }
  static constexpr int kSkip = -(1 << 28);
  template <int CW>
  __device__ __forceinline__ void chunk(const OzArgs& g, const OzTile& tl, int c0, const long long* hi,
                                        const long long* lo, const OzPre<CW>& q, uint8_t*) const {
    const int p = tl.mt * g.a_rpt + tl.r, col = tl.nt * g.b_rpt + tl.c0 + c0, N2 = 2 * t.N;
    if (!q.on || col >= N2) return;
    const int ds = tl.b / t.nw, w = t.w0 + tl.b - ds * t.nw;
    const long row = ((long)ds * t.W + w) * N2 + col;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      if (col + c >= N2) break;
      double v = q.e[c0 + c] != kSkip ? scaled_sum(hi[c], lo[c], q.e[c0 + c]) : 0.0;
      if (t.unit && p < t.N) v = col + c == p ? 1.0 : 0.0;
      t.theta[(row + c) * t.M + p] = v;
      if (t.th_lo) store_lo(t.th_lo, t.lo_kind, (row + c) * t.Mp + p, v);
    }
  }
  template <int EW>
  __device__ __forceinline__ void finish(const OzArgs&, const OzTile&, uint8_t*) const {}
};

// Products of a walker's rows with each other (2 N x 2 N per batch entry).
struct EpiOzGram {
  static constexpr int kStages = 4;
  static constexpr int kSmemBytes = 0;
  int N2;
  double* gram;
  template <int CW>
  __device__ __forceinline__ void pre(const OzArgs& g, const OzTile& tl, OzPre<CW>& q) const {
    const int* e = g.ea + (long)tl.b * g.ea_batch;
    q.on = tl.r < N2;
    const int ea = q.on ? e[tl.r] : 0;
#pragma unroll
    for (int c = 0; c < CW; ++c) q.e[c] = ea + (tl.c0 + c < N2 ? e[tl.c0 + c] : 0);
  }
  template <int CW>
  __device__ __forceinline__ void chunk(const OzArgs&, const OzTile& tl, int c0, const long long* hi,
                                        const long long* lo, const OzPre<CW>& q, uint8_t*) const {
    const int cc = tl.c0 + c0;
    if (!q.on || cc >= N2) return;
    double* out = gram + ((long)tl.b * N2 + tl.r) * N2 + cc;
#pragma unroll
    for (int c = 0; c < 8; ++c)
      if (cc + c < N2) out[c] = scaled_sum(hi[c], lo[c], q.e[c0 + c]);
  }
  template <int EW>
  __device__ __forceinline__ void finish(const OzArgs&, const OzTile&, uint8_t*) const {}
};

// Exchange (M = 100, N = 10, 1024 walkers: 1.19 ms for 14364 tiles, 24 k cycles
// a tile, the drain, conversion and traces against 8 k of products; holding the
// sums in registers so that the next products start earlier spilled and
// measured 1.48 ms).  The tile of T into shared memory, then sum_ij T_ij T_ji per walker
// of the tile over the tile's vectors; every unordered pair {i, j} once, at
// twice its weight (j = i + d mod N), by the lane of row (g, i); nw warps per
// walker, their sums added in a fixed order.
struct EpiOzExchange {
  static constexpr int kStages = 3;
  static constexpr int LD = 65;
  static constexpr int kSmemBytes = BM * LD * 8 + 2 * 16 * 8;
  int N, W, G, RG, WT, nup, nchunk;  // RG vectors, WT walkers per tile
  double* part;
  template <int CW>
  __device__ __forceinline__ void pre(const OzArgs& g, const OzTile& tl, OzPre<CW>& q) const {
    const int row = tl.mt * g.a_rpt + tl.r, col = tl.nt * g.b_rpt + tl.c0;
    q.on = tl.r < g.a_rpt && row < G * N;
    const int ea = q.on ? g.ea[row] : 0;
#pragma unroll
    for (int c = 0; c < CW; ++c)
      q.e[c] = ea + (q.on && tl.c0 + c < g.b_rpt && col + c < 2 * N * W ? g.eb[col + c] : kOff);
  }
  static constexpr int kOff = -(1 << 28);  // no element there: T is zero
  template <int CW>
  __device__ __forceinline__ void chunk(const OzArgs&, const OzTile& tl, int c0, const long long* hi,
                                        const long long* lo, const OzPre<CW>& q, uint8_t* sm) const {
    double* T = reinterpret_cast<double*>(sm) + tl.r * LD + tl.c0 + c0;
#pragma unroll
    for (int c = 0; c < 8; ++c) T[c] = q.e[c0 + c] > kOff / 2 ? scaled_sum(hi[c], lo[c], q.e[c0 + c]) : 0.0;
  }
  template <int EW>
  __device__ __forceinline__ void finish(const OzArgs& g, const OzTile& tl, uint8_t* smraw) const {
    const double* T = reinterpret_cast<const double*>(smraw);
    double* red = reinterpret_cast<double*>(smraw) + BM * LD;
    const int ew = tl.ew, lane = tl.lane;
    asm volatile("bar.sync 2, %0;" ::"n"(32 * EW) : "memory");
    const int nw = WT >= EW ? 1 : EW / WT, per = EW / nw;  // warps per walker, walkers at a time
    const int nrow = RG * N, nd = (N - 1) / 2;
    const int sub = ew % nw;
    for (int w0 = 0; w0 < WT; w0 += per) {
      const int wl = w0 + ew / nw, w = tl.nt * WT + wl;
      const bool mine = ew < per * nw && wl < WT && w < W;
      double er = 0.0, ei = 0.0;
      if (mine) {
        const double* Tw = T + wl * 2 * N;
        for (int rr = sub * 32 + lane; rr < nrow; rr += 32 * nw) {
          const int gl = rr / N, i = rr - gl * N;
          const double* own = Tw + rr * LD;
          const double* colp = Tw + gl * N * LD + i;
          const double dr = own[i], di = own[N + i];
          double pr = 0.0, pi = 0.0;
          for (int d = 1; d <= nd; ++d) {
            const int j = i + d < N ? i + d : i + d - N;
            if (nup > 0 && (i < nup) != (j < nup)) continue;
            const double ar = own[j], ai = own[N + j], br = colp[j * LD], bi = colp[j * LD + N];
            pr = fma(ar, br, fma(-ai, bi, pr));
            pi = fma(ar, bi, fma(ai, br, pi));
          }
          double sr = fma(dr, dr, fma(-di, di, 2.0 * pr)), si = fma(2.0 * dr, di, 2.0 * pi);
          if ((N & 1) == 0) {
            const int j = i + N / 2 < N ? i + N / 2 : i - N / 2;
            if (nup <= 0 || (i < nup) == (j < nup)) {
              const double ar = own[j], ai = own[N + j], br = colp[j * LD], bi = colp[j * LD + N];
              sr = fma(ar, br, fma(-ai, bi, sr));
              si = fma(ar, bi, fma(ai, br, si));
            }
          }
          er += sr;
          ei += si;
        }
        er = warp_sum(er);
        ei = warp_sum(ei);
        if (lane == 0) {
          red[2 * ew] = er;
          red[2 * ew + 1] = ei;
        }
      }
      asm volatile("bar.sync 2, %0;" ::"n"(32 * EW) : "memory");
      if (mine && sub == 0 && lane < 2) {
        double sum = 0.0;
        for (int k = 0; k < nw; ++k) sum += red[2 * (ew + k) + lane];
        part[((long)w * nchunk + tl.mt) * 2 + lane] = sum;
      }
      asm volatile("bar.sync 2, %0;" ::"n"(32 * EW) : "memory");
    }
  }
};

template <int BN, class Epi, bool MULTI>
int launch_oz_as(const OzArgs& g, const Epi& e, cudaStream_t st) {
  static std::atomic<unsigned long long> attr{0};
  constexpr int smem = OzSmem<BN, Epi>::TOTAL;
  static_assert(smem <= 227 * 1024, "shared memory");
  AFQ_TRY(smem_attr_once(k_oz_gemm<BN, Epi, MULTI>, smem, attr));
  const int sms = tc_sm_count();
  AFQ_LAUNCH((k_oz_gemm<BN, Epi, MULTI>), g.ntiles < sms ? g.ntiles : sms, kOzThreads<BN>, smem, st, g, e);
  return AFQMC_OK;
}
template <int BN, class Epi>
int launch_oz(const OzArgs& g, const Epi& e, cudaStream_t st) {
  if (g.ntiles <= 0) return AFQMC_OK;
  return g.nseg > 1 ? launch_oz_as<BN, Epi, true>(g, e, st) : launch_oz_as<BN, Epi, false>(g, e, st);
}

OzArgs oz_args(const OzOperand& A, const OzOperand& B, long m, long n, int batch, int* err) {
  OzArgs g;
  g.A = static_cast<const char*>(A.data);
  g.B = static_cast<const char*>(B.data);
  g.a_batch = A.batch_stride;
  g.b_batch = B.batch_stride;
  g.ea = A.exps;
  g.eb = B.exps;
  g.ea_batch = A.batch_exp_stride;
  g.eb_batch = B.batch_exp_stride;
  g.a_rpt = A.rows_per_tile;
  g.b_rpt = B.rows_per_tile;
  g.RTA = A.RT;
  g.a_bytes = kS * A.RT * 32;
  g.nkb = A.nkb;
  g.nseg = (A.nkb + kOzSegBlk - 1) / kOzSegBlk;
  g.nmt = (int)oz_tiles(m, A.rows_per_tile);
  g.nnt = (int)oz_tiles(n, B.rows_per_tile);
  g.ntiles = g.nmt * g.nnt * batch;
  g.a_mod = batch;
  g.err = err;
  return g;
}

int check_operand(const OzOperand& A, const OzOperand& B, int bn) {
  if (!A.data || !B.data || !A.exps || !B.exps || A.nkb != B.nkb || A.nkb < 1 || A.RT % 8 || A.RT < A.rows_per_tile ||
      A.RT > BM || B.RT != bn || B.rows_per_tile > bn || A.rows_per_tile < 1 || B.rows_per_tile < 1) {
    set_error("sliced contraction: operands do not match");
    return AFQMC_EINVAL;
  }
  return AFQMC_OK;
}

}  // namespace

// The slicing kernels of a few blocks per SM overlap their predecessor's tail (see
// AFQ_LAUNCH_PDL): launched one by one, five steps and an energy of 32 and 300
// walkers take at M = 36, N = 4 1366 -> 1151 and 1586 -> 1398 us, at M = 100, N = 10
// 2109 -> 1950 and 3739 -> 3554 us.  In a graph larger ones gain nothing and lose up
// to 0.5 %.
#define OZ_LAUNCH(kernel, grid, ...)                                          \
  do {                                                                        \
    const dim3 g_(grid);                                                      \
    if ((long)g_.x * g_.y * g_.z <= 4L * tc_sm_count())                       \
      AFQ_LAUNCH_PDL(kernel, g_, __VA_ARGS__);                                \
    else                                                                      \
      AFQ_LAUNCH(kernel, g_, __VA_ARGS__);                                    \
  } while (0)

int oz_slice_rows(const double* src, long rows, int k, long ld, const OzOperand& o, cudaStream_t st) {
  if (rows <= 0) return AFQMC_OK;
  const long groups = (long)oz_tiles(rows, o.rows_per_tile) * ((o.rows_per_tile + 7) / 8);
  OZ_LAUNCH(k_oz_slice_rows, (unsigned)groups, 256, 0, st, src, rows, k, ld, o);
  return AFQMC_OK;
}

int oz_slice_v(const double* Y, long ldy, int W, int M, int Mp, const OzOperand& o, cudaStream_t st) {
  dim3 grid((unsigned)(oz_tiles(M, o.rows_per_tile) * ((o.rows_per_tile + 7) / 8)), W);
  OZ_LAUNCH(k_oz_slice_v, grid, 256, 0, st, Y, ldy, M, Mp, o);
  return AFQMC_OK;
}

int oz_slice_term(const double* t, int W, int N, int M, int Mp, const OzOperand& o, cudaStream_t st) {
  dim3 grid(cdiv(N, 8), W);
  OZ_LAUNCH(k_oz_slice_term, grid, 256, 0, st, t, N, M, Mp, o);
  return AFQMC_OK;
}

int oz_gemm_store(const OzGemm& g, cudaStream_t st) {
  AFQ_TRY(check_operand(g.A, g.B, 64));
  EpiOzStore e{g.C, g.ldc, g.c_batch, g.m, g.n, g.alpha_log2, g.mask, g.mask_rows};
  return launch_oz<64>(oz_args(g.A, g.B, g.m, g.n, g.batch, g.err), e, st);
}

int oz_term_width(int N) { return 2 * N <= 16 ? 16 : 2 * N <= 32 ? 32 : 64; }

int oz_taylor_term(const OzTerm& t, cudaStream_t st) {
  const int bn = oz_term_width(t.N);
  AFQ_TRY(check_operand(t.V, t.T, bn));
  EpiOzTerm e{t.M, 2 * t.N, t.k == 1, t.last ? 1 : 0, t.scale, t.tin, t.tout, t.acc};
  const OzArgs g = oz_args(t.V, t.T, t.M, 2 * t.N, t.W, t.err);
  if (bn == 16) return launch_oz<16>(g, e, st);
  if (bn == 32) return launch_oz<32>(g, e, st);
  return launch_oz<64>(g, e, st);
}

int oz_row_exps(const double* src, long n, int M, int* exps, cudaStream_t st) {
  AFQ_LAUNCH_PDL(k_oz_row_exps, (unsigned)((n + 31) / 32), 256, 0, st, src, n, M, exps);
  return AFQMC_OK;
}

int oz_slice_cols(const double* phi, int W, int N, int M, const int* planes, const OzOperand& o, cudaStream_t st) {
  OZ_LAUNCH(k_oz_slice_cols, dim3(cdiv(M, 32), W), 256, 0, st, phi, N, M, planes, o);
  return AFQMC_OK;
}

int oz_slice_densities(const double* phi, const double* thA, const double* thB, int W, int N, int M, int w0,
                       int nz, int cw, int* planes, const OzOperand& A, const OzOperand& B, cudaStream_t st) {
  const int n = W - w0 < nz * cw ? W - w0 : nz * cw;
  AFQ_TRY(oz_row_exps(phi + (long)w0 * 2 * N * M, 2L * N * n, M, planes, st));
  OZ_LAUNCH(k_oz_slice_densities, dim3(cdiv(M, 32), nz, 4), 256, 0, st, phi, thA, thB, W, N, M, w0, cw, planes, A, B);
  return AFQMC_OK;
}

int oz_slice_inverse(const double2* sinv, int W, int w0, int nw, int nds, int N, const int* planes,
                     const OzOperand& o, cudaStream_t st) {
  OZ_LAUNCH(k_oz_slice_inverse, dim3(nw, nds), 256, 0, st, sinv, W, w0, N, planes, o);
  return AFQMC_OK;
}

int oz_theta(const OzTheta& t, cudaStream_t st) {
  const int bn = oz_term_width(t.N);
  AFQ_TRY(check_operand(t.A, t.B, bn));
  EpiOzTheta e{t};
  OzArgs g = oz_args(t.A, t.B, t.M, 2 * t.N, t.nds * t.nw, t.err);
  g.a_mod = t.nw;
  if (bn == 16) return launch_oz_as<16, EpiOzTheta, false>(g, e, st);
  if (bn == 32) return launch_oz_as<32, EpiOzTheta, false>(g, e, st);
  return launch_oz_as<64, EpiOzTheta, false>(g, e, st);
}

int oz_gram(const OzOperand& rows, int W, int N, double* gram, int* err, cudaStream_t st) {
  const int bn = oz_term_width(N);
  AFQ_TRY(check_operand(rows, rows, bn));
  EpiOzGram e{2 * N, gram};
  const OzArgs g = oz_args(rows, rows, 2 * N, 2 * N, W, err);
  if (bn == 16) return launch_oz<16>(g, e, st);
  if (bn == 32) return launch_oz<32>(g, e, st);
  return launch_oz<64>(g, e, st);
}

int oz_exchange_vectors(int N) { return BM / N > 0 ? BM / N : 1; }
int oz_exchange_walkers(int N) { return 64 / (2 * N); }

int oz_exchange(const OzExchange& x, cudaStream_t st) {
  AFQ_TRY(check_operand(x.A, x.B, 64));
  EpiOzExchange e{x.N, x.W, x.G, x.A.rows_per_tile / x.N, x.B.rows_per_tile / (2 * x.N),
                  x.nup, x.nchunk, x.part};
  return launch_oz<64>(oz_args(x.A, x.B, (long)x.G * x.N, 2L * x.N * x.W, 1, x.err), e, st);
}

}  // namespace afq
