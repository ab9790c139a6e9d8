// digit.cu -- the FP64 sine transforms of Eq. 4.6 as digit products on the
// tensor cores (digit.cuh).
//
// P-hat^-1 v = (1-Phi) S W1 + Phi S W2 with S = S_{n2} (x) S_{n1}, W = S v,
// W1 = W / (1 - Lx - Ly), W2 = W / (1 + dt/eta - Lx - Ly).  As matrices (rows
// y, columns x) the passes are those of the split-BF16 form (dst_gemm.cu),
// every product's output FP64 and transposed, with a split into digits before
// each:
//   1. v               -> digits,  T^T  = (v S_x)^T             (n1 x n2)
//   2. T^T             -> digits,  W1, W2 from T^T S_y          (each n2 x n1)
//   3. [W1; W2]        -> digits,  Y^T  = ([W1; W2] S_x)^T      (two n1 x n2)
//   4. Y^T             -> digits,  z = S_y Y_c where the mask selects channel c
// The operator M z (Eq. 2.14-2.17) is two more such products, with the symmetric
// Toeplitz matrices in place of S: they are centrosymmetric too (T[n-1-i][n-1-j]
// = T[i][j]), so with z+_j = z_j + z_{n-1-j} and z-_j = z_j - z_{n-1-j}
//     (T z)_i, (T z)_{n-1-i} = sum_j U_ij z+_j +- sum_j V_ij z-_j,
//     U_ij, V_ij = (T_ij +- T_{i,n-1-j}) / 2,   i, j < (n+1)/2:
// the layout of the symmetric sine product, half the work of the full one.
//
// A product's epilogue also finds the largest exponent of every row of its
// output, so the next split is one elementwise pass.
#include <cmath>
#include <cstring>
#include <vector>

#include "digit.cuh"
#include "internal.h"
#include "transforms.cuh"

namespace rsfde {

namespace {

int pad16(int n) { return (n + 15) / 16 * 16; }

// The digits of one operand: eight planes of rows x 2 hk BF16.
struct DigitMat {
  __nv_bfloat16* d = nullptr;
  int rows = 0, hk = 0;
  size_t plane() const { return (size_t)rows * 2 * hk; }
  CUtensorMap map[3];  // A: [0]; S: tiles of 64, 32 and 16 rows
};

// Tiles of box_rows rows of one digit plane, or of box_z planes stacked.
bool digit_map(const DigitMat* m, CUtensorMap* map, int box_rows, int box_z) {
  EncodeTiledFn enc = encode_fn();
  if (!enc) return false;
  cuuint64_t dim[3] = {(cuuint64_t)(2 * m->hk), (cuuint64_t)m->rows, (cuuint64_t)kDgDigits};
  cuuint64_t stride[2] = {(cuuint64_t)(2 * m->hk) * 2, (cuuint64_t)m->plane() * 2};
  cuuint32_t box[3] = {(cuuint32_t)kDgBK, (cuuint32_t)box_rows, (cuuint32_t)box_z};
  cuuint32_t es[3] = {1, 1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, m->d, dim, stride, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Digits of one row's eight consecutive columns x = 8c .. 8c + 7 (quantised q,
// zero past the row's end): the even x to columns 4c .. 4c + 3 of the even
// half, the odd x to those of the odd half.
__device__ __forceinline__ void store_digits(const long long* q, __nv_bfloat16* row, size_t plane, int hk, int c) {
#pragma unroll
  for (int i = 0; i < kDgDigits; ++i) {
    uint32_t v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = dg_digit((unsigned long long)(q[k] + kDgBias), i);
    __nv_bfloat16* p = row + i * plane + 4 * c;
    *reinterpret_cast<uint2*>(p) = make_uint2(dg_pack(v[0], v[2]), dg_pack(v[4], v[6]));
    *reinterpret_cast<uint2*>(p + hk) = make_uint2(dg_pack(v[1], v[3]), dg_pack(v[5], v[7]));
  }
}

// The digits of four quantised values p (to columns 4c .. 4c + 3 of the first
// half) and m (of the second half).
__device__ __forceinline__ void store_digits4(const long long* p, const long long* m, __nv_bfloat16* row, size_t plane,
                                              int hk, int c) {
  long long q[8];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    q[2 * k] = p[k];
    q[2 * k + 1] = m[k];
  }
  store_digits(q, row, plane, hk, c);
}

// The first operand: rows y of scale * v (one block per row, one group of
// eight columns per thread: n1 <= 2048, so at most 256), the row's exponent to
// rexp[y]; resets the exponent arrays of the later operands.
template <typename Tin>
__global__ void __launch_bounds__(256)
    digit_split_rows_kernel(const Tin* __restrict__ v, const double* scale, __nv_bfloat16* __restrict__ d, int n1,
                            size_t plane, int hk, int* __restrict__ rexp, int* __restrict__ reset, int nreset, int* err,
                            const int* gate) {
  pdl_wait();
  pdl_trigger();
  if (gate && *(volatile const int*)gate == 0) return;
  __shared__ uint32_t wmax[8];
  const int y = blockIdx.x, c = threadIdx.x;
  for (int k = y * blockDim.x + c; k < nreset; k += gridDim.x * blockDim.x) reset[k] = kDgNone;
  if (y == 0 && c == 0) *err = 0;  // an earlier application's give-up is that application's
  const double sc = scale ? *scale : 1.0;
  double x[8];
  uint32_t e = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int p = 8 * c + k;
    x[k] = p < n1 ? scaled_load<double>(sc, 0.0f, v[(size_t)y * n1 + p]) : 0.0;
    e = max(e, dg_exponent(x[k]));
  }
  e = __reduce_max_sync(0xffffffffu, e);
  if ((c & 31) == 0) wmax[c >> 5] = e;
  __syncthreads();
  for (int w = 0; w < (int)blockDim.x / 32; ++w) e = max(e, wmax[w]);
  if (c == 0) rexp[y] = e == 2047 ? kDgNan : e ? (int)e : 1;
  if (4 * c >= hk) return;
  long long q[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) q[k] = e == 2047 ? 0 : dg_quantize(x[k], e ? (int)e : 1);
  store_digits(q, d + (size_t)y * 2 * hk, plane, hk, c);
}

// round(W 2^-sh), |.| <= 2^55
__device__ __forceinline__ long long dg_shift(long long w, int sh) {
  if (sh <= 0) return w << (-sh);
  return sh < 63 ? (w + (1ll << (sh - 1))) >> sh : 0ll;
}

// A later operand from a product's W: rows of length len of src0 (rows below
// row_b) and src1 (the others); column m's values are W 2^(cexp[m] + kexp)
// (the second channel's exponents follow the first's), row r's entries below
// 2^(rexp[r] - 1022).
__global__ void __launch_bounds__(kBlock)
    digit_split_kernel(const long long* __restrict__ src0, const long long* __restrict__ src1, int row_b, int rows,
                       int len, const int* __restrict__ cexp, int kexp, const int* __restrict__ rexp,
                       __nv_bfloat16* __restrict__ d, size_t plane, int hk, const int* gate) {
  pdl_wait();
  pdl_trigger();
  if (gate && *(volatile const int*)gate == 0) return;
  const int gpr = hk >> 2;  // groups of eight columns per row
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int row = t / gpr, c = t - row * gpr;
  if (row >= rows) return;
  const bool ch = row >= row_b;
  const long long* __restrict__ s = ch ? src1 + (size_t)(row - row_b) * len : src0 + (size_t)row * len;
  const int* __restrict__ ce = ch ? cexp + len : cexp;
  const int E = __ldg(rexp + row);
  const bool live = E != kDgNone && E != kDgNan;
  long long q[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int p = 8 * c + k;
    q[k] = (p < len && live) ? dg_shift(s[p], E - 1077 - (__ldg(ce + p) + kexp)) : 0;
  }
  store_digits(q, d + (size_t)row * 2 * hk, plane, hk, c);
}

// The operand [W1; W2]: both quotients of the tau divides (as products with the
// tabulated reciprocals) of row y's W, as rows y and rows + y.
__global__ void __launch_bounds__(kBlock)
    digit_split_quotients_kernel(const long long* __restrict__ src, int rows, int len, const int* __restrict__ cexp,
                                 int kexp, const double* __restrict__ inv0, const double* __restrict__ inv1,
                                 const int* __restrict__ rexp, __nv_bfloat16* __restrict__ d, size_t plane, int hk,
                                 const int* gate) {
  pdl_wait();
  pdl_trigger();
  if (gate && *(volatile const int*)gate == 0) return;
  const int gpr = hk >> 2;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int row = t / gpr, c = t - row * gpr;
  if (row >= rows) return;
  const size_t o = (size_t)row * len;
  const int E0 = __ldg(rexp + row), E1 = __ldg(rexp + rows + row);
  const bool live = E0 != kDgNone && E0 != kDgNan;  // (the two rows are zero, or not finite, together)
  long long q0[8], q1[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int p = 8 * c + k;
    q0[k] = q1[k] = 0;
    if (p < len && live) {
      const double v = ldexp_i64(src[o + p], __ldg(cexp + p) + kexp);
      q0[k] = dg_quantize(v * __ldg(inv0 + o + p), E0);
      q1[k] = dg_quantize(v * __ldg(inv1 + o + p), E1);
    }
  }
  store_digits(q0, d + (size_t)row * 2 * hk, plane, hk, c);
  store_digits(q1, d + (size_t)(rows + row) * 2 * hk, plane, hk, c);
}

// The digits of S_n's first (n + 1) / 2 rows from tab[m] = round(2^sh
// sqrt(2/(n+1)) sin(pi m / (n+1))), m mod 2 (n+1); one block per row.
// *rowsum: the largest sum of |digits| over half a row (the exactness bound).
__global__ void __launch_bounds__(256)
    digit_sine_kernel(const long long* __restrict__ tab, int n, __nv_bfloat16* __restrict__ d, size_t plane, int hk,
                      int* rowsum) {
  const int i = blockIdx.x, per = 2 * (n + 1);
  __shared__ int half[2];
  if (threadIdx.x < 2) half[threadIdx.x] = 0;
  __syncthreads();
  int sum[2] = {0, 0};
  for (int c = threadIdx.x; 4 * c < hk; c += blockDim.x) {
    long long q[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int j = 8 * c + k;
      q[k] = j < n ? tab[(int)(((long long)(i + 1) * (j + 1)) % per)] : 0;
      for (int g = 0; g < kDgDigits; ++g)
        sum[k & 1] += abs((int)dg_digit((unsigned long long)(q[k] + kDgBias), g) - 64);
    }
    store_digits(q, d + (size_t)i * 2 * hk, plane, hk, c);
  }
  atomicAdd(&half[0], sum[0]);
  atomicAdd(&half[1], sum[1]);
  __syncthreads();
  if (threadIdx.x < 2) atomicMax(rowsum, half[threadIdx.x]);
}

// Both operands of the operator from z, in one launch, and the part of M z that
// is not left to the products.  The first `rblocks` blocks take the rows (one or
// more warps each): row y folded (z+, z-) to digits dr, its exponent to er[y], and
//     pre = (1 - t0x - t0y) z - t1x (z_left + z_right) - t1y (z_below + z_above),
// the identity and the three middle diagonals of both Toeplitz matrices in FP64.  The others take CPB columns each, held in shared memory
// (read once, for the largest entries and for the digits): digits dc (rows x),
// exponents ec[x].
//
// The middle diagonals stay out of the digits because they are far larger than the rest: from
// the weights of Eq. 2.6 |t0 / t2| = 12 / ((alpha - 1)(2 - alpha)), 48 at alpha = 1.5 and more
// towards 1 and 2, and |t1 / t2| >= 22.  The products' absolute error is set by the largest
// coefficient and would be 1e-15 to 5e-15 of M z (an FP64 FFT: 2e-16 to 3e-16); without them it is
// at least 48 times smaller: measured over 1 x 1 .. 2048 x 64, M z is then
// within 1.6e-16 (2-norm) of the extended-precision product, the FFTs 3.2e-16.
template <typename Tin, int CPB>
__global__ void __launch_bounds__(256)
    digit_fold_kernel(const Tin* __restrict__ z, int n1, int n2, int rblocks, const double* __restrict__ near, double* __restrict__ pre,
                      __nv_bfloat16* __restrict__ dr, size_t pr, int h1, int* __restrict__ er,
                      __nv_bfloat16* __restrict__ dc, size_t pc, int h2, int* __restrict__ ec, int* err,
                      const int* gate) {
  pdl_wait();
  pdl_trigger();
  if (gate && *(volatile const int*)gate == 0) return;
  __shared__ uint32_t wmax[8][CPB];
  extern __shared__ __align__(16) double fold_sm[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (blockIdx.x == 0 && tid == 0) *err = 0;
  if ((int)blockIdx.x < rblocks) {
    const int wpr = (h1 / 4 + 31) / 32, rpb = 8 / wpr;  // warps per row (at most 8), rows per block
    const int y = blockIdx.x * rpb + warp / wpr, c = (warp % wpr) * 32 + lane, half = (n1 + 1) / 2;
    const bool row = warp / wpr < rpb && y < n2;
    double a[4], b[4];  // z_j and its mirror
    uint32_t e = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int j = 4 * c + k;
      const bool in = row && j < half;
      a[k] = in ? cvt<double>(z[(size_t)y * n1 + j]) : 0.0;
      b[k] = in ? cvt<double>(z[(size_t)y * n1 + n1 - 1 - j]) : 0.0;
      e = max(e, max(dg_exponent(a[k]), dg_exponent(b[k])));
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) wmax[warp][0] = e;
    __syncthreads();
    if (!row) return;
    for (int w = 0; w < wpr; ++w) e = max(e, wmax[warp / wpr * wpr + w][0]);
    if (c == 0) er[y] = e == 2047 ? kDgNan : (e ? (int)e : 1) + 1;
    if (4 * c >= h1) return;
    const double c0 = __ldg(near), t1x = __ldg(near + 1), t1y = __ldg(near + 2);
    long long p[4], m[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int j = 4 * c + k, E = (e ? (int)e : 1) + 1;
      const bool mid = 2 * j + 1 == n1;
      const long long qa = e == 2047 ? 0 : dg_quantize(a[k], E);
      const long long qb = (e == 2047 || mid) ? 0 : dg_quantize(b[k], E);  // the middle once
      p[k] = qa + qb;
      m[k] = mid ? 0 : qa - qb;
      if (j < half) {
#pragma unroll
        for (int mir = 0; mir < 2; ++mir) {
          if (mir && mid) break;
          const int x = mir ? n1 - 1 - j : j;
          const size_t o = (size_t)y * n1 + x;
          const double sx = (x > 0 ? cvt<double>(z[o - 1]) : 0.0) + (x + 1 < n1 ? cvt<double>(z[o + 1]) : 0.0);
          const double sy = (y > 0 ? cvt<double>(z[o - n1]) : 0.0) + (y + 1 < n2 ? cvt<double>(z[o + n1]) : 0.0);
          const double v = __fma_rn(-t1x, sx, c0 * (mir ? b[k] : a[k]));
          pre[o] = __fma_rn(-t1y, sy, v);
        }
      }
    }
    store_digits4(p, m, dr + (size_t)y * 2 * h1, pr, h1, c);
    return;
  }
  const int x0 = (blockIdx.x - rblocks) * CPB, ncol = min(CPB, n1 - x0), half = (n2 + 1) / 2;
  const int ld = n2 + 1;
  uint32_t e[CPB] = {0};
  for (int y = tid; y < n2; y += blockDim.x) {
#pragma unroll
    for (int c = 0; c < CPB; ++c) {
      const double v = c < ncol ? cvt<double>(z[(size_t)y * n1 + x0 + c]) : 0.0;
      fold_sm[c * ld + y] = v;
      e[c] = max(e[c], dg_exponent(v));
    }
  }
#pragma unroll
  for (int c = 0; c < CPB; ++c) {
    const uint32_t w = __reduce_max_sync(0xffffffffu, e[c]);
    if (lane == 0) wmax[warp][c] = w;
  }
  __syncthreads();
  if (tid < ncol) {
    uint32_t w = 0;
    for (int k = 0; k < 8; ++k) w = max(w, wmax[k][tid]);
    ec[x0 + tid] = w == 2047 ? kDgNan : (w ? (int)w : 1) + 1;
  }
  const int gpc = h2 >> 2;  // groups of four per column
  for (int t = tid; t < ncol * gpc; t += blockDim.x) {
    const int c = t / gpc, g = t - c * gpc;
    uint32_t w = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) w = max(w, wmax[k][c]);
    const int E = (w ? (int)w : 1) + 1;
    long long p[4], m[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int j = 4 * g + k;
      const bool in = j < half && w != 2047, mid = 2 * j + 1 == n2;
      const long long qa = in ? dg_quantize(fold_sm[c * ld + j], E) : 0;
      const long long qb = (in && !mid) ? dg_quantize(fold_sm[c * ld + n2 - 1 - j], E) : 0;
      p[k] = qa + qb;
      m[k] = mid ? 0 : qa - qb;
    }
    store_digits4(p, m, dc + (size_t)(x0 + c) * 2 * h2, pc, h2, g);
  }
}

// The digits of [2U | 2V] from tq[k] = round(2^sh t_k); one block per row i < (n + 1) / 2.
__global__ void __launch_bounds__(256)
    digit_toeplitz_kernel(const long long* __restrict__ tq, int n, __nv_bfloat16* __restrict__ d, size_t plane, int hk,
                          int* rowsum) {
  const int i = blockIdx.x, half = (n + 1) / 2;
  __shared__ int hsum[2];
  if (threadIdx.x < 2) hsum[threadIdx.x] = 0;
  __syncthreads();
  int sum[2] = {0, 0};
  for (int c = threadIdx.x; 4 * c < hk; c += blockDim.x) {
    long long u[4], v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int j = 4 * c + k;
      const long long a = j < half ? tq[abs(i - j)] : 0, b = j < half ? tq[abs(i - (n - 1 - j))] : 0;
      u[k] = a + b;
      v[k] = a - b;
      for (int g = 0; g < kDgDigits; ++g) {
        sum[0] += abs((int)dg_digit((unsigned long long)(u[k] + kDgBias), g) - 64);
        sum[1] += abs((int)dg_digit((unsigned long long)(v[k] + kDgBias), g) - 64);
      }
    }
    store_digits4(u, v, d + (size_t)i * 2 * hk, plane, hk, c);
  }
  atomicAdd(&hsum[0], sum[0]);
  atomicAdd(&hsum[1], sum[1]);
  __syncthreads();
  if (threadIdx.x < 2) atomicMax(rowsum, hsum[threadIdx.x]);
}

// 1 / (1 - lx - ly) and 1 / (1 + dt/eta - lx - ly) at [y * n1 + x]
__global__ void __launch_bounds__(kBlock)
    digit_reciprocals_kernel(const double* __restrict__ lx, const double* __restrict__ ly, double pen, int n1, int n2,
                             double* __restrict__ i0, double* __restrict__ i1) {
  const size_t N = (size_t)n1 * n2;
  for (size_t p = blockIdx.x * (size_t)blockDim.x + threadIdx.x; p < N; p += (size_t)gridDim.x * blockDim.x) {
    const int y = (int)(p / (size_t)n1), x = (int)(p - (size_t)y * n1);
    const double base = 1.0 - lx[x] - ly[y];
    i0[p] = 1.0 / base;
    i1[p] = 1.0 / (base + pen);
  }
}

}  // namespace

struct DigitPlan {
  int n1 = 0, n2 = 0;
  DigitMat Sx, Sy, A0, T, W, Y;  // A0, T, W and Y share one buffer (each is consumed before the next is written)
  int kx = 0, ky = 0;            // scale of a product with S_x, S_y (DigitEpiParams::kexp)
  double* inv = nullptr;         // the two tables of reciprocals (N each)
  int* exps = nullptr;           // row exponents: n2 (A0), n1 (T), 2 n2 (W), 2 n1 (Y)
  int* err = nullptr;            // an application's give-up flag (digit_gemm_kernel), and a word for the setup
  int* gave_up = nullptr;        // the context's
  void* mem = nullptr;
  long long wait_cycles = kWaitCycles;
};

// S_n as digits; *kexp the scale of a product with it.  RSFDE_EINVAL: none of the
// scales keeps the accumulators exact.  So it is for 21 of the sides up to 2048: 1869, 1895,
// 1907, 1915, 1919, 1931, 1947, 1959, 1963, 1969, 1975, 1979, 1983, 1987, 1991, 1999, 2015, 2023, 2031,
// 2039 and 2047.  There n + 1 has divisors d such that some rows' sines take few values; one
// magnitude then stands in most of half a row, and if its digits sum to more than about 256 they
// are not averaged over the row as other rows' are.
static int build_sine(DigitMat* S, int n, long long* tab_dev, int* rowsum_dev, int* kexp, cudaStream_t s) {
  const long per = 2L * (n + 1);
  std::vector<long long> tab(per);
  const long double sc = sqrtl(2.0L / (n + 1));
  int E = 0;
  frexpl(sc, &E);  // sc < 2^E
  for (int extra = 0; extra < 3; ++extra) {
    const int sh = 55 - (E + extra);
    for (long m = 0; 2 * m <= n + 1; ++m) {  // a quarter wave; the rest by symmetry
      const long long v =
          llroundl(ldexpl(sc * sinl(3.14159265358979323846264338327950288L * m / (n + 1)), sh));
      tab[m] = tab[n + 1 - m] = v;
      tab[(per - m) % per] = tab[n + 1 + m] = -v;
    }
    tab[0] = tab[n + 1] = 0;
    int rowsum = 0;
    if (cudaMemcpyAsync(tab_dev, tab.data(), per * sizeof(long long), cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaMemsetAsync(rowsum_dev, 0, sizeof(int), s) != cudaSuccess)
      return RSFDE_ECUDA;
    digit_sine_kernel<<<S->rows, 256, 0, s>>>(tab_dev, n, S->d, S->plane(), S->hk, rowsum_dev);
    if (cudaMemcpyAsync(&rowsum, rowsum_dev, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
      return RSFDE_ECUDA;
    // x = x_q 2^(E_x - 1077), S = S_q 2^-sh, sum x S = W 2^(9 + 49) 2^(E_x - 1077 - sh)
    *kexp = 58 - 1077 - sh;
    if (64LL * rowsum <= (1LL << 24)) return RSFDE_OK;
  }
  return RSFDE_EINVAL;
}

bool digit_sizes_ok(int n1, int n2) { return n1 <= kDgMaxN && n2 <= kDgMaxN; }

int digit_plan_create(DigitPlan** out, int n1, int n2, int* gave_up, cudaStream_t s) {
  *out = nullptr;
  if (!digit_sizes_ok(n1, n2)) return RSFDE_EINVAL;
  DigitPlan* p = new (std::nothrow) DigitPlan();
  if (!p) return RSFDE_ENOMEM;
  p->gave_up = gave_up;
  p->n1 = n1;
  p->n2 = n2;
  const int h1 = pad16((n1 + 1) / 2), h2 = pad16((n2 + 1) / 2);
  auto shape = [](DigitMat* m, int rows, int hk) {
    m->rows = rows;
    m->hk = hk;
  };
  shape(&p->Sx, (n1 + 1) / 2, h1);
  shape(&p->Sy, (n2 + 1) / 2, h2);
  shape(&p->A0, n2, h1);
  shape(&p->T, n1, h2);
  shape(&p->W, 2 * n2, h1);
  shape(&p->Y, 2 * n1, h2);
  auto bytes = [](const DigitMat& m) { return (m.plane() * kDgDigits * 2 + 255) / 256 * 256; };
  const size_t sx = bytes(p->Sx), sy = n1 == n2 ? 0 : bytes(p->Sy), sw = bytes(p->W) > bytes(p->Y) ? bytes(p->W) : bytes(p->Y);
  const size_t si = ((size_t)2 * n1 * n2 * sizeof(double) + 255) / 256 * 256;
  const int nexp = 3 * (n1 + n2);
  const size_t se = ((size_t)nexp * sizeof(int) + 255) / 256 * 256;
  const size_t stab = (size_t)2 * (kDgMaxN + 1) * sizeof(long long);
  if (cudaMalloc(&p->mem, sx + sy + sw + si + se + 256 + stab) != cudaSuccess) {
    take_launch_error();
    delete p;
    return RSFDE_ENOMEM;
  }
  uint8_t* b = static_cast<uint8_t*>(p->mem);
  p->Sx.d = reinterpret_cast<__nv_bfloat16*>(b);
  p->Sy.d = reinterpret_cast<__nv_bfloat16*>(n1 == n2 ? b : b + sx);  // equal sides share one matrix
  for (DigitMat* m : {&p->A0, &p->T, &p->W, &p->Y}) m->d = reinterpret_cast<__nv_bfloat16*>(b + sx + sy);
  p->inv = reinterpret_cast<double*>(b + sx + sy + sw);
  p->exps = reinterpret_cast<int*>(b + sx + sy + sw + si);
  p->err = reinterpret_cast<int*>(b + sx + sy + sw + si + se);
  long long* tab = reinterpret_cast<long long*>(b + sx + sy + sw + si + se + 256);
  bool good = cudaMemsetAsync(p->err, 0, 256, s) == cudaSuccess &&
              cudaMemsetAsync(p->exps, 0, nexp * sizeof(int), s) == cudaSuccess;
  int rc = good ? build_sine(&p->Sx, n1, tab, p->err + 1, &p->kx, s) : RSFDE_ECUDA;
  p->ky = p->kx;
  if (n1 != n2 && rc == RSFDE_OK) rc = build_sine(&p->Sy, n2, tab, p->err + 1, &p->ky, s);
  good = rc == RSFDE_OK;
  for (DigitMat* m : {&p->A0, &p->T, &p->W, &p->Y}) good = good && digit_map(m, &m->map[0], kDgBM, 1);
  for (DigitMat* m : {&p->Sx, &p->Sy})
    for (int k = 0; k < 3; ++k) good = good && digit_map(m, &m->map[k], 64 >> k, kDgDigits);
  if (!good) {
    take_launch_error();
    digit_plan_destroy(p);
    return rc != RSFDE_OK ? rc : RSFDE_ECUDA;
  }
  *out = p;
  return RSFDE_OK;
}

void digit_plan_destroy(DigitPlan* p) {
  if (!p) return;
  if (p->mem) cudaFree(p->mem);
  delete p;
}

void digit_plan_params(DigitPlan* p, const double* lamx, const double* lamy, double pen, cudaStream_t s) {
  const size_t N = (size_t)p->n1 * p->n2;
  digit_reciprocals_kernel<<<vec_grid(N), kBlock, 0, s>>>(lamx, lamy, pen, p->n1, p->n2, p->inv, p->inv + N);
}

void digit_plan_set_wait(DigitPlan* p, long long cycles) {
  if (p) p->wait_cycles = cycles > 0 ? cycles : kWaitCycles;
}

template <typename Tin>
static void launch_split_rows(DigitPlan* p, const Tin* v, const double* vscale, const int* gate, cudaStream_t s) {
  const int thr = (p->A0.hk / 4 + 31) / 32 * 32;
  launch_pdl(digit_split_rows_kernel<Tin>, dim3(p->n2), dim3(thr), 0, s, v, vscale, p->A0.d, p->n1, p->A0.plane(),
             p->A0.hk, p->exps, p->exps + p->n2, 3 * p->n1 + 2 * p->n2, p->err, gate);
}
static dim3 split_grid(long rows, int hk) { return dim3((unsigned)((rows * (hk / 4) + kBlock - 1) / kBlock)); }
static void launch_split_fixed(const DigitMat& m, const long long* s0, const long long* s1, int row_b, int len,
                               const int* cexp, int kexp, const int* rexp, const int* gate, cudaStream_t s) {
  launch_pdl(digit_split_kernel, split_grid(m.rows, m.hk), dim3(kBlock), 0, s, s0, s1, row_b, m.rows, len, cexp, kexp,
             rexp, m.d, m.plane(), m.hk, gate);
}
// Width of the tiles: the one whose waves take least, a tile costing its 64-wide
// slices (2 per half) and a fixed part (fill, sums and stores).  Measured, in
// SM clocks: 3300 per slice at 16 and 32 (shared-memory reads of A), 4620 at 64
// (the tensor pipe); fixed 6000, 9600 and 25000.  P-hat^-1 at 64 x 64 with 16, 32
// or 64 throughout: 48.5, 56.3, 73.1 us; 512 x 512: 113, 112, 154; 1023 x 641:
// 335, 237, 241; 1024 x 1024: 457, 278, 282.
static int dg_bn(int N, int M, int hk) {
  const int width[3] = {64, 32, 16}, slice[3] = {4620, 3300, 3300}, fixed[3] = {25000, 9600, 6000};
  const long my = (M + kDgBM - 1) / kDgBM, slices = 2 * ((hk + kDgBK - 1) / kDgBK);
  int best = 64;
  long least = 1L << 60;
  for (int k = 0; k < 3; ++k) {
    const long waves = ((N + width[k] - 1) / width[k] * my + kNumSMs - 1) / kNumSMs;
    const long t = waves * (slices * slice[k] + fixed[k]);
    if (t < least) {
      least = t;
      best = width[k];
    }
  }
  return best;
}
template <int EPI, int BN>
static void launch_digit_bn(const DigitMat& A, const DigitMat& S, const DigitEpiParams& ep, int* err, const int* gate,
                            cudaStream_t s) {
  auto k = digit_gemm_kernel<EPI, BN>;
  raise_smem_limit((const void*)k, dg_smem(BN));
  launch_pdl(k, dim3((ep.N + BN - 1) / BN, (ep.M + kDgBM - 1) / kDgBM), dim3(kDgThreads), dg_smem(BN), s, A.map[0],
             S.map[BN == 64 ? 0 : BN == 32 ? 1 : 2], ep, err, gate);
}
// Columns per block of the operator's fold: four (32-byte pieces of z's rows, 64 KB at n2 =
// 2048: three blocks per SM) while that gives every SM a block, else two; and its blocks.
static int fold_cols(int n1) { return n1 >= 4 * kNumSMs ? 4 : 2; }
static int fold_rblocks(int n1, int n2) {
  const int wpr = (pad16((n1 + 1) / 2) / 4 + 31) / 32, rpb = 8 / wpr;
  return (n2 + rpb - 1) / rpb;
}
static int fold_blocks(int n1, int n2) {
  return fold_rblocks(n1, n2) + (n1 + fold_cols(n1) - 1) / fold_cols(n1);
}
// A S for a transform of length n; next: the blocks of the elementwise kernel that follows (0:
// another product).  An early trigger hides the next launch, but puts its blocks
// where there is room: beside a product that leaves SMs idle an elementwise grid
// lands on those few SMs, several blocks each, and waits there.  So the
// products trigger early only if the next blocks find an idle SM each.  Against
// triggering always: P-hat^-1 at 1023 x 641 216 -> 201 us, a step at 512 x 512 10.03 -> 9.40
// ms (never: 200 us and 9.52 ms); against never: a step at 64 x 64 2.74 -> 2.68 ms.
template <int EPI, typename Plan>
static void launch_digit(const Plan* p, const DigitMat& A, const DigitMat& S, int n, int kexp, int next,
                         DigitEpiParams ep, const int* gate, cudaStream_t s) {
  ep.M = A.rows;  // (DG_ROWS: A the matrix, S the operand's rows)
  ep.N = S.rows;
  ep.n_full = n;
  ep.hk = A.hk;
  ep.kexp = kexp;
  ep.wait_cycles = p->wait_cycles;
  ep.gave_up = p->gave_up;
  const int bn = dg_bn(ep.N, ep.M, ep.hk);
  ep.early = next == 0 || (ep.N + bn - 1) / bn * ((ep.M + kDgBM - 1) / kDgBM) + next <= kNumSMs;
  if (bn == 64) launch_digit_bn<EPI, 64>(A, S, ep, p->err, gate, s);
  else if (bn == 32) launch_digit_bn<EPI, 32>(A, S, ep, p->err, gate, s);
  else launch_digit_bn<EPI, 16>(A, S, ep, p->err, gate, s);
}

// The common start: v -> digits, T^T = (v S_x)^T as W into t, -> digits.
template <typename Tin>
static void digit_first(DigitPlan* p, const Tin* v, const double* vscale, double* t, const int* gate,
                        cudaStream_t s) {
  int* e1 = p->exps + p->n2;
  long long* w = reinterpret_cast<long long*>(t);
  launch_split_rows(p, v, vscale, gate, s);
  DigitEpiParams ep{};
  ep.rexp = p->exps;
  ep.row_b = 1 << 30;
  ep.out0 = w;
  ep.ldo = p->n2;
  ep.oexp = e1;
  launch_digit<DG_FIXED>(p, p->A0, p->Sx, p->n1, p->kx, split_grid(p->T.rows, p->T.hk).x, ep, gate, s);
  launch_split_fixed(p->T, w, nullptr, 1 << 30, p->n2, p->exps, p->kx, e1, gate, s);
}

template <typename Tin>
void digit_precond(DigitPlan* p, const Tin* v, const double* vscale, double* z, const uint8_t* phi, double* t,
                   double* wa, double* wb, const int* gate, cudaStream_t s) {
  const int n1 = p->n1, n2 = p->n2;
  const size_t N = (size_t)n1 * n2;
  int* e1 = p->exps + n2;
  int* e2 = e1 + n1;
  int* e3 = e2 + 2 * n2;
  long long* a = reinterpret_cast<long long*>(wa);
  long long* b = reinterpret_cast<long long*>(wb);
  digit_first(p, v, vscale, t, gate, s);
  DigitEpiParams ep{};
  ep.rexp = e1;
  ep.row_b = 1 << 30;
  ep.out0 = a;
  ep.ldo = n1;
  ep.oexp = e2;
  ep.oexp_b = n2;
  ep.inv0 = p->inv;
  ep.inv1 = p->inv + N;
  launch_digit<DG_QUOTIENT>(p, p->T, p->Sy, n2, p->ky, split_grid(n2, p->W.hk).x, ep, gate, s);
  launch_pdl(digit_split_quotients_kernel, split_grid(n2, p->W.hk), dim3(kBlock), 0, s, (const long long*)a, n2, n1,
             (const int*)e1, p->ky, (const double*)p->inv, (const double*)(p->inv + N), (const int*)e2, p->W.d,
             p->W.plane(), p->W.hk, gate);
  ep = DigitEpiParams{};
  ep.rexp = e2;
  ep.row_b = n2;
  ep.out0 = a;  // (W lives on as digits)
  ep.out1 = b;
  ep.ldo = n2;
  ep.oexp = e3;
  ep.oexp_b = n1;
  launch_digit<DG_FIXED>(p, p->W, p->Sx, n1, p->kx, split_grid(p->Y.rows, p->Y.hk).x, ep, gate, s);
  launch_split_fixed(p->Y, a, b, n1, n2, e2, p->kx, e3, gate, s);
  ep = DigitEpiParams{};
  ep.rexp = e3;
  ep.row_b = n1;
  ep.out0 = z;
  ep.ldo = n1;
  ep.phi = phi;
  launch_digit<DG_COMBINE>(p, p->Y, p->Sy, n2, p->ky, fold_blocks(n1, n2), ep, gate, s);
}

void digit_dst2(DigitPlan* p, const double* v, double* out, double* t, cudaStream_t s) {
  digit_first(p, v, nullptr, t, nullptr, s);
  DigitEpiParams ep{};
  ep.rexp = p->exps + p->n2;
  ep.row_b = 1 << 30;
  ep.out0 = out;
  ep.ldo = p->n1;
  launch_digit<DG_STORE>(p, p->T, p->Sy, p->n2, p->ky, p->n2, ep, nullptr, s);  // (another call's split)
}

// ---- the operator ------------------------------------------------------------
struct DigitOperator {
  int n1 = 0, n2 = 0;
  DigitMat Tx, Ty, R, C;  // [U | V] of each axis; the rows and the columns of z
  int* exps = nullptr;     // n2 (rows), n1 (columns)
  int* err = nullptr;
  int* gave_up = nullptr;
  // the parameters, on the device (captured launches read them where they are):
  double* near = nullptr;  // 1 - t0x - t0y, t1x, t1y
  int* kexp = nullptr;     // the scales of the two products
  long long* tq = nullptr;
  void* mem = nullptr;
  long long wait_cycles = kWaitCycles;
};

// [2U | 2V] of t without its first two entries; *kexp the scale of a product with it.
static bool build_toeplitz(DigitOperator* p, DigitMat* T, const std::vector<double>& t, int* kexp, cudaStream_t s) {
  const int n = (int)t.size();
  double big = 0.0;
  for (int k = 2; k < n; ++k) big = std::fmax(big, std::fabs(t[k]));
  int E = 0;
  std::frexp(big, &E);  // |t_k| < 2^E
  std::vector<long long> q(n, 0);
  for (int extra = 0; extra < 3; ++extra) {
    const int sh = 54 - (E + extra);  // |2U|, |2V| <= 2^55
    for (int k = 2; k < n; ++k) q[k] = std::llround(std::ldexp(t[k], sh));
    int rowsum = 0;
    if (cudaMemcpyAsync(p->tq, q.data(), n * sizeof(long long), cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaMemsetAsync(p->err + 1, 0, sizeof(int), s) != cudaSuccess)
      return false;
    digit_toeplitz_kernel<<<T->rows, 256, 0, s>>>(p->tq, n, T->d, T->plane(), T->hk, p->err + 1);
    if (cudaMemcpyAsync(&rowsum, p->err + 1, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
      return false;
    // z = z_q 2^(E_z - 1077), 2U = U_q 2^-sh, sum z U = W 2^(9 + 49 - 1) 2^(E_z - 1077 - sh)
    *kexp = 57 - 1077 - sh;
    if (64LL * rowsum <= (1LL << 24)) return true;
  }
  return false;
}

bool digit_operator_params(DigitOperator* p, const std::vector<double>& tx, const std::vector<double>& ty,
                           cudaStream_t s) {
  int k[2];
  if (!build_toeplitz(p, &p->Tx, tx, &k[0], s) || !build_toeplitz(p, &p->Ty, ty, &k[1], s)) return false;
  const double near[3] = {1.0 - tx[0] - ty[0], tx.size() > 1 ? tx[1] : 0.0, ty.size() > 1 ? ty[1] : 0.0};
  return cudaMemcpyAsync(p->near, near, sizeof(near), cudaMemcpyHostToDevice, s) == cudaSuccess &&
         cudaMemcpyAsync(p->kexp, k, sizeof(k), cudaMemcpyHostToDevice, s) == cudaSuccess &&
         cudaStreamSynchronize(s) == cudaSuccess;
}

int digit_operator_create(DigitOperator** out, int n1, int n2, int* gave_up, cudaStream_t s) {
  *out = nullptr;
  if (!digit_sizes_ok(n1, n2)) return RSFDE_EINVAL;
  DigitOperator* p = new (std::nothrow) DigitOperator();
  if (!p) return RSFDE_ENOMEM;
  p->gave_up = gave_up;
  p->n1 = n1;
  p->n2 = n2;
  const int h1 = pad16((n1 + 1) / 2), h2 = pad16((n2 + 1) / 2);
  size_t off[5] = {0, 0, 0, 0, 0};
  DigitMat* mats[4] = {&p->Tx, &p->Ty, &p->R, &p->C};
  const int rows[4] = {(n1 + 1) / 2, (n2 + 1) / 2, n2, n1}, hk[4] = {h1, h2, h1, h2};
  for (int k = 0; k < 4; ++k) {
    mats[k]->rows = rows[k];
    mats[k]->hk = hk[k];
    off[k + 1] = off[k] + (mats[k]->plane() * kDgDigits * 2 + 255) / 256 * 256;
  }
  const size_t se = ((size_t)(n1 + n2) * sizeof(int) + 255) / 256 * 256;
  if (cudaMalloc(&p->mem, off[4] + se + 256 + kDgMaxN * sizeof(long long)) != cudaSuccess) {
    take_launch_error();
    delete p;
    return RSFDE_ENOMEM;
  }
  uint8_t* b = static_cast<uint8_t*>(p->mem);
  for (int k = 0; k < 4; ++k) mats[k]->d = reinterpret_cast<__nv_bfloat16*>(b + off[k]);
  p->exps = reinterpret_cast<int*>(b + off[4]);
  p->err = reinterpret_cast<int*>(b + off[4] + se);
  p->near = reinterpret_cast<double*>(b + off[4] + se + 64);
  p->kexp = reinterpret_cast<int*>(b + off[4] + se + 128);
  p->tq = reinterpret_cast<long long*>(b + off[4] + se + 256);
  bool good = cudaMemsetAsync(p->err, 0, 256, s) == cudaSuccess;
  good = good && digit_map(&p->Tx, &p->Tx.map[0], kDgBM, 1) && digit_map(&p->C, &p->C.map[0], kDgBM, 1);
  for (DigitMat* m : {&p->R, &p->Ty})
    for (int k = 0; k < 3; ++k) good = good && digit_map(m, &m->map[k], 64 >> k, kDgDigits);
  if (!good) {
    take_launch_error();
    digit_operator_destroy(p);
    return RSFDE_ECUDA;
  }
  *out = p;
  return RSFDE_OK;
}

void digit_operator_destroy(DigitOperator* p) {
  if (!p) return;
  if (p->mem) cudaFree(p->mem);
  delete p;
}
void digit_operator_set_wait(DigitOperator* p, long long cycles) {
  if (p) p->wait_cycles = cycles > 0 ? cycles : kWaitCycles;
}

template <typename Tin, int CPB>
static void launch_fold(DigitOperator* p, const Tin* z, double* pre, const int* gate, cudaStream_t s) {
  const int n1 = p->n1, n2 = p->n2, rblocks = fold_rblocks(n1, n2), smem = CPB * (n2 + 1) * (int)sizeof(double);
  auto k = digit_fold_kernel<Tin, CPB>;
  // (always, and always the largest: the limit is the function's, for every context, and the
  // kernel's static shared memory counts towards the 48 KB that need none)
  raise_smem_limit((const void*)k, CPB * (kDgMaxN + 1) * (int)sizeof(double));
  launch_pdl(k, dim3(fold_blocks(n1, n2)), dim3(256), smem, s, z, n1, n2, rblocks,
             (const double*)p->near, pre, p->R.d, p->R.plane(), p->R.hk, p->exps, p->C.d, p->C.plane(), p->C.hk,
             p->exps + n2, p->err, gate);
}

template <typename Tin>
void digit_apply_M(DigitOperator* p, const Tin* z, double* w, const uint8_t* phi, double pen, double* pre,
                   const int* gate, cudaStream_t s) {
  const int n1 = p->n1, n2 = p->n2;
  if (fold_cols(n1) == 4) launch_fold<Tin, 4>(p, z, pre, gate, s);
  else launch_fold<Tin, 2>(p, z, pre, gate, s);
  DigitEpiParams ep{};
  ep.rexp = p->exps;
  ep.kexp_dev = p->kexp;
  ep.row_b = 1 << 30;
  ep.pre = pre;
  ep.out0 = pre;
  ep.ldo = n1;
  launch_digit<DG_ROWS>(p, p->Tx, p->R, n1, 0, 0, ep, gate, s);
  ep.rexp = p->exps + n2;
  ep.kexp_dev = p->kexp + 1;
  ep.out0 = w;
  ep.phi = phi;
  ep.z = z;
  ep.z_float = sizeof(Tin) == 4;
  ep.pen = pen;
  launch_digit<DG_COLS>(p, p->C, p->Ty, n2, 0, fold_blocks(n1, n2), ep, gate, s);
}
template void digit_apply_M<double>(DigitOperator*, const double*, double*, const uint8_t*, double, double*,
                                    const int*, cudaStream_t);
template void digit_apply_M<float>(DigitOperator*, const float*, double*, const uint8_t*, double, double*, const int*,
                                   cudaStream_t);

template void digit_precond<double>(DigitPlan*, const double*, const double*, double*, const uint8_t*, double*,
                                    double*, double*, const int*, cudaStream_t);
template void digit_precond<df>(DigitPlan*, const df*, const double*, double*, const uint8_t*, double*, double*,
                                double*, const int*, cudaStream_t);
template void digit_precond<float>(DigitPlan*, const float*, const double*, double*, const uint8_t*, double*, double*,
                                   double*, const int*, cudaStream_t);

}  // namespace rsfde
