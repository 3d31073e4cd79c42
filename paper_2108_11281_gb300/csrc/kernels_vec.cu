// Vector-block kernels: noise generation, precision conversion and column scaling
// (dot products and multi-AXPY are in kernels_dots.cu).
// Vector blocks are [row][k] with the k columns (independent right-hand
// sides / samples) innermost, so a warp touches consecutive columns of one row.
#include <algorithm>
#include <atomic>

#include "mlmc_internal.cuh"

namespace mlmc {

void check_cuda(cudaError_t e, const char *where) {
  if (e != cudaSuccess) throw cuda_error{e, where};
}

unsigned resident_grid(size_t units, int per_sm) {
  static std::atomic<int> sms_of[64];              // SM count per device ordinal, 0 = not looked up
  int dev = 0;
  MLMC_CUDA(cudaGetDevice(&dev));
  int sms = dev < 64 ? sms_of[dev].load(std::memory_order_relaxed) : 0;
  if (sms == 0) {
    MLMC_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    if (dev < 64) sms_of[dev].store(sms, std::memory_order_relaxed);
  }
  const size_t g = std::min(units, (size_t)sms * (size_t)per_sm);
  return (unsigned)std::max<size_t>(g, 1);
}

// ------------------------------------------------------------------ Philox
// Philox4x64-10 (Salmon, Moraes, Dror, Shaw, SC'11): 10 rounds of two
// 64x64->128-bit products, key bumped by two Weyl constants between rounds.
struct u64x4 { uint64_t v[4]; };

__device__ inline u64x4 philox4x64_10(u64x4 c, uint64_t k0, uint64_t k1) {
  const uint64_t M0 = 0xD2E7470EE14C6C93ull, M1 = 0xCA5A826395121157ull;
  const uint64_t W0 = 0x9E3779B97F4A7C15ull, W1 = 0xBB67AE8584CAA73Bull;
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r > 0) { k0 += W0; k1 += W1; }
    uint64_t lo0 = M0 * c.v[0], hi0 = __umul64hi(M0, c.v[0]);
    uint64_t lo1 = M1 * c.v[2], hi1 = __umul64hi(M1, c.v[2]);
    u64x4 o;
    o.v[0] = hi1 ^ c.v[1] ^ k0;
    o.v[1] = lo1;
    o.v[2] = hi0 ^ c.v[3] ^ k1;
    o.v[3] = lo0;
    c = o;
  }
  return c;
}

// kind 0 = Rademacher (256 rows per counter), 1 = Z4 (128 rows per counter).
// key = (seed, key_hi), counter = (row_block, first_sample + col, 0, 0).
template <class T>
__global__ void k_noise(int kind, uint64_t seed, uint64_t key_hi, uint64_t first_sample, size_t n,
                        int k, T *out) {
  const int rows_per = kind == 0 ? 256 : 128;
  size_t nblk = (n + rows_per - 1) / rows_per;
  size_t total = nblk * (size_t)k;
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total;
       t += (size_t)gridDim.x * blockDim.x) {
    int col = (int)(t % k);
    size_t blk = t / k;
    u64x4 c = {{(uint64_t)blk, first_sample + (uint64_t)col, 0ull, 0ull}};
    u64x4 w = philox4x64_10(c, seed, key_hi);
    size_t row0 = blk * rows_per;
    if (kind == 0) {
      for (int q = 0; q < 4; ++q)
        for (int b = 0; b < 64; ++b) {
          size_t row = row0 + q * 64 + b;
          if (row < n) {
            double v = ((w.v[q] >> b) & 1ull) ? -1.0 : 1.0;
            out[row * k + col] = make<T>(v, 0.0);
          }
        }
    } else {
      for (int q = 0; q < 4; ++q)
        for (int b = 0; b < 32; ++b) {
          size_t row = row0 + q * 32 + b;
          if (row < n) {
            int v = (int)((w.v[q] >> (2 * b)) & 3ull);   // x = i^v
            double r = v == 0 ? 1.0 : v == 2 ? -1.0 : 0.0;
            double i = v == 1 ? 1.0 : v == 3 ? -1.0 : 0.0;
            out[row * k + col] = make<T>(r, i);
          }
        }
    }
  }
}

void launch_noise(int kind, uint64_t seed, uint64_t key_hi, uint64_t first_sample, size_t n, int k,
                  DType t, void *out, cudaStream_t s) {
  size_t nblk = (n + (kind == 0 ? 255 : 127)) / (kind == 0 ? 256 : 128);
  unsigned g = grid_for(nblk * k, 128, 152 * 64);
  MLMC_DISPATCH(t, T, k_noise<T><<<g, 128, 0, s>>>(kind, seed, key_hi, first_sample, n, k, (T *)out));
  MLMC_LAUNCH_CHECK("k_noise");
}

// ------------------------------------------------------------------ convert / fill
template <class To, class From>
__global__ void k_convert(To *dst, const From *src, size_t count) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count;
       i += (size_t)gridDim.x * blockDim.x)
    dst[i] = cvt<To, From>(src[i]);
}

void launch_convert(DType to, void *dst, DType from, const void *src, size_t count, cudaStream_t s) {
  unsigned g = grid_for(count, 256);
  if (to == F32 && from == F64) k_convert<float, double><<<g, 256, 0, s>>>((float *)dst, (const double *)src, count);
  else if (to == F64 && from == F32) k_convert<double, float><<<g, 256, 0, s>>>((double *)dst, (const float *)src, count);
  else if (to == C32 && from == C64) k_convert<cfloat, cdouble><<<g, 256, 0, s>>>((cfloat *)dst, (const cdouble *)src, count);
  else if (to == C64 && from == C32) k_convert<cdouble, cfloat><<<g, 256, 0, s>>>((cdouble *)dst, (const cfloat *)src, count);
  else if (to == from) {
    MLMC_CUDA(cudaMemcpyAsync(dst, src, count * dtype_size(to), cudaMemcpyDeviceToDevice, s));
    return;
  } else throw cuda_error{cudaErrorInvalidValue, "launch_convert: field mismatch"};
  MLMC_LAUNCH_CHECK("k_convert");
}

template <class T>
__global__ void k_fill_one(T *dst, size_t count) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x)
    dst[i] = make<T>(1.0, 0.0);
}

void launch_fill_one(DType t, void *dst, size_t count, cudaStream_t s) {
  MLMC_DISPATCH(t, T, k_fill_one<T><<<grid_for(count, 256), 256, 0, s>>>((T *)dst, count));
  MLMC_LAUNCH_CHECK("k_fill_one");
}

// out = a - b (elementwise)
template <class T>
__global__ void k_sub(T *out, const T *a, const T *b, size_t count) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x)
    out[i] = a[i] - b[i];
}

void launch_sub(DType t, void *out, const void *a, const void *b, size_t count, cudaStream_t s) {
  MLMC_DISPATCH(t, T, k_sub<T><<<grid_for(count, 256), 256, 0, s>>>((T *)out, (const T *)a, (const T *)b, count));
  MLMC_LAUNCH_CHECK("k_sub");
}

void launch_fill_zero(DType t, void *dst, size_t count, cudaStream_t s) {
  MLMC_CUDA(cudaMemsetAsync(dst, 0, count * dtype_size(t), s));
}

// ------------------------------------------------------------------ column scaling
static unsigned column_grid(size_t total, int k) {
  // threads = a multiple of k, about 4 waves of 152 SMs x 2048 threads at most
  size_t want = (total + 255) / 256;
  size_t cap = 152 * 8;
  size_t g = want < cap ? want : cap;
  if (g < 1) g = 1;
  // round up so that g * 256 is a multiple of k
  size_t per = (size_t)k / std::__gcd((size_t)k, (size_t)256);
  g = ((g + per - 1) / per) * per;
  return (unsigned)g;
}

// y[r][c] = x[r][c] * alpha[c]  (alpha real FP64)
template <class T>
__global__ void __launch_bounds__(256) k_scale_cols(T *y, const T *x, const double *alpha, size_t total, int k) {
  typedef typename real_of<T>::type R;
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  const size_t t0 = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  const R a = (R)alpha[t0 % k];
  for (size_t i = t0; i < total; i += stride) y[i] = rmul(a, x[i]);
}

void launch_scale_cols(DType t, void *y, const void *x, const void *alpha, int, size_t rows, int k,
                       cudaStream_t s) {
  size_t total = rows * (size_t)k;
  unsigned g = column_grid(total, k);
  MLMC_DISPATCH(t, T, k_scale_cols<T><<<g, 256, 0, s>>>((T *)y, (const T *)x, (const double *)alpha, total, k));
  MLMC_LAUNCH_CHECK("k_scale_cols");
}

// ------------------------------------------------------------------ arithmetic rate probe
// Eight independent FMA chains per thread (x <- x a + b; or additions x <- x + b),
// enough to keep the FP64 or FP32 pipes busy; the result is stored only under a condition that never
// holds, so the chains are not removed.  Measures the ALU ceiling that FP64
// kernels (apply, Arnoldi) meet on this GPU.
template <class T, bool ADD>
__global__ void __launch_bounds__(256) k_fma_rate(T *out, int iters, T a, T b) {
  T x[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) x[q] = (T)(threadIdx.x + q) * (T)1e-3;
  for (int i = 0; i < iters; ++i) {
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] = ADD ? x[q] + b : fma(x[q], a, b);
  }
  T sum = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) sum += x[q];
  if (sum == (T)-1.2345) out[blockIdx.x * blockDim.x + threadIdx.x] = sum;
}

void launch_fma_rate(DType t, int add, void *out, int blocks, int iters, cudaStream_t s) {
  if (t == F64 && add)
    k_fma_rate<double, true><<<blocks, 256, 0, s>>>((double *)out, iters, 0.999999, 1e-7);
  else if (t == F64)
    k_fma_rate<double, false><<<blocks, 256, 0, s>>>((double *)out, iters, 0.999999, 1e-7);
  else
    k_fma_rate<float, false><<<blocks, 256, 0, s>>>((float *)out, iters, 0.999999f, 1e-7f);
  MLMC_LAUNCH_CHECK("k_fma_rate");
}

// Bandwidth probe: `passes` copies of n 16-byte packs between two buffers, a -> b, then
// b -> a, ... in one launch (every thread keeps its indices, so no pass reads what another
// thread writes); an L2-resident pair gives the L2 ceiling of the small coarse-level kernels
// without launch overhead in the measurement.
__global__ void __launch_bounds__(256) k_copy16(uint4 *a, uint4 *b, size_t n, int passes) {
  for (int p = 0; p < passes; ++p) {
    const uint4 *src = (p & 1) ? b : a;
    uint4 *dst = (p & 1) ? a : b;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
      dst[i] = src[i];
  }
}

void launch_copy16(void *a, void *b, size_t n16, int passes, int blocks, cudaStream_t s) {
  k_copy16<<<blocks, 256, 0, s>>>((uint4 *)a, (uint4 *)b, n16, passes);
  MLMC_LAUNCH_CHECK("k_copy16");
}

}  // namespace mlmc
