// Nearest-neighbour block-stencil kernels: operator apply / residual (the generic
// d x d block stencil, its row-split form for d = 8 and the constant-coefficient
// Example 5.1 operator) and red-black block Gauss-Seidel half-sweeps.  Transfers
// and the setup filter are in kernels_transfer.cu, the 9-point levels of the
// bilinear hierarchy in kernels_bilinear.cu.
//
// Layout: the operator of a level is coef[site][dir][r][c] (dir 0 self, 1 +x,
// 2 -x, 3 +y, 4 -y; periodic indexing, Dirichlet boundaries are zero blocks);
// vector blocks are [site][dof][k] with the k right-hand sides innermost, so
// the k threads of one site read consecutive addresses and share the
// coefficient loads through L1.
#include <cstring>
#include <type_traits>

#include "mlmc_internal.cuh"

namespace mlmc {

// ------------------------------------------------------------------ apply / residual
// One thread per (site, VEC consecutive columns): the d x d coefficient blocks
// are loaded once per VEC columns, the vector entries as 16-byte packs.
template <class T, int VEC> struct alignas(sizeof(T) * VEC) Pack { T v[VEC]; };

// Row r of a d x d coefficient block, with 16-byte loads when the row allows.
template <class T, int D>
__device__ inline void load_row(const T *__restrict__ p, T out[D]) {
  if constexpr ((D * sizeof(T)) % 16 == 0) {
    const uint4 *q = reinterpret_cast<const uint4 *>(p);
#pragma unroll
    for (int i = 0; i < (int)(D * sizeof(T) / 16); ++i) {
      uint4 w = __ldg(q + i);
      memcpy(&out[i * (16 / sizeof(T))], &w, 16);
    }
  } else {
#pragma unroll
    for (int i = 0; i < D; ++i) out[i] = p[i];
  }
}

template <class T, int D, int VEC>
__device__ __forceinline__ void stencil_body(const T *__restrict__ coef, const T *__restrict__ x,
                                             const T *__restrict__ b, T *__restrict__ y, int nx, int ny, int kv,
                                             int mode, int j, int t) {
  // j = lattice row; t = (site i of the row, pack c of VEC columns)
  typedef Pack<T, VEC> V;
  if (t < nx * kv) {
    const int i = t / kv, c = t - (t / kv) * kv;
    const int s = j * nx + i;
    int nb[5];
    nb[0] = s;
    nb[1] = j * nx + (i + 1 == nx ? 0 : i + 1);
    nb[2] = j * nx + (i == 0 ? nx - 1 : i - 1);
    nb[3] = (j + 1 == ny ? 0 : j + 1) * nx + i;
    nb[4] = (j == 0 ? ny - 1 : j - 1) * nx + i;
    T acc[D][VEC];
#pragma unroll
    for (int r = 0; r < D; ++r)
#pragma unroll
      for (int u = 0; u < VEC; ++u) acc[r][u] = zero<T>();
#pragma unroll
    for (int dir = 0; dir < 5; ++dir) {
      const T *B = coef + ((size_t)s * 5 + dir) * D * D;
      const V *xs = (const V *)x + (size_t)nb[dir] * D * kv + c;
      V xq[D];
#pragma unroll
      for (int q = 0; q < D; ++q) xq[q] = xs[(size_t)q * kv];
#pragma unroll
      for (int r = 0; r < D; ++r) {
        T row[D];
        load_row<T, D>(B + r * D, row);
#pragma unroll
        for (int q = 0; q < D; ++q)
#pragma unroll
          for (int u = 0; u < VEC; ++u) acc[r][u] = madd(acc[r][u], row[q], xq[q].v[u]);
      }
    }
    size_t o = (size_t)s * D * kv + c;
#pragma unroll
    for (int r = 0; r < D; ++r) {
      V out;
      if (mode) {
        V bb = ((const V *)b)[o + (size_t)r * kv];
#pragma unroll
        for (int u = 0; u < VEC; ++u) out.v[u] = bb.v[u] - acc[r][u];
      } else {
#pragma unroll
        for (int u = 0; u < VEC; ++u) out.v[u] = acc[r][u];
      }
      ((V *)y)[o + (size_t)r * kv] = out;
    }
  }
}

// Threads per block of the generic kernels.  FP64 is bound by the FP64 pipe, two operations per
// clock and SM, so what counts is that every SM gets the same number of threads: blocks of 32
// (the 48^2 x 4 level at 21 columns: smoother half-sweep 7.1 us and apply 11.7 us with 256, whose
// 96 and 192 blocks load some of 152 SMs twice; a 192^2 FP64 solve takes 8.34 ms with 256, 7.97
// with 64 and 7.77 with 32).  One dof per site has so little arithmetic that the loads count, and 32
// blocks of 32 threads are half of what an SM holds: 128 (128^2 x 1 at 32 columns, apply: 10.3 us
// with 32, 8.4 with 128; 128^2 x 2 8.4 and 8.4).
template <class T, int D> __host__ __device__ constexpr int gen_threads() {
  return sizeof(typename real_of<T>::type) == 8 ? (D == 1 ? 128 : 32) : 256;
}

// Resident grid striding over the units (row j, chunk of one block's threads of the row): the
// FP64 block applies are bound by the FP64 pipe, which one block per unit leaves idle between
// blocks.
template <class T, int D, int VEC>
__global__ void __launch_bounds__(gen_threads<T, D>()) k_stencil(const T *__restrict__ coef, const T *__restrict__ x,
                                                 const T *__restrict__ b, T *__restrict__ y, int nx, int ny, int kv,
                                                 int mode, int bpr) {
  const int units = bpr * ny;
  for (int u = blockIdx.x; u < units; u += gridDim.x) {
    const int j = u / bpr;
    stencil_body<T, D, VEC>(coef, x, b, y, nx, ny, kv, mode, j, (u - j * bpr) * gen_threads<T, D>() + threadIdx.x);
  }
}

// The same in blocks of 128 threads pinned at 8 per SM (<= 64 registers), for FP32
// blocks with d = 4 (the aggregation levels of the Laplace hierarchy), like the
// block smoother: both are load-latency bound.  The grid is resident (8 blocks per
// SM) and strides over the units (row j, chunk of 128 threads of the row), in
// row order, so the rows in flight stay a narrow band (vertical neighbours from L2).
// rev = 1 walks the rows from the last: the apply follows a smoothing half-sweep that
// ended there, whose last writes are then still in L2 when they are read.
template <class T, int D, int VEC>
__global__ void __launch_bounds__(128, 8) k_stencil_p(const T *__restrict__ coef, const T *__restrict__ x,
                                                      const T *__restrict__ b, T *__restrict__ y, int nx, int ny,
                                                      int kv, int mode, int bpr, int rev) {
  const int units = bpr * ny;
  for (int u0 = blockIdx.x; u0 < units; u0 += gridDim.x) {
    const int u = rev ? units - 1 - u0 : u0;
    const int j = u / bpr;
    stencil_body<T, D, VEC>(coef, x, b, y, nx, ny, kv, mode, j, (u - j * bpr) * 128 + threadIdx.x);
  }
}

// columns per thread for the generic kernels: 16-byte packs for FP32 data on
// small blocks; fewer columns per thread as d grows, to bound registers
template <class T, int D> struct gen_vec { static const int v = 1; };
template <int D> struct gen_vec<float, D> { static const int v = D <= 4 ? 4 : 2; };
template <int D> struct gen_vec<cfloat, D> { static const int v = D <= 2 ? 2 : 1; };

#define MLMC_DDISPATCH(d, DD, ...)                       \
  switch (d) {                                           \
    case 1: { const int DD = 1; __VA_ARGS__; } break;    \
    case 2: { const int DD = 2; __VA_ARGS__; } break;    \
    case 4: { const int DD = 4; __VA_ARGS__; } break;    \
    case 8: { const int DD = 8; __VA_ARGS__; } break;    \
    default: throw cuda_error{cudaErrorInvalidValue, "unsupported dofs per site"}; \
  }

// Row-split kernels for large site blocks (d >= 8, the small coarse lattices of the Wilson
// hierarchy): one thread per (RPT rows of a site, CV consecutive columns); block = 32 x CV
// columns x D / RPT row groups of one site.  These levels live in L2 and a launch is a few
// microseconds, so what counts is one round trip to L2: the site's coefficient blocks (one
// contiguous run) go to shared memory by cp.async while every thread loads its vector entries
// of all (or, with wide packs, some) of the neighbours into registers.  Beside that FP32 is
// bound by the load unit: a broadcast of 16 coefficient bytes takes it as long as 32 lanes'
// 16-byte vector entries, so two rows per thread share the vector entries and CV = 2 halves
// the coefficient reads per column.  FP64 is bound by its arithmetic and keeps one row.
// Wilson 128^2, level 2 (32^2 sites, complex FP32), one row per thread and coefficients through
// the cache before: smoother sweep 16.4 -> 12.3 us at k = 32 and 27.7 -> 16.6 us at k = 128,
// apply 8.2 -> 6.2 and 19.5 -> 14.4 us, 12.3 with the smoother's madd4 (two rows per thread alone:
// 18.5 us per sweep at both).
template <class T> constexpr int rows_rpt() { return sizeof(typename real_of<T>::type) == 4 ? 2 : 1; }

// Real FP64 with more blocks than SMs reads the coefficients through the cache instead (STAGED
// false): its arithmetic fills the FP64 pipe only with other blocks beside a block that waits, and
// with all neighbours' entries in registers two fit on an SM.  128^2 x 8 sites, FP64: apply 317 us
// staged and 285 through the cache at k = 32, 1228 and 1119 at k = 128, smoother sweep 1183 and 1097;
// 32^2 x 8: apply 25.8 and 22.5 at k = 32; 24^2 x 8: sweep 18.3 and 16.6.  Fewer blocks wait for one
// round trip to L2: 8^2 x 8 at k = 64 9.2 and 10.3, sweep of 16^2 x 8 at k = 21 12.5 and 14.4.
template <class T> static bool rows_staged(size_t blocks) { return !std::is_same<T, double>::value || blocks <= 152; }
// go(CV, STAGED) with both as compile-time constants
template <class T, class F> static void rows_dispatch(int k, int sites, F &&go) {
  const int cv = (k % 2 == 0 && k >= 64) ? 2 : 1;        // two columns per thread on blocks of at least 64 even columns
  const dim3 grid((k / cv + 31) / 32, sites);
  auto with_cv = [&](auto c) {
    if constexpr (std::is_same<T, double>::value)
      if (!rows_staged<T>((size_t)grid.x * grid.y)) return go(c, std::false_type(), grid);
    go(c, std::true_type(), grid);
  };
  if (cv == 2) with_cv(std::integral_constant<int, 2>());
  else with_cv(std::integral_constant<int, 1>());
}

__device__ __forceinline__ void copy16_async(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// `bytes` (a multiple of 16) from 16-byte aligned src to dst, by the block's threads
__device__ __forceinline__ void block_copy_async(void *dst, const void *src, int bytes, int tid, int threads) {
  for (int e = tid * 16; e < bytes; e += threads * 16) copy16_async((char *)dst + e, (const char *)src + e);
}

// acc[r] +- sum over NDIR neighbour blocks of rows r0 + r (blk: [NDIR][D][D], STAGED in shared
// memory) times their x, XB neighbours' entries in flight at a time.  ready(): STAGED, called after
// the first loads are issued and before the coefficients are read.  SUB is the smoother's form (msub4).
template <class T, int D, int CV, int RPT, int NDIR, bool SUB, bool STAGED, class F>
__device__ __forceinline__ void rows_accumulate(const T *blk, const T *x, const int nb[NDIR], int r0, int k, int c,
                                                bool live, Pack<T, CV> acc[RPT], F ready) {
  typedef Pack<T, CV> V;
  constexpr int WORDS = D * CV * (int)sizeof(T) / 4;                    // registers of one neighbour
  constexpr int XB = !STAGED ? 1 : WORDS * NDIR <= 80 ? NDIR : WORDS <= 32 ? 2 : 1;   // neighbours in flight
  const int kv = k / CV;
#pragma unroll
  for (int d0 = 0; d0 < NDIR; d0 += XB) {
    V xv[XB][D];
#pragma unroll
    for (int e = 0; e < XB; ++e)
      if (d0 + e < NDIR && live) {
        const V *xs = reinterpret_cast<const V *>(x + (size_t)nb[d0 + e] * D * k + c);
#pragma unroll
        for (int q = 0; q < D; ++q) xv[e][q] = xs[(size_t)q * kv];
      }
    if constexpr (STAGED) {
      asm volatile("" ::: "memory");                                    // the loads stay in front
      if (d0 == 0) ready();
    }
#pragma unroll
    for (int e = 0; e < XB; ++e)
      if (d0 + e < NDIR) {
#pragma unroll
        for (int r = 0; r < RPT; ++r) {
          T row[D];
          const T *src = blk + ((size_t)(d0 + e) * D + r0 + r) * D;
          if constexpr (STAGED) memcpy(row, __builtin_assume_aligned(src, 16), sizeof(row));
          else load_row<T, D>(src, row);
#pragma unroll
          for (int q = 0; q < D; ++q)
#pragma unroll
            for (int u = 0; u < CV; ++u)
              acc[r].v[u] = SUB ? msub4(acc[r].v[u], row[q], xv[e][q].v[u]) : madd(acc[r].v[u], row[q], xv[e][q].v[u]);
        }
      }
  }
}

__device__ __forceinline__ void async_ready() {
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
}

template <class T, int D, int CV, int RPT, bool STAGED>
__global__ void __launch_bounds__(32 * D / RPT) k_stencil_rows(const T *__restrict__ coef, const T *x, const T *b,
                                                               T *y, int nx, int ny, int k, int mode) {
  typedef Pack<T, CV> V;
  __shared__ __align__(16) unsigned char blk_mem[STAGED ? 5 * D * D * sizeof(T) : 16];
  const int s = blockIdx.y;
  const T *blk = STAGED ? (const T *)blk_mem : coef + (size_t)s * 5 * D * D;
  const int i = s % nx, j = s / nx;
  const int r0 = threadIdx.y * RPT;
  const int c = (blockIdx.x * 32 + threadIdx.x) * CV;   // k is a multiple of CV
  const bool live = c < k;
  if constexpr (STAGED)
    block_copy_async(blk_mem, coef + (size_t)s * 5 * D * D, 5 * D * D * (int)sizeof(T), threadIdx.y * 32 + threadIdx.x,
                     32 * D / RPT);
  int nb[5];
  nb[0] = s;
  nb[1] = j * nx + (i + 1 == nx ? 0 : i + 1);
  nb[2] = j * nx + (i == 0 ? nx - 1 : i - 1);
  nb[3] = (j + 1 == ny ? 0 : j + 1) * nx + i;
  nb[4] = (j == 0 ? ny - 1 : j - 1) * nx + i;
  V acc[RPT];
#pragma unroll
  for (int r = 0; r < RPT; ++r)
#pragma unroll
    for (int u = 0; u < CV; ++u) acc[r].v[u] = zero<T>();
  rows_accumulate<T, D, CV, RPT, 5, false, STAGED>(blk, x, nb, r0, k, c, live, acc, async_ready);
  if (!live) return;
#pragma unroll
  for (int r = 0; r < RPT; ++r) {
    const size_t o = ((size_t)s * D + r0 + r) * k + c;
    V out = acc[r];
    if (mode) {
      const V bb = *reinterpret_cast<const V *>(b + o);
#pragma unroll
      for (int u = 0; u < CV; ++u) out.v[u] = bb.v[u] - acc[r].v[u];
    }
    *reinterpret_cast<V *>(y + o) = out;
  }
}

template <class T, int D>
static void stencil_go(const StencilView &A, const void *x, const void *b, void *y, int k, int mode, cudaStream_t s) {
  if constexpr (D >= 8) {
    if (A.nx * A.ny <= 65535) {
      constexpr int RPT = rows_rpt<T>();
      rows_dispatch<T>(k, A.nx * A.ny, [&](auto cv, auto staged, dim3 grid) {
        k_stencil_rows<T, D, decltype(cv)::value, RPT, decltype(staged)::value><<<grid, dim3(32, D / RPT), 0, s>>>(
            (const T *)A.coef, (const T *)x, (const T *)b, (T *)y, A.nx, A.ny, k, mode);
      });
      return;
    }
  }
  constexpr int VW = gen_vec<T, D>::v, TB = gen_threads<T, D>();
  if (VW > 1 && k % VW == 0) {
    int kv = k / VW;
    if constexpr (std::is_same<T, float>::value && D == 4)
    {
      const int bpr = (A.nx * kv + 127) / 128;
      k_stencil_p<T, D, VW><<<resident_grid(bpr * A.ny, 8), 128, 0, s>>>(
          (const T *)A.coef, (const T *)x, (const T *)b, (T *)y, A.nx, A.ny, kv, mode, bpr, 0);
    }
    else {
      const int bpr = (A.nx * kv + TB - 1) / TB;
      static const int occ = blocks_per_sm(k_stencil<T, D, VW>, TB, 0);
      k_stencil<T, D, VW><<<resident_grid((size_t)bpr * A.ny, occ), TB, 0, s>>>(
          (const T *)A.coef, (const T *)x, (const T *)b, (T *)y, A.nx, A.ny, kv, mode, bpr);
    }
  } else {
    const int bpr = (A.nx * k + TB - 1) / TB;
    static const int occ = blocks_per_sm(k_stencil<T, D, 1>, TB, 0);
    k_stencil<T, D, 1><<<resident_grid((size_t)bpr * A.ny, occ), TB, 0, s>>>(
        (const T *)A.coef, (const T *)x, (const T *)b, (T *)y, A.nx, A.ny, k, mode, bpr);
  }
}

// ------------------------------------------------------------------ Example 5.1, constant coefficients
// The four neighbours of site (i, j), each with a flag: present, or outside a
// Dirichlet lattice (periodic lattices wrap).  Straight-line code: no array
// indexed at run time, so nothing goes through local memory.
struct Nbrs {
  int s[4];
  bool on[4];
};

__device__ __forceinline__ Nbrs laplace_nbrs(int i, int j, int nx, int ny, int periodic) {
  Nbrs n;
  const int s = j * nx + i;
  n.on[0] = i + 1 < nx || periodic;
  n.s[0] = i + 1 < nx ? s + 1 : j * nx;
  n.on[1] = i > 0 || periodic;
  n.s[1] = i > 0 ? s - 1 : j * nx + nx - 1;
  n.on[2] = j + 1 < ny || periodic;
  n.s[2] = j + 1 < ny ? s + nx : i;
  n.on[3] = j > 0 || periodic;
  n.s[3] = j > 0 ? s - nx : (ny - 1) * nx + i;
  return n;
}

// Sum of the present neighbours' packs: (x_+x + x_-x) + (x_+y + x_-y), absent ones zero.
template <class T, int VEC>
__device__ __forceinline__ void laplace_nbr_sum(const Pack<T, VEC> *__restrict__ X, const Nbrs &n, int kv, int c,
                                                T sum[VEC]) {
  Pack<T, VEC> v[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (n.on[q]) {
      v[q] = X[(size_t)n.s[q] * kv + c];
    } else {
#pragma unroll
      for (int u = 0; u < VEC; ++u) v[q].v[u] = zero<T>();
    }
  }
#pragma unroll
  for (int u = 0; u < VEC; ++u) sum[u] = (v[0].v[u] + v[1].v[u]) + (v[2].v[u] + v[3].v[u]);
}

// y = diag x - (sum of the in-grid neighbours), r = b - that, or the setup filter's
// y = diag x + scale (sum of the neighbours); VEC columns per thread with 16-byte loads, rows in
// order, so the +-y neighbours of a block are the rows just touched by the blocks before it (L2
// hits).  FP32, and FP64 data of small lattices and narrow blocks; larger ones take
// k_laplace_march (see laplace_fp64).
enum { LAP_APPLY = 0, LAP_RESIDUAL = 1, LAP_JACOBI = 2 };

template <class T, int VEC, int MODE>
__device__ __forceinline__ void laplace_body(const T *__restrict__ x, const T *__restrict__ b, T *__restrict__ y,
                                             int nx, int ny, int kv, T diag, T scale, int periodic, int j, int t) {
  typedef Pack<T, VEC> V;
  if (t >= nx * kv) return;
  const int i = t / kv, c = t - (t / kv) * kv;
  const V *X = (const V *)x;
  const int s = j * nx + i;
  const Nbrs n = laplace_nbrs(i, j, nx, ny, periodic);
  V xc = X[(size_t)s * kv + c];
  T sum[VEC];
  laplace_nbr_sum<T, VEC>(X, n, kv, c, sum);
  V out;
  if (MODE == LAP_RESIDUAL) {
    V bb = ((const V *)b)[(size_t)s * kv + c];
#pragma unroll
    for (int u = 0; u < VEC; ++u) out.v[u] = (bb.v[u] + sum[u]) - diag * xc.v[u];
  } else if (MODE == LAP_JACOBI) {
#pragma unroll
    for (int u = 0; u < VEC; ++u) out.v[u] = diag * xc.v[u] + scale * sum[u];
  } else {
#pragma unroll
    for (int u = 0; u < VEC; ++u) out.v[u] = diag * xc.v[u] - sum[u];
  }
  ((V *)y)[(size_t)s * kv + c] = out;
}

// Resident grid striding over the units (row j, chunk of 256 threads of the row) in row order.
template <class T, int VEC, int MODE>
__global__ void __launch_bounds__(256) k_laplace(const T *__restrict__ x, const T *__restrict__ b, T *__restrict__ y,
                                                 int nx, int ny, int kv, T diag, T scale, int periodic, int bpr) {
  const int units = bpr * ny;
  for (int u = blockIdx.x; u < units; u += gridDim.x) {
    const int j = u / bpr;
    laplace_body<T, VEC, MODE>(x, b, y, nx, ny, kv, diag, scale, periodic, j, (u - j * bpr) * 256 + threadIdx.x);
  }
}

// Threads per block of the half-sweep below.  FP64: small blocks for an even share per SM, but not so
// small that 32 of them, the most an SM holds, leave it half empty (512^2 at 21 columns: sweep 67.8 us
// with 32, 65.7 with 64; 192^2 at 5: 12.3 and 10.0).  FROM_ZERO is a compile-time flag: as an argument
// it cost the FP64 pipe a multiply-add per entry (512^2 at 21 columns: 78.0 us).  The register bound
// keeps 2048 threads on an SM: the FP32 form takes 34 without it (1024^2 x 64: 135 us, 126 with).
template <class T> __host__ __device__ constexpr int lap_threads() { return sizeof(T) == 8 ? 64 : 256; }

// Red-black Gauss-Seidel half-sweep for Example 5.1: x_s = (b_s + sum of neighbours) / diag
// on the sites of `colour`.  other_zero = 1: the other colour holds zeros (not read).
// Colour 1 takes the rows from the last: consecutive half-sweeps alternate direction, so
// each starts on the rows the previous one wrote last.
// FROM_ZERO: the whole first sweep from x = 0 as one pass over colour 1,
// x_1 = (b_1 + sum of b_0 / diag) / diag; colour 0 is left unset (see launch_rbgs_first).
// The grid strides over the units (row, chunk of one block's threads of the row).
template <class T, int VEC, bool FROM_ZERO>
__device__ __forceinline__ void laplace_rbgs_body(T *__restrict__ x, const T *__restrict__ b, int nx, int ny, int kv,
                                                  T dinv, int periodic, int colour, int other_zero, int j, int t) {
  typedef Pack<T, VEC> V;
  const int i0 = (j + colour) & 1;
  const int hx = (nx - i0 + 1) >> 1;      // sites of this colour in row j (odd nx too)
  if (t >= hx * kv) return;
  const int m = t / kv, c = t - (t / kv) * kv;
  const int i = 2 * m + i0;
  const int s = j * nx + i;
  V *X = (V *)x;
  V acc = ((const V *)b)[(size_t)s * kv + c];
  if (!other_zero) {
    const Nbrs n = laplace_nbrs(i, j, nx, ny, periodic);
    T sum[VEC];
    laplace_nbr_sum<T, VEC>(FROM_ZERO ? (const V *)b : X, n, kv, c, sum);
#pragma unroll
    for (int u = 0; u < VEC; ++u) acc.v[u] = FROM_ZERO ? madd(acc.v[u], dinv, sum[u]) : acc.v[u] + sum[u];
  }
#pragma unroll
  for (int u = 0; u < VEC; ++u) acc.v[u] = acc.v[u] * dinv;
  X[(size_t)s * kv + c] = acc;
}

template <class T, int VEC, bool FROM_ZERO>
__global__ void __launch_bounds__(lap_threads<T>(), 2048 / lap_threads<T>())
    k_laplace_rbgs(T *__restrict__ x, const T *__restrict__ b, int nx, int ny, int kv, T dinv, int periodic, int colour,
                   int other_zero, int bpr) {
  const int units = bpr * ny;
  for (int u = blockIdx.x; u < units; u += gridDim.x) {
    const int jr = u / bpr;
    laplace_rbgs_body<T, VEC, FROM_ZERO>(x, b, nx, ny, kv, dinv, periodic, colour, other_zero,
                                         colour ? ny - 1 - jr : jr, (u - jr * bpr) * lap_threads<T>() + threadIdx.x);
  }
}

template <class T>
static int laplace_vec(int k) {
  const int v = 16 / (int)sizeof(T);
  return k % v == 0 ? v : 1;
}

// ------------------------------------------------------------------ Example 5.1 in FP64
// Bound by the FP64 pipe (1.7 - 2 operations per clock and SM).  The neighbour sum of site
// (i, j) is u(i, j) + u(i - 1, j - 1) with u(i, j) = x(i + 1, j) + x(i, j + 1): each u serves two
// sites, so a site costs about two additions and one multiply-add instead of three and one.
// A thread holds a strip of MP lattice columns (one 16-byte pack of right-hand sides) and walks
// up JB rows, keeping the last row's u; a site's x is loaded about 1.5 times instead of five.
// The additions are issued as multiply-adds by 1 (same result; 0.63 against 0.53 T/s).
// 1024^2 x 64: 402 us (3.3 operations per site: 350 us at the measured rate), 531 us with the
// neighbour sum per site.
constexpr int MP = 4;

template <int VEC, int MODE>
__global__ void __launch_bounds__(128) k_laplace_march(const double *__restrict__ x, const double *__restrict__ b,
                                                       double *__restrict__ y, int nx, int ny, int kv, double diag,
                                                       double scale, double one, int periodic, int JB) {
  typedef Pack<double, VEC> V;
  const unsigned strips = (nx + MP - 1) / MP, segs = (ny + JB - 1) / JB;
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= strips * segs * (unsigned)kv) return;
  const unsigned q = t / (unsigned)kv;
  const int c = (int)(t - q * (unsigned)kv);
  const int i0 = (int)(q % strips) * MP, j0 = (int)(q / strips) * JB, j1 = min(ny, j0 + JB);
  // lattice columns i0 - 1 .. i0 + MP: offsets into a row; a column outside a Dirichlet lattice, or
  // more than one past the end, reads as zero
  int col[MP + 2];
  unsigned on = 0;
#pragma unroll
  for (int u = 0; u < MP + 2; ++u) {
    int i = i0 + u - 1;
    bool ok = i >= 0 && i < nx;
    if (!ok && periodic && i <= nx) {
      i = i < 0 ? nx - 1 : 0;
      ok = true;
    }
    on |= (unsigned)ok << u;
    col[u] = (ok ? i : 0) * kv + c;
  }
  const V *X = (const V *)x;
  auto load = [&](int j, V v[MP + 2]) {
    bool ok = j >= 0 && j < ny;
    if (!ok && periodic) {
      j = j < 0 ? ny - 1 : 0;
      ok = true;
    }
    const V *row = X + (size_t)(ok ? j : 0) * nx * kv;
#pragma unroll
    for (int u = 0; u < MP + 2; ++u) {
      if (ok && (on >> u & 1)) {
        v[u] = row[col[u]];
      } else {
#pragma unroll
        for (int e = 0; e < VEC; ++e) v[u].v[e] = 0.0;
      }
    }
  };
  V cur[MP + 2], nxt[MP + 2], up[MP];
  load(j0 - 1, nxt);
  load(j0, cur);
#pragma unroll
  for (int m = 0; m < MP; ++m)
#pragma unroll
    for (int e = 0; e < VEC; ++e) up[m].v[e] = fma(nxt[m + 1].v[e], one, cur[m].v[e]);
#pragma unroll 2
  for (int j = j0; j < j1; ++j) {
    load(j + 1, nxt);
    V u[MP + 1];                              // u(i0 - 1 + m, j)
#pragma unroll
    for (int m = 0; m <= MP; ++m)
#pragma unroll
      for (int e = 0; e < VEC; ++e) u[m].v[e] = fma(cur[m + 1].v[e], one, nxt[m].v[e]);
    const size_t row = (size_t)j * nx * kv;
#pragma unroll
    for (int p = 0; p < MP; ++p) {
      if (i0 + p < nx) {
        V out;
        if (MODE == LAP_RESIDUAL) out = ((const V *)b)[row + col[p + 1]];
#pragma unroll
        for (int e = 0; e < VEC; ++e) {
          const double sum = fma(u[p + 1].v[e], one, up[p].v[e]), xc = cur[p + 1].v[e];
          if (MODE == LAP_APPLY) out.v[e] = fma(diag, xc, -sum);
          if (MODE == LAP_RESIDUAL) out.v[e] = fma(-diag, xc, fma(sum, one, out.v[e]));
          if (MODE == LAP_JACOBI) out.v[e] = fma(scale, sum, diag * xc);
        }
        ((V *)y)[row + col[p + 1]] = out;
      }
    }
#pragma unroll
    for (int m = 0; m < MP; ++m) up[m] = u[m];
#pragma unroll
    for (int m = 0; m < MP + 2; ++m) cur[m] = nxt[m];
  }
}

template <int MODE>
static void laplace_march(const StencilView &A, const void *x, const void *b, void *y, int k, double diag, double scale,
                          cudaStream_t s) {
  const int vec = k % 2 == 0 ? 2 : 1, kv = k / vec;
  const size_t strips = (A.nx + MP - 1) / MP;
  // Rows per walk: the smallest time of the busiest SM, blocks x (13 operations per row and 4
  // before the first, for the strip and pack), with at least four blocks per SM where any walk
  // allows it; the longer walk where that is equal.  Powers of two alone left 937 blocks on 152
  // SMs: 768^2 x 13 took 75.8 us.
  int JB = 2;
  size_t best = ~(size_t)0;
  for (int jb = 64; jb >= 2; --jb) {
    const size_t blocks = (strips * ((A.ny + jb - 1) / jb) * kv + 127) / 128;
    const size_t cost = (blocks + 151) / 152 * (13 * jb + 4);
    if (blocks >= 4 * 152 && cost < best) {
      best = cost;
      JB = jb;
    }
  }
  const size_t threads = strips * ((A.ny + JB - 1) / JB) * kv;
  const unsigned g = (unsigned)((threads + 127) / 128);
  if (vec == 2)
    k_laplace_march<2, MODE><<<g, 128, 0, s>>>((const double *)x, (const double *)b, (double *)y, A.nx, A.ny, kv, diag,
                                               scale, 1.0, A.periodic, JB);
  else
    k_laplace_march<1, MODE><<<g, 128, 0, s>>>((const double *)x, (const double *)b, (double *)y, A.nx, A.ny, kv, diag,
                                               scale, 1.0, A.periodic, JB);
}

template <class T, int VEC, int MODE>
static void laplace_sites(const StencilView &A, const void *x, const void *b, void *y, int k, T diag, T scale,
                          cudaStream_t s) {
  const int kv = k / VEC, bpr = (A.nx * kv + 255) / 256;
  static const int occ = blocks_per_sm(k_laplace<T, VEC, MODE>, 256, 0);
  k_laplace<T, VEC, MODE><<<resident_grid((size_t)bpr * A.ny, occ), 256, 0, s>>>(
      (const T *)x, (const T *)b, (T *)y, A.nx, A.ny, kv, diag, scale, A.periodic, bpr);
}

// FP64: strips walked by few threads only pay where the pipe is busy.  Below about 4600 entries
// per SM a launch is a round trip or two to L2, and a thread per site and pack is shorter
// (whole calls, site against strip: 64^2 x 2 12.3 / 15.2 us, 256^2 x 5 15.3 / 16.2, 512^2 x 2
// 16.6 / 17.7, 128^2 x 32 16.9 / 17.0; 192^2 x 21 19.0 / 18.3, 128^2 x 64 21.9 / 20.5).
template <int MODE>
static void laplace_fp64(const StencilView &A, const void *x, const void *b, void *y, int k, double diag, double scale,
                         cudaStream_t s) {
  if ((size_t)A.nx * A.ny * k >= (size_t)152 * 4608) laplace_march<MODE>(A, x, b, y, k, diag, scale, s);
  else if (laplace_vec<double>(k) == 2) laplace_sites<double, 2, MODE>(A, x, b, y, k, diag, scale, s);
  else laplace_sites<double, 1, MODE>(A, x, b, y, k, diag, scale, s);
}

// One damped-Jacobi sweep of the setup filter for Example 5.1 in one pass (out must not alias x):
// x - omega D^-1 (A x) with A x = diag x - (sum of the in-grid neighbours), written as
// (1 - omega) x + (omega / diag) (sum of the neighbours).
void launch_laplace_jacobi(const StencilView &A, const void *x, void *out, int k, double omega, cudaStream_t s) {
  if (!A.const_laplace || A.t != F64)
    throw cuda_error{cudaErrorInvalidValue, "laplace_jacobi: constant-coefficient Laplacian in FP64 only"};
  laplace_fp64<LAP_JACOBI>(A, x, nullptr, out, k, 1.0 - omega, omega / A.diag, s);
  MLMC_LAUNCH_CHECK("k_laplace_march");
}

static void launch_laplace(const StencilView &A, const void *x, const void *b, void *y, int k, int mode,
                           cudaStream_t s) {
  if (A.t == F64) {
    if (mode) laplace_fp64<LAP_RESIDUAL>(A, x, b, y, k, A.diag, 0.0, s);
    else laplace_fp64<LAP_APPLY>(A, x, b, y, k, A.diag, 0.0, s);
  } else if (A.t == F32) {
    auto go = [&](auto vec) {
      constexpr int VEC = decltype(vec)::value;
      if (mode) laplace_sites<float, VEC, LAP_RESIDUAL>(A, x, b, y, k, (float)A.diag, 0.f, s);
      else laplace_sites<float, VEC, LAP_APPLY>(A, x, b, y, k, (float)A.diag, 0.f, s);
    };
    if (laplace_vec<float>(k) == 4) go(std::integral_constant<int, 4>());
    else go(std::integral_constant<int, 1>());
  } else {
    throw cuda_error{cudaErrorInvalidValue, "constant-coefficient Laplacian is real"};
  }
  MLMC_LAUNCH_CHECK("k_laplace");
}

static void launch_laplace_rbgs(const StencilView &A, void *x, const void *b, int k, int colour, int other_zero,
                                cudaStream_t s, bool from_zero = false) {
  auto launch = [&](auto tag, auto vtag, auto ztag) {
    typedef decltype(tag) T;
    constexpr int VEC = decltype(vtag)::value, TB = lap_threads<T>();
    constexpr bool FROM_ZERO = decltype(ztag)::value;
    int kv = k / VEC;
    const int bpr = (((A.nx + 1) / 2) * kv + TB - 1) / TB;
    static const int occ = blocks_per_sm(k_laplace_rbgs<T, VEC, FROM_ZERO>, TB, 0);
    // FP64: a resident grid (FP64-pipe bound); FP32: one block per unit, measured faster
    // there (119 against 124 us per sweep on 1024^2 x 64)
    const unsigned grid = std::is_same<T, double>::value ? resident_grid((size_t)bpr * A.ny, occ)
                                                         : (unsigned)(bpr * A.ny);
    k_laplace_rbgs<T, VEC, FROM_ZERO><<<grid, TB, 0, s>>>((T *)x, (const T *)b, A.nx, A.ny, kv, (T)(1.0 / A.diag),
                                                          A.periodic, colour, other_zero, bpr);
  };
  auto go = [&](auto tag, auto vtag) {
    if (from_zero) launch(tag, vtag, std::true_type());
    else launch(tag, vtag, std::false_type());
  };
  if (A.t == F64) {
    if (laplace_vec<double>(k) == 2) go(double(), std::integral_constant<int, 2>());
    else go(double(), std::integral_constant<int, 1>());
  } else if (A.t == F32) {
    if (laplace_vec<float>(k) == 4) go(float(), std::integral_constant<int, 4>());
    else go(float(), std::integral_constant<int, 1>());
  } else {
    throw cuda_error{cudaErrorInvalidValue, "constant-coefficient Laplacian is real"};
  }
  MLMC_LAUNCH_CHECK("k_laplace_rbgs");
}

void launch_stencil(const StencilView &A, const void *x, const void *b, void *y, int k, int mode,
                    cudaStream_t s) {
  if (A.const_laplace) {
    launch_laplace(A, x, b, y, k, mode, s);
    return;
  }
  if (A.taps == 9) {
    launch_stencil9(A, x, b, y, k, mode, s);
    return;
  }
  MLMC_DISPATCH(A.t, T, MLMC_DDISPATCH(A.d, D, stencil_go<T, D>(A, x, b, y, k, mode, s)));
  MLMC_LAUNCH_CHECK("k_stencil");
}

// ------------------------------------------------------------------ red-black block GS
// For every site s of colour `colour` ((i + j) % 2):
//   x_s = D_s^{-1} (b_s - sum over the 4 neighbour blocks A_{s,nb} x_nb),
// the exact solve of the site's row block given its neighbours, so the old x_s
// is not read.  Sites of one colour couple only to the other colour, so the
// half-sweep is an exact block Gauss-Seidel step in red-black order (needs nx,
// ny even).  other_zero = 1: the other colour holds zeros (not read), so the
// first half-sweep from x = 0 needs no initialised x.
// the smoother keeps 16-byte packs for complex FP32 blocks up to d = 8 (measured faster there)
// 16-byte packs where the block allows (measured on a level-2 shape, d = 4 FP32:
// 16-byte packs on a row-per-block grid 0.095 ms per sweep, 8-byte packs 0.107 ms)
template <class T, int D> struct rbgs_vec { static const int v = D <= 4 ? 16 / (int)sizeof(T) : 8 / (int)sizeof(T) > 0 ? 8 / (int)sizeof(T) : 1; };
template <int D> struct rbgs_vec<cfloat, D> { static const int v = D <= 8 ? 2 : 1; };
template <int D> struct rbgs_vec<cdouble, D> { static const int v = 1; };

// grid.y = lattice row j; threads of a row cover (site m of the colour, VEC columns).
template <class T, int D, int VEC>
__device__ __forceinline__ void rbgs_half_body(const T *__restrict__ coef, const T *__restrict__ dinv,
                                               T *x, const T *src, const T *b, int nx, int ny, int kv,
                                               int colour, int other_zero, int j, int t) {
  // src: where the neighbours' entries are read, x or (launch_rbgs_first) b; j = lattice row; t = (site m of the colour in the row, pack c of VEC columns)
  typedef Pack<T, VEC> V;
  const int hx = nx / 2;
  if (t < hx * kv) {
    const int m = t / kv, c = t - (t / kv) * kv;
    const int i = 2 * m + ((j + colour) & 1);
    const int s = j * nx + i;
    int nb[5];
    nb[0] = s;
    nb[1] = j * nx + (i + 1 == nx ? 0 : i + 1);
    nb[2] = j * nx + (i == 0 ? nx - 1 : i - 1);
    nb[3] = (j + 1 == ny ? 0 : j + 1) * nx + i;
    nb[4] = (j == 0 ? ny - 1 : j - 1) * nx + i;
    T res[D][VEC];
    size_t o = (size_t)s * D * kv + c;
#pragma unroll
    for (int r = 0; r < D; ++r) {
      V bb = ((const V *)b)[o + (size_t)r * kv];
#pragma unroll
      for (int u = 0; u < VEC; ++u) res[r][u] = bb.v[u];
    }
    if (!other_zero) {
#pragma unroll
      for (int dir = 1; dir < 5; ++dir) {
        const T *B = coef + ((size_t)s * 5 + dir) * D * D;
        const V *xs = (const V *)src + (size_t)nb[dir] * D * kv + c;
        V xq[D];
#pragma unroll
        for (int q = 0; q < D; ++q) xq[q] = xs[(size_t)q * kv];
#pragma unroll
        for (int r = 0; r < D; ++r) {
          T row[D];
          load_row<T, D>(B + r * D, row);
#pragma unroll
          for (int q = 0; q < D; ++q)
#pragma unroll
            for (int u = 0; u < VEC; ++u) res[r][u] = msub4(res[r][u], row[q], xq[q].v[u]);
        }
      }
    }
    const T *Di = dinv + (size_t)s * D * D;
    V *X = (V *)x;
#pragma unroll
    for (int r = 0; r < D; ++r) {
      V out;
      T row[D];
      load_row<T, D>(Di + r * D, row);
#pragma unroll
      for (int u = 0; u < VEC; ++u) out.v[u] = zero<T>();
#pragma unroll
      for (int q = 0; q < D; ++q)
#pragma unroll
        for (int u = 0; u < VEC; ++u) out.v[u] = madd4(out.v[u], row[q], res[q][u]);
      X[o + (size_t)r * kv] = out;
    }
  }
}

template <class T, int D, int VEC>
__global__ void __launch_bounds__(gen_threads<T, D>()) k_rbgs_half(const T *__restrict__ coef, const T *__restrict__ dinv,
                                                   T *x, const T *src, const T *b, int nx, int ny, int kv,
                                                   int colour, int other_zero, int bpr) {
  // resident grid striding over the units (row j, chunk of one block's threads of the row)
  const int units = bpr * ny;
  for (int u = blockIdx.x; u < units; u += gridDim.x) {
    const int j = u / bpr;
    rbgs_half_body<T, D, VEC>(coef, dinv, x, src, b, nx, ny, kv, colour, other_zero, j,
                              (u - j * bpr) * gen_threads<T, D>() + threadIdx.x);
  }
}

// The same half-sweep in blocks of 128 threads with residency pinned at 8 blocks
// per SM (<= 64 registers), for FP32 blocks with d = 4 (the aggregation levels of
// the Laplace hierarchy), on a resident grid striding over the units (row j, chunk of
// 128 threads of the row) in row order.  The kernel is load-latency bound; measured
// on the 256^2 x 4 level, k = 128, per sweep: 86.7-87.0 us here, 88.3 us with one
// block per unit (a grid of 8192 blocks), 90.6 us with 256 threads x 4
// blocks, 93.7 us unpinned (256 threads), 96-99 us with two or four neighbour
// blocks' loads issued together (80-128 registers, 2-3 blocks of 256 per SM) and
// 100-104 us with 5-8 blocks of 256 per SM (8-byte packs or spills).
template <class T, int D, int VEC>
__global__ void __launch_bounds__(128, 8) k_rbgs_half_p(const T *__restrict__ coef, const T *__restrict__ dinv,
                                                        T *x, const T *src, const T *b, int nx, int ny,
                                                        int kv, int colour, int other_zero, int bpr) {
  // colour 1 walks the rows from the last: consecutive half-sweeps alternate direction,
  // so each starts on the rows the previous one wrote last (still in L2)
  const int units = bpr * ny;
  for (int u0 = blockIdx.x; u0 < units; u0 += gridDim.x) {
    const int u = colour ? units - 1 - u0 : u0;
    const int j = u / bpr;
    rbgs_half_body<T, D, VEC>(coef, dinv, x, src, b, nx, ny, kv, colour, other_zero, j, (u - j * bpr) * 128 + threadIdx.x);
  }
}

// Row-split half-sweep for large site blocks (see k_stencil_rows).  Phase 1: res_r = b_r - sum
// over the 4 neighbour blocks of row r times their x; phase 2, after a block barrier:
// x_r = sum_q Dinv[r][q] res_q from shared memory.  Grid = (column chunks, sites of the colour).
template <class T, int D, int CV, int RPT, bool STAGED>
__global__ void __launch_bounds__(32 * D / RPT) k_rbgs_half_rows(const T *__restrict__ coef,
                                                                 const T *__restrict__ dinv, T *x, const T *src,
                                                                 const T *b, int nx,
                                                                 int ny, int k, int colour, int other_zero) {
  typedef Pack<T, CV> V;
  constexpr int BLK = D * D * (int)sizeof(T);
  __shared__ __align__(16) unsigned char blk_mem[STAGED ? 5 * BLK : 16];   // the four neighbour blocks, then D^-1
  __shared__ V res[D][32];
  const int hx = nx / 2;
  const int idx = blockIdx.y;                       // site of this colour: row j, position m
  const int j = idx / hx, m = idx - (idx / hx) * hx;
  const int i = 2 * m + ((j + colour) & 1);
  const int s = j * nx + i;
  const int cl = threadIdx.x, r0 = threadIdx.y * RPT, tid = threadIdx.y * 32 + threadIdx.x;
  const int c = (blockIdx.x * 32 + cl) * CV;        // k is a multiple of CV
  const bool live = c < k;
  const T *blk = STAGED ? (const T *)blk_mem : coef + ((size_t)s * 5 + 1) * D * D;
  if constexpr (STAGED) {
    if (!other_zero) block_copy_async(blk_mem, coef + ((size_t)s * 5 + 1) * D * D, 4 * BLK, tid, 32 * D / RPT);
    block_copy_async(blk_mem + 4 * BLK, dinv + (size_t)s * D * D, BLK, tid, 32 * D / RPT);
  }
  V acc[RPT];
#pragma unroll
  for (int r = 0; r < RPT; ++r)
    if (live) acc[r] = *reinterpret_cast<const V *>(b + ((size_t)s * D + r0 + r) * k + c);
  if (!other_zero) {
    int nb[4];
    nb[0] = j * nx + (i + 1 == nx ? 0 : i + 1);
    nb[1] = j * nx + (i == 0 ? nx - 1 : i - 1);
    nb[2] = (j + 1 == ny ? 0 : j + 1) * nx + i;
    nb[3] = (j == 0 ? ny - 1 : j - 1) * nx + i;
    rows_accumulate<T, D, CV, RPT, 4, true, STAGED>(blk, src, nb, r0, k, c, live, acc, async_ready);
  } else if constexpr (STAGED) {
    async_ready();
  }
#pragma unroll
  for (int r = 0; r < RPT; ++r) res[r0 + r][cl] = acc[r];
  __syncthreads();
  if (!live) return;
  V out[RPT];
#pragma unroll
  for (int r = 0; r < RPT; ++r) {
    T row[D];
    if constexpr (STAGED)
      memcpy(row, __builtin_assume_aligned(blk_mem + 4 * BLK + (size_t)(r0 + r) * D * sizeof(T), 16), sizeof(row));
    else
      load_row<T, D>(dinv + ((size_t)s * D + r0 + r) * D, row);
#pragma unroll
    for (int u = 0; u < CV; ++u) out[r].v[u] = zero<T>();
#pragma unroll
    for (int q = 0; q < D; ++q) {
      const V rv = res[q][cl];
#pragma unroll
      for (int u = 0; u < CV; ++u) out[r].v[u] = madd4(out[r].v[u], row[q], rv.v[u]);
    }
    *reinterpret_cast<V *>(x + ((size_t)s * D + r0 + r) * k + c) = out[r];
  }
}

template <class T, int D>
static void rbgs_go(const StencilView &A, const void *coef, void *x, const void *src, const void *b, int k, int colour,
                    int other_zero, cudaStream_t s) {
  if constexpr (D >= 8) {
    if ((A.nx / 2) * A.ny <= 65535) {
      constexpr int RPT = rows_rpt<T>();
      rows_dispatch<T>(k, (A.nx / 2) * A.ny, [&](auto cv, auto staged, dim3 grid) {
        k_rbgs_half_rows<T, D, decltype(cv)::value, RPT, decltype(staged)::value><<<grid, dim3(32, D / RPT), 0, s>>>(
            (const T *)coef, (const T *)A.dinv, (T *)x, (const T *)src, (const T *)b, A.nx, A.ny, k, colour, other_zero);
      });
      return;
    }
  }
  constexpr int VW = rbgs_vec<T, D>::v, TB = gen_threads<T, D>();
  if (VW > 1 && k % VW == 0) {
    int kv = k / VW;
    if constexpr (std::is_same<T, float>::value && D == 4)
    {
      const int bpr = ((A.nx / 2) * kv + 127) / 128;
      k_rbgs_half_p<T, D, VW><<<resident_grid(bpr * A.ny, 8), 128, 0, s>>>(
          (const T *)coef, (const T *)A.dinv, (T *)x, (const T *)src, (const T *)b, A.nx, A.ny, kv, colour, other_zero, bpr);
    }
    else {
      const int bpr = ((A.nx / 2) * kv + TB - 1) / TB;
      static const int occ = blocks_per_sm(k_rbgs_half<T, D, VW>, TB, 0);
      k_rbgs_half<T, D, VW><<<resident_grid((size_t)bpr * A.ny, occ), TB, 0, s>>>(
          (const T *)coef, (const T *)A.dinv, (T *)x, (const T *)src, (const T *)b, A.nx, A.ny, kv, colour, other_zero, bpr);
    }
  } else {
    const int bpr = ((A.nx / 2) * k + TB - 1) / TB;
    static const int occ = blocks_per_sm(k_rbgs_half<T, D, 1>, TB, 0);
    k_rbgs_half<T, D, 1><<<resident_grid((size_t)bpr * A.ny, occ), TB, 0, s>>>(
        (const T *)coef, (const T *)A.dinv, (T *)x, (const T *)src, (const T *)b, A.nx, A.ny, k, colour, other_zero, bpr);
  }
}

void launch_rbgs_half(const StencilView &A, void *x, const void *b, int k, int colour, cudaStream_t s) {
  if (A.const_laplace) {
    launch_laplace_rbgs(A, x, b, k, colour, 0, s);
    return;
  }
  if (A.taps == 9) throw cuda_error{cudaErrorInvalidValue, "9-point stencils are smoothed in four colours"};
  MLMC_DISPATCH(A.t, T, MLMC_DDISPATCH(A.d, D, rbgs_go<T, D>(A, A.coef, x, x, b, k, colour, 0, s)));
  MLMC_LAUNCH_CHECK("k_rbgs_half");
}

void launch_rbgs_sweep(const StencilView &A, void *x, const void *b, int k, int order, int x_zero,
                       cudaStream_t s) {
  int first = order == 0 ? 0 : 1;
  if (A.const_laplace) {
    launch_laplace_rbgs(A, x, b, k, first, x_zero, s);
    launch_laplace_rbgs(A, x, b, k, 1 - first, 0, s);
    return;
  }
  if (A.taps == 9) {
    launch_gs9_sweep(A, x, b, k, order, x_zero, s);
    return;
  }
  // x_zero: the first half-sweep reads no neighbours and the second none of its own
  // old values, so x needs no initialisation
  MLMC_DISPATCH(A.t, T, MLMC_DDISPATCH(A.d, D, rbgs_go<T, D>(A, A.coef, x, x, b, k, first, x_zero ? 1 : 0, s)));
  MLMC_LAUNCH_CHECK("k_rbgs_half");
  launch_rbgs_half(A, x, b, k, 1 - first, s);
}

// ------------------------------------------------------------------ the first sweep from x = 0
// A red-black sweep from x = 0 sets x_0 = D_0^{-1} b_0 and then x_1 = D_1^{-1} (b_1 - A_10 x_0).  When
// another sweep follows, it overwrites x_0 without reading it, so only x_1 is wanted, and
// x_1 = D_1^{-1} (b_1 - (A_10 D_0^{-1}) b_0) is a half-sweep of the same form with b in the place of x
// and the products A_10 D_0^{-1} (StencilView::first, formed once at setup) in the place of A_10:
// one launch and 1.5 vector passes instead of two and 2.5.
void launch_rbgs_first(const StencilView &A, void *x, const void *b, int k, cudaStream_t s) {
  if (A.const_laplace) {
    launch_laplace_rbgs(A, x, b, k, 1, 0, s, true);
    return;
  }
  if (!A.first) throw cuda_error{cudaErrorInvalidValue, "rbgs_first: no products on this level"};
  MLMC_DISPATCH(A.t, T, MLMC_DDISPATCH(A.d, D, rbgs_go<T, D>(A, A.first, x, b, b, k, 1, 0, s)));
  MLMC_LAUNCH_CHECK("k_rbgs_half");
}

// first[s][dir] = A_{s,dir} D_{nb(dir)}^{-1} for the sites s of colour 1, dir = 1 .. 4 (other entries unset)
template <class T>
__global__ void k_first_blocks(const T *__restrict__ coef, const T *__restrict__ dinv, T *__restrict__ first, int nx,
                               int ny, int d) {
  const unsigned per = 4u * d * d, total = (unsigned)nx * ny / 2 * per;
  for (unsigned t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
    const unsigned h = t / per, e = t - h * per;
    const int dir = 1 + (int)(e / (d * d)), r = (int)(e / d) % d, q = (int)e % d;
    const int j = (int)(h / (nx / 2)), i = 2 * (int)(h % (nx / 2)) + ((j + 1) & 1), s = j * nx + i;
    const int nb = dir == 1 ? j * nx + (i + 1 == nx ? 0 : i + 1) : dir == 2 ? j * nx + (i == 0 ? nx - 1 : i - 1)
                 : dir == 3 ? (j + 1 == ny ? 0 : j + 1) * nx + i : (j == 0 ? ny - 1 : j - 1) * nx + i;
    const T *a = coef + ((size_t)s * 5 + dir) * d * d + r * d, *w = dinv + (size_t)nb * d * d + q;
    T v = zero<T>();
    for (int m = 0; m < d; ++m) v = madd(v, a[m], w[(size_t)m * d]);
    first[((size_t)s * 5 + dir) * d * d + r * d + q] = v;
  }
}

void launch_first_blocks(DType t, const void *coef, const void *dinv, void *first, int nx, int ny, int d,
                         cudaStream_t s) {
  const size_t total = (size_t)nx * ny / 2 * 4 * d * d;
  MLMC_DISPATCH(t, T, k_first_blocks<T><<<grid_for(total, 256), 256, 0, s>>>((const T *)coef, (const T *)dinv,
                                                                             (T *)first, nx, ny, d));
  MLMC_LAUNCH_CHECK("k_first_blocks");
}

}  // namespace mlmc
