// Column dot products and multi-AXPY of the batched Krylov solvers, and the per-column
// algebra of the fixed-length FGMRES (Saad, Alg. 9.6, with an unnormalised basis).
//
// Vector blocks are [row][k] with the k columns (independent systems) innermost.  A thread
// owns one 16-byte pack of consecutive columns (VEC columns; 1 where k or a pointer does
// not allow it) and walks the rows of its block's contiguous chunk, so every load is
// coalesced and a column's sum stays in one lane until the end of the chunk.
//
// FP64 additions run at 1.7 per clock and SM on this GPU (0.53 T/s), FP32 ones at 128.  A thread
// adds up its own FP32 products in FP32; a block's lane sums meet as float pairs (a hi + lo sum by
// the two-sum of Knuth, TAOCP 4.2.2; 48 significant bits, far below the rounding of the FP32 lane
// sums), or in FP64 where a pair leaves FP32's range, and everything beyond a block is FP64.
// Sums of FP64 data are FP64 throughout.
#include <algorithm>
#include <initializer_list>
#include <mutex>
#include <type_traits>

#include "mlmc_internal.cuh"

namespace mlmc {

namespace {

constexpr int DT = 512;            // threads per block
constexpr int DOT_PARTS = 152;     // row chunks of a dot product: one block per SM (FP64 data: two)
constexpr int AXPY_PARTS = 304;    // row chunks of a multi-AXPY: two blocks per SM
constexpr int DOT_MAXV = 8;        // basis vectors per pass over w
constexpr int RT = 512;            // threads of a reduction block

template <class T, int VEC> struct alignas(sizeof(T) * VEC) DPack { T v[VEC]; };

// Scalars of a column (real: 1, complex: 2) and their running sums over lanes and blocks.
struct FF { float h, l; };
template <class T> struct lane_of;
template <> struct lane_of<float> { typedef float S; typedef FF A; static constexpr int C = 1; };
template <> struct lane_of<double> { typedef double S; typedef double A; static constexpr int C = 1; };
template <> struct lane_of<cfloat> { typedef float S; typedef FF A; static constexpr int C = 2; };
template <> struct lane_of<cdouble> { typedef double S; typedef double A; static constexpr int C = 2; };
template <class T> struct acc_of { typedef double type; };
template <> struct acc_of<cdouble> { typedef cdouble type; };
template <> struct acc_of<cfloat> { typedef cdouble type; };

__device__ __forceinline__ void acc_zero(FF &a) { a.h = a.l = 0.f; }
__device__ __forceinline__ void acc_zero(double &a) { a = 0.0; }
// a += x: the rounding error of each addition goes into the low part
__device__ __forceinline__ void acc_add(FF &a, float x) {
  const float s = a.h + x, t = s - a.h;
  a.l += (a.h - (s - t)) + (x - t);
  a.h = s;
}
__device__ __forceinline__ void acc_add(FF &a, FF b) {
  acc_add(a, b.h);
  a.l += b.l;
}
__device__ __forceinline__ void acc_add(double &a, double x) { a += x; }
__device__ __forceinline__ double acc_value(FF a) { return (double)a.h + (double)a.l; }
__device__ __forceinline__ double acc_value(double a) { return a; }

// a += conj(x) * y on scalars
__device__ __forceinline__ void dot_fma(float a[1], float x, float y) { a[0] += x * y; }
__device__ __forceinline__ void dot_fma(double a[1], double x, double y) { a[0] += x * y; }
// complex FP32: the product is formed first, so that the running sum is rounded once per term
// (262144 x 64: rms error 1.5e-9 of the terms' size, 2.2e-9 with two multiply-adds on the sum)
__device__ __forceinline__ void dot_fma(float a[2], cfloat x, cfloat y) {
  a[0] += fmaf(x.im, y.im, x.re * y.re);
  a[1] += fmaf(-x.im, y.re, x.re * y.im);
}
__device__ __forceinline__ void dot_fma(double a[2], cdouble x, cdouble y) {
  a[0] = fma(x.im, y.im, fma(x.re, y.re, a[0]));
  a[1] = fma(-x.im, y.re, fma(x.re, y.im, a[1]));
}

template <class T> struct VecList { const T *v[DOT_MAXV]; };

__device__ __forceinline__ void chunk_of(size_t rows, size_t &r0, size_t &r1) {
  const size_t chunk = (rows + gridDim.x - 1) / gridDim.x;
  r0 = min((size_t)blockIdx.x * chunk, rows);
  r1 = min(r0 + chunk, rows);
}

// out[r * E + e] = sum over the block's slots, in fixed order, of the nr <= RB rows of NC scalars per
// thread in val; e < E = k * C scalars of a row.  The rows are summed together, and the threads that
// share a scalar meet in steps of at most eight: with a row at a time and one chain over those
// threads, 511 long for one column, eight FP64 vectors of 1024 x 1 took 174 us (11 now), of
// 1024 x 8 41 us (14) and of 4096 x 64 20 us (12).  red: RB * DT * NC lane values, red2: DT sums.
// Ends with the block synchronised.
template <class T, int NC, int RB>
__device__ __forceinline__ void block_sums(const typename lane_of<T>::S (*val)[NC], int nr, typename lane_of<T>::S *red,
                                           typename lane_of<T>::A *red2, int E, int slots, bool live, double *out) {
  typedef typename lane_of<T>::A A;
  const int tid = threadIdx.x;
  // the sum as FP64; lane values whose float pair left FP32's range (or are not finite) are added again
  auto finish = [&](const A &a, const typename lane_of<T>::S *src) {
    double v = acc_value(a);
    if (sizeof(typename lane_of<T>::S) == 4 && !isfinite(v)) {
      v = 0.0;
      for (int s = 0; s < slots; ++s) v += (double)src[s * E];
    }
    return v;
  };
#pragma unroll
  for (int r = 0; r < RB; ++r)
    if (r < nr) {
#pragma unroll
      for (int u = 0; u < NC; ++u) red[(r * DT + tid) * NC + u] = live ? val[r][u] : 0;
    }
  __syncthreads();
  // scalar e of row r sits at red[r * DT * NC + slot * E + e]; G threads share its slots
  const int items = nr * E;
  int G = min(DT / items, slots);
  if (G < 2) {
    for (int i = tid; i < items; i += DT) {
      const int r = i / E;
      const typename lane_of<T>::S *src = red + r * DT * NC + (i - r * E);
      A a;
      acc_zero(a);
      for (int s = 0; s < slots; ++s) acc_add(a, src[s * E]);
      out[i] = finish(a, src);
    }
  } else {
    const int g = tid / items, i = tid - g * items, r = i / E;
    const typename lane_of<T>::S *src = red + r * DT * NC + (i - r * E);
    A a;
    acc_zero(a);
    if (g < G) {
      for (int s = g; s < slots; s += G) acc_add(a, src[s * E]);
      red2[tid] = a;
    }
    while (G > 8) {
      const int H = G > 64 ? 64 : 8;
      __syncthreads();
      if (g < H) {
        for (int q = g + H; q < G; q += H) acc_add(a, red2[q * items + i]);
        red2[tid] = a;               // read by this thread alone in this step
      }
      G = H;
    }
    __syncthreads();
    if (g == 0) {
      for (int q = 1; q < G; ++q) acc_add(a, red2[q * items + i]);
      out[i] = finish(a, src);
    }
  }
  __syncthreads();
}

}  // namespace

// ------------------------------------------------------------------ dot products
// partial[part][row0 + r][c] = sum over the chunk's rows of conj(V_r[row][c]) w[row][c], r < NV,
// then (EXTRA & 2) v0.v0 and (EXTRA & 1) w.w in the following rows: quantities of the same
// read of the data that would otherwise need passes of their own.
// HBM-bound on large blocks: 16 warps per SM with about eight 16-byte loads in flight per
// thread; one block per SM, so only 152 partial sums per column are left to add (complex FP32,
// whose 304 blocks keep the lane sums short, two per SM: 8 vectors of 4096 x 200 24.7 -> 20.7 us,
// 30 of 4096 x 64 49 -> 41).  Four FP32
// vectors of 1024^2 x 64 with the reduction: 210 us, 6.37 TB/s (250 us with 608 blocks of 256
// threads, 8-byte loads and FP64 block sums); 16384 x 128, L2-resident: 12.4 us (22.6).
template <class T, int VEC, int NV, int EXTRA>
__global__ void __launch_bounds__(DT, std::is_same<T, cfloat>::value ? 2 : 1)
    k_dots(VecList<T> V, const T *__restrict__ w, size_t rows, int k, double *__restrict__ partial, int row0, int nrows) {
  typedef typename lane_of<T>::S S;
  typedef typename lane_of<T>::A A;
  typedef DPack<T, VEC> P;
  constexpr int C = lane_of<T>::C, NC = VEC * C;
  constexpr int R = NV + (EXTRA & 1) + (EXTRA >> 1);
  constexpr int U = NV <= 1 ? 4 : NV <= 3 ? 2 : 1;
  constexpr int RB = R < 4 ? R : 4;                          // rows summed together
  __shared__ __align__(16) S red[RB * DT * NC];
  __shared__ A red2[DT];
  const int kv = k / VEC, slots = DT / kv;
  const int cv = threadIdx.x % kv, slot = threadIdx.x / kv;
  const bool live = slot < slots;
  size_t r0, r1;
  chunk_of(rows, r0, r1);
  S acc[R][NC];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int u = 0; u < NC; ++u) acc[r][u] = 0;
  const P *W = (const P *)w;
  auto step = [&](const P &wv, const P *x) {
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
      for (int u = 0; u < VEC; ++u) dot_fma(&acc[v][u * C], x[v].v[u], wv.v[u]);
    if (EXTRA & 2)
#pragma unroll
      for (int u = 0; u < VEC; ++u) dot_fma(&acc[NV][u * C], x[0].v[u], x[0].v[u]);
    if (EXTRA & 1)
#pragma unroll
      for (int u = 0; u < VEC; ++u) dot_fma(&acc[NV + (EXTRA >> 1)][u * C], wv.v[u], wv.v[u]);
  };
  if (live) {
    size_t r = r0 + slot;
    for (; r + (size_t)(U - 1) * slots < r1; r += (size_t)U * slots) {
      P wv[U], x[U][NV];
#pragma unroll
      for (int q = 0; q < U; ++q) {
        const size_t o = (r + (size_t)q * slots) * kv + cv;
        wv[q] = W[o];
#pragma unroll
        for (int v = 0; v < NV; ++v) x[q][v] = ((const P *)V.v[v])[o];
      }
#pragma unroll
      for (int q = 0; q < U; ++q) step(wv[q], x[q]);
    }
    for (; r < r1; r += slots) {
      P wv, x[NV];
      const size_t o = r * kv + cv;
      wv = W[o];
#pragma unroll
      for (int v = 0; v < NV; ++v) x[v] = ((const P *)V.v[v])[o];
      step(wv, x);
    }
  }
  const int E = k * C;
#pragma unroll
  for (int r = 0; r < R; r += RB)
    block_sums<T, NC, RB>(acc + r, R - r < RB ? R - r : RB, red, red2, E, slots, live,
                          partial + ((size_t)blockIdx.x * nrows + row0 + r) * E);
}

// out[e] = sum over parts of partial[part][e], e < nrows * k scalars, in fixed order: a block per
// eight consecutive scalars, 64 threads each taking every 64th part, met in steps of eight.
constexpr int RE = 8, RS = RT / RE;
static __global__ void __launch_bounds__(RT) k_dots_reduce(const double *__restrict__ partial, int nparts, int entries,
                                                           double *__restrict__ out) {
  __shared__ double red[RS][RE];
  const int lane = threadIdx.x % RE, sl = threadIdx.x / RE;
  const int e = blockIdx.x * RE + lane;
  double a = 0.0;
  if (e < entries)
    for (int p = sl; p < nparts; p += RS) a += partial[(size_t)p * entries + e];
  red[sl][lane] = a;
  __syncthreads();
  if (sl < 8) {
    for (int q = sl + 8; q < min(nparts, RS); q += 8) a += red[q][lane];
    red[sl][lane] = a;               // read by this thread alone in this step
  }
  __syncthreads();
  if (sl == 0 && e < entries) {
    for (int q = 1; q < min(nparts, 8); ++q) a += red[q][lane];
    out[e] = a;
  }
}

// Columns per pack: 16 bytes, or 8 of an FP32 block (k = 2 mod 4; 4 vectors of 262144 x 62: 84 us,
// 144 with single columns), where every row allows it.
static int pack_of(DType t, int k) {
  const int vw = 16 / (int)dtype_size(t);
  return k % vw == 0 ? vw : vw == 4 && k % 2 == 0 ? 2 : 1;
}

template <class T> constexpr DType type_of() {
  return std::is_same<T, double>::value ? F64 : std::is_same<T, float>::value ? F32
       : std::is_same<T, cdouble>::value ? C64 : C32;
}

int multidot_parts(DType t, size_t rows, int k) {
  // a row of packs per thread where the rows are few; FP32 packs of four columns at most one block
  // per SM, narrower ones and FP64 two, so that a lane adds up half as many, but whole waves only:
  // a block of k_dots has an SM to itself or half of one (8 FP64 vectors of 4096 x 200: 205 blocks 39 us, 304 with
  // block_sums 29)
  const int pack = pack_of(t, k);
  const bool fp64 = dtype_lower(t) != t;       // no lane sums in FP32 to keep short
  const size_t packs = std::max(k / pack, 1), slots = std::max<size_t>(1, DT / packs);
  const size_t p = std::max<size_t>(1, (rows + slots - 1) / slots);
  // complex FP64 that would stay on less than half of the SMs: 64 packs per block, whose arithmetic
  // otherwise takes longer than the loads (four vectors of 128 x 8: 12.4 -> 10.4 us; real ones lose 1 us
  // to the longer second stage where it is not that)
  if (t == C64 && p <= 64) {
    const size_t few = std::max<size_t>(1, 64 / packs);
    return (int)std::min<size_t>(DOT_PARTS, (rows + few - 1) / few);
  }
  if (p <= DOT_PARTS || pack == 4) return (int)std::min<size_t>(DOT_PARTS, p);
  return fp64 && p < 2 * DOT_PARTS ? DOT_PARTS : 2 * DOT_PARTS;
}

namespace {

// The widest pack, of the width pack_of gives or less, that every pointer allows.
template <class T>
int pack_at(int k, size_t vstride, std::initializer_list<const void *> ptrs) {
  int vec = pack_of(type_of<T>(), k);
  for (const void *p : ptrs)
    while (vec > 1 && ((uintptr_t)p % (vec * sizeof(T)) || vstride % vec)) vec /= 2;
  return vec;
}

// f(VEC) with the pack as a compile-time width
template <class T, class F>
void with_pack(int vec, F &&f) {
  constexpr int VW = 16 / (int)sizeof(T);
  if constexpr (VW == 4)
    if (vec == 4) return f(std::integral_constant<int, 4>());
  if constexpr (VW >= 2)
    if (vec == 2) return f(std::integral_constant<int, 2>());
  f(std::integral_constant<int, 1>());
}

template <class T, int VEC, int EXTRA>
void dots_go(const VecList<T> &V, int nv, const T *w, size_t rows, int k, void *partial, int nparts, int row0,
             int nrows, cudaStream_t s) {
  auto go = [&](auto n) {
    constexpr int NV = decltype(n)::value;
    if constexpr (NV == 1 || EXTRA < 2)           // v0.v0 is asked for with the first vector alone
      k_dots<T, VEC, NV, EXTRA><<<nparts, DT, 0, s>>>(V, w, rows, k, (double *)partial, row0, nrows);
    else
      throw cuda_error{cudaErrorInvalidValue, "multidot: v0.v0 needs a single vector"};
  };
  switch (nv) {
    case 1: go(std::integral_constant<int, 1>()); break;
    case 2: go(std::integral_constant<int, 2>()); break;
    case 3: go(std::integral_constant<int, 3>()); break;
    case 4: go(std::integral_constant<int, 4>()); break;
    case 5: go(std::integral_constant<int, 5>()); break;
    case 6: go(std::integral_constant<int, 6>()); break;
    case 7: go(std::integral_constant<int, 7>()); break;
    default: go(std::integral_constant<int, 8>()); break;
  }
  MLMC_LAUNCH_CHECK("k_dots");
}

// Partial sums of w against nvec basis vectors (v0, then V + i * vstride elements), then
// (extra & 2) v0.v0 and (extra & 1) w.w; returns the number of passes (launches).
template <class T>
int dots_partial(const void *v0, const void *V, size_t vstride, int nvec, const void *w, size_t rows, int k,
                 void *partial, int nparts, int extra, cudaStream_t s) {
  const int pack = pack_at<T>(k, vstride, {v0, V, w});
  if (k / pack > DT) throw cuda_error{cudaErrorInvalidValue, "multidot: more column groups than threads"};
  const int nrows = nvec + (extra & 1) + (extra >> 1);
  int passes = 0;
  for (int i0 = 0; i0 < nvec; i0 += DOT_MAXV) {
    VecList<T> L;
    const int nv = std::min(nvec - i0, DOT_MAXV);
    for (int i = 0; i < DOT_MAXV; ++i) {
      const int id = i0 + std::min(i, nv - 1);
      L.v[i] = id == 0 ? (const T *)v0 : (const T *)V + (size_t)id * vstride;
    }
    // the extra rows ride on the last pass (w.w) or need v0 in it (v0.v0: nvec = 1)
    const int ex = i0 + nv < nvec ? 0 : extra;
    with_pack<T>(pack, [&](auto vec) {
      constexpr int VEC = decltype(vec)::value;
      if (ex == 0) dots_go<T, VEC, 0>(L, nv, (const T *)w, rows, k, partial, nparts, i0, nrows, s);
      else if (ex == 1) dots_go<T, VEC, 1>(L, nv, (const T *)w, rows, k, partial, nparts, i0, nrows, s);
      else if (ex == 2) dots_go<T, VEC, 2>(L, nv, (const T *)w, rows, k, partial, nparts, i0, nrows, s);
      else dots_go<T, VEC, 3>(L, nv, (const T *)w, rows, k, partial, nparts, i0, nrows, s);
    });
    ++passes;
  }
  return passes;
}

}  // namespace

void launch_multidot(DType t, const void *V, size_t vstride, int nvec, const void *w, size_t rows, int k,
                     void *partials, int nparts, void *out, cudaStream_t s) {
  MLMC_DISPATCH(t, T, {
    dots_partial<T>(V, V, vstride, nvec, w, rows, k, partials, nparts, 0, s);
    const int entries = nvec * k * lane_of<T>::C;
    k_dots_reduce<<<(entries + RE - 1) / RE, RT, 0, s>>>((const double *)partials, nparts, entries, (double *)out);
    MLMC_LAUNCH_CHECK("k_dots_reduce");
  });
}

// ------------------------------------------------------------------ multi-AXPY
// w[r][c] = (INIT ? 0 : w[r][c]) + sign * sum_v V_v[r][c] * h[v * k + c], v0 <= v < v0 + nv, V_0 = first and
// V_v = V + v * vstride: one pass over w for all vectors whose coefficients, rounded to the
// storage precision, fit in 32 KB of shared memory.  norm (optional): per block and column the
// sum of |w_new|^2 over its rows, for the Arnoldi step, summed per thread in row order (float
// pairs every 16 rows) and over the block's slots in fixed order; INIT updates (the solution) need none.
// HBM-bound on large blocks ((nv + 2) passes, nv + 1 with INIT): all vectors in one pass, not
// eight, since a restarted solve has up to 64 of them.  30 FP64 vectors of 65536 x 64: 223 us
// (284 in passes of eight, 238 with 256 threads striding over packs), FP32 94 (145, 112);
// 27 FP64 vectors of 1024 x 8: 10.4 us (30.9, 8.3); 12 FP32 vectors of 262144 x 64: 157 us,
// 6.0 TB/s (196, 173).  A block has one row of packs per thread where the rows are few: with
// four, 8 vectors of 1024 x 8 complex FP64 were on four SMs and took 22.6 us, now 8.3.
template <class T, class H, int VEC, bool INIT>
__global__ void __launch_bounds__(DT, 2) k_axpy(T *__restrict__ w, const T *__restrict__ first, const T *__restrict__ V,
                                                size_t vstride, int v0, int nv, const H *__restrict__ h, double sign,
                                                size_t rows, int k, double *__restrict__ norm) {
  typedef typename lane_of<T>::S S;
  typedef typename lane_of<T>::A A;
  typedef DPack<T, VEC> P;
  constexpr int UN = std::is_same<T, cfloat>::value ? 2 : 4;   // vectors in flight (complex FP32 with 4: 5 % slower)
  extern __shared__ __align__(16) unsigned char axpy_smem[];
  __shared__ __align__(16) S red[DT * VEC];
  __shared__ A red2[DT];
  T *hs = (T *)axpy_smem;
  for (int e = threadIdx.x; e < nv * k; e += DT)
    hs[e] = cvt<T, H>(rmul((typename real_of<H>::type)sign, h[(size_t)v0 * k + e]));
  __syncthreads();
  const int kv = k / VEC, slots = DT / kv;
  const int cv = threadIdx.x % kv, slot = threadIdx.x / kv;
  const bool live = slot < slots;
  size_t r0, r1;
  chunk_of(rows, r0, r1);
  P *W = (P *)w;
  const P *Hp = (const P *)hs + cv;
  S sq[VEC];
  A tot[VEC];
#pragma unroll
  for (int u = 0; u < VEC; ++u) {
    sq[u] = 0;
    acc_zero(tot[u]);
  }
  // rows r, r + slots, ...: U of them
  auto step = [&](size_t r, auto count) {
    constexpr int U = decltype(count)::value;
    P a[U];
    size_t o[U];
#pragma unroll
    for (int q = 0; q < U; ++q) {
      o[q] = (r + (size_t)q * slots) * kv + cv;
      if (INIT) {
#pragma unroll
        for (int u = 0; u < VEC; ++u) a[q].v[u] = zero<T>();
      } else {
        a[q] = W[o[q]];
      }
    }
    const T *src = v0 == 0 ? first : V + (size_t)v0 * vstride;
#pragma unroll UN
    for (int v = 0; v < nv; ++v) {
      const P hh = Hp[v * kv];
      P x[U];
#pragma unroll
      for (int q = 0; q < U; ++q) x[q] = ((const P *)src)[o[q]];
      src = V + (size_t)(v0 + v + 1) * vstride;
#pragma unroll
      for (int q = 0; q < U; ++q)
#pragma unroll
        for (int u = 0; u < VEC; ++u) a[q].v[u] = madd(a[q].v[u], x[q].v[u], hh.v[u]);
    }
#pragma unroll
    for (int q = 0; q < U; ++q) {
      W[o[q]] = a[q];
      if (!INIT)
#pragma unroll
        for (int u = 0; u < VEC; ++u) sq[u] += abs2(a[q].v[u]);
    }
  };
  if (live) {
    int n = 0;
    size_t r = r0 + slot;
    for (; r + slots < r1; r += 2 * (size_t)slots) {
      step(r, std::integral_constant<int, 2>());
      if (!INIT && sizeof(S) == 4 && (++n & 7) == 0) {
#pragma unroll
        for (int u = 0; u < VEC; ++u) {
          acc_add(tot[u], sq[u]);
          sq[u] = 0;
        }
      }
    }
    if (r < r1) step(r, std::integral_constant<int, 1>());
  }
  if (!INIT && norm) {
    S v[1][VEC];
#pragma unroll
    for (int u = 0; u < VEC; ++u) {
      acc_add(tot[u], sq[u]);
      if constexpr (sizeof(S) == 4) v[0][u] = tot[u].h + tot[u].l;   // one rounding to the lane precision
      else v[0][u] = tot[u];
    }
    // |w|^2 is real for complex data too: one scalar per column
    block_sums<typename real_of<T>::type, VEC, 1>(v, 1, red, red2, k, slots, live, norm + (size_t)blockIdx.x * k);
  }
}

static const int AXPY_SMEM = 32 * 1024;

// A row of packs per thread, at most two blocks per SM.  FP64: 64 packs per block where the rows are
// few, since a block's FP64 arithmetic takes its SM longer than the loads (four vectors of 1024 x 32:
// 7.2 us with 512 packs per block, 4.5 now).
int multiaxpy_norm_parts(DType t, size_t rows, int k) {
  const size_t packs = std::max(k / pack_of(t, k), 1), slots = std::max<size_t>(1, (dtype_lower(t) != t ? 64 : DT) / packs);
  return (int)std::min<size_t>(AXPY_PARTS, std::max<size_t>(1, (rows + slots - 1) / slots));
}

namespace {

template <class T, class H>
int axpy_all(void *w, const void *v0, const void *V, size_t vstride, int nvec, const void *h, double sign, size_t rows,
             int k, bool init, void *norm, cudaStream_t s) {
  const int pack = pack_at<T>(k, vstride, {w, v0, V});
  if (k / pack > DT) throw cuda_error{cudaErrorInvalidValue, "multiaxpy: more column groups than threads"};
  const int group = std::max(1, AXPY_SMEM / (k * (int)sizeof(T)));
  const int parts = multiaxpy_norm_parts(type_of<T>(), rows, k);
  int passes = 0;
  for (int i0 = 0; i0 < nvec; i0 += group) {
    const int nv = std::min(nvec - i0, group);
    const bool first = init && i0 == 0, last = i0 + nv >= nvec;
    const size_t smem = (size_t)nv * k * sizeof(T);
    with_pack<T>(pack, [&](auto vec) {
      auto go = [&](auto ini) {
        k_axpy<T, H, decltype(vec)::value, decltype(ini)::value><<<parts, DT, smem, s>>>(
            (T *)w, (const T *)v0, (const T *)V, vstride, i0, nv, (const H *)h, sign, rows, k, last ? (double *)norm : nullptr);
      };
      if (first) go(std::true_type());
      else go(std::false_type());
    });
    MLMC_LAUNCH_CHECK("k_axpy");
    ++passes;
  }
  return passes;
}

}  // namespace

int launch_multiaxpy(DType t, void *w, const void *V, size_t vstride, int nvec, const void *h, double sign,
                     size_t rows, int k, bool init, cudaStream_t s) {
  int passes = 0;
  if (nvec <= 0) return passes;
  MLMC_DISPATCH(t, T, passes = (axpy_all<T, typename acc_of<T>::type>(w, V, V, vstride, nvec, h, sign, rows, k, init,
                                                                      nullptr, s)));
  return passes;
}

// ------------------------------------------------------------------ fixed-length FGMRES, per column
// The solver keeps its basis unnormalised: u_0 = b, A z_j = sum_{i <= j} c_ij u_i + u_{j+1} with
// c_ij = d_ij / n_i, d_ij = u_i^* A z_j, n_i = |u_i|^2.  k_fgmres_mid turns step j's partial dot
// products into the coefficients -c_ij of the multi-AXPY; k_fgmres_tail does the last step's
// and then solves min || s_0 e_1 - G y ||, G_ij = d_ij / s_i (i <= j), G_{j+1,j} = s_{j+1}, with
// s_i = sqrt(n_i), by Givens rotations; x = sum_j y_j z_j.  The norm of the last residual
// vector u_m is needed only inside G, so it is taken as n_m = |w|^2 - sum_i |d_i|^2 / n_i
// (w = A z_{m-1}) and u_m is never formed: a relative error eps in the dot products enters
// R_mm^2 as eps |w|^2, the size of the other entries' errors.  Where w lies in the span of the
// earlier A z_j, R_mm itself vanishes and the difference is rounding of either sign; it is then held
// at the unit roundoff of |w|^2, which is at least its error, so that y_m is damped and the last
// step never adds to the residual (a preconditioner of rank one: up to 0.0065 |b| without).
// Residuals after 1 .. 32 steps on eight hierarchies agree with those of the formed norm to four
// digits, down to where FP32 or FP64 stagnates.
// Columns whose right-hand side is zero or not finite, and columns that break down (a zero
// new vector or a zero pivot), stop there: their later y are zero.
// Both kernels give a block a few columns and let all its threads add the parts (latency-
// bound); a tile is two scalars wide, since the FP64 additions of one block's share would
// otherwise take longer than its loads.  Per step they stand in place of two
// reductions of one warp per output (4.7 us each, strided loads), a cleared counter and a
// per-column Givens kernel (4.7 us, 9 us complex; a 4-byte memset node costs 4 us and the
// kernel after it 5 us of gap in a replayed graph).  Two steps, 64 columns, 152 parts: k_fgmres_mid
// 3.3 us and k_fgmres_tail 6.7 (FP32), 4.3 and 8.3 (complex FP32, 304 parts), 4.2 and 7.6 (FP64);
// mostly dependent FP64 instructions, so what earlier steps left is loaded before the sums, and
// the norm of u_j is added up with the dots.  Tiles of eight scalars with float-pair parts took
// 3.8 and 8.6 us (FP32).
namespace {

template <class T> struct fg {
  typedef typename acc_of<T>::type H;
  static constexpr int C = lane_of<T>::C;
  static constexpr int ET = 2;                   // scalars per tile
  static constexpr int CB = ET / C;              // columns per tile
  static constexpr int SL = RT / ET;             // part slices
  static constexpr int MAXROWS = 34;             // 32 steps, v0.v0, w.w
};

// sums[r * ET + e] (r < nrows, e < ET) = scalar e0 + e of output row r summed over the parts in
// fixed order; parts are nrows * E scalars apart, rows E.  With norm (nullable; parts k columns
// apart) also nsum[c] = column c0 + c of it, c < CB, in the same pass.  red: (TR + 1) * RT sums.
constexpr int TR = 8;              // rows whose loads are in flight together
template <class T>
__device__ void tile_sum(const double *__restrict__ partial, int nparts, int nrows, int E, int e0,
                         const double *__restrict__ norm, int norm_parts, int k, int c0, double *red, double *sums,
                         double *nsum) {
  constexpr int ET = fg<T>::ET, SL = fg<T>::SL, CB = fg<T>::CB;
  const int e = threadIdx.x % ET, sl = threadIdx.x / ET;
  const size_t stride = (size_t)nrows * E;
  for (int r0 = 0; r0 < nrows; r0 += TR) {
    const int nr = min(nrows - r0, TR);
    const bool with_norm = r0 == 0 && norm;
    const int used = min(SL, with_norm ? max(nparts, norm_parts) : nparts);   // slices that hold anything
    double a[TR], an = 0.0;
#pragma unroll
    for (int r = 0; r < TR; ++r) a[r] = 0.0;
    if (with_norm && e < CB && c0 + e < k && sl < norm_parts) {
      an = norm[(size_t)sl * k + c0 + e];
      for (int p = sl + SL; p < norm_parts; p += SL) an += norm[(size_t)p * k + c0 + e];
    }
    if (e0 + e < E && sl < nparts) {
      const double *src = partial + (size_t)r0 * E + e0 + e;
#pragma unroll
      for (int r = 0; r < TR; ++r)
        if (r < nr) a[r] = src[sl * stride + (size_t)r * E];
      for (int p = sl + SL; p < nparts; p += SL) {
        double v[TR];
#pragma unroll
        for (int r = 0; r < TR; ++r)
          if (r < nr) v[r] = src[p * stride + (size_t)r * E];
#pragma unroll
        for (int r = 0; r < TR; ++r)
          if (r < nr) a[r] += v[r];
      }
    }
#pragma unroll
    for (int r = 0; r < TR; ++r)
      if (r < nr) red[(r * SL + sl) * ET + e] = a[r];
    if (with_norm) red[(nr * SL + sl) * ET + e] = an;
    const int rows = nr + with_norm;
    __syncthreads();
    // 16 threads per sum take the slices q, q + 16, ...; then one adds the 16
    for (int t = threadIdx.x; t < rows * ET * 16; t += RT) {
      const int ee = t % ET, q = t / ET % 16, r = t / (ET * 16);
      double v = red[(r * SL + q) * ET + ee];
#pragma unroll 4
      for (int s2 = q + 16; s2 < used; s2 += 16) v += red[(r * SL + s2) * ET + ee];
      red[(r * SL + q) * ET + ee] = v;
    }
    __syncthreads();
    for (int re = threadIdx.x; re < rows * ET; re += RT) {
      const int r = re / ET, ee = re % ET;
      double v = red[(r * SL) * ET + ee];
#pragma unroll
      for (int q = 1; q < 16; ++q) v += red[(r * SL + q) * ET + ee];
      if (r < nr) sums[(r0 + r) * ET + ee] = v;
      else if (ee < CB) nsum[ee] = v;
    }
    __syncthreads();
  }
}

__device__ __forceinline__ double usable(double n) { return n > 0.0 && isfinite(n) ? n : 1.0; }

__device__ __forceinline__ double at(const double *s, int c, double) { return s[c]; }
__device__ __forceinline__ cdouble at(const double *s, int c, cdouble) { return {s[2 * c], s[2 * c + 1]}; }
__device__ __forceinline__ double shfl(double v, int l) { return __shfl_sync(0xffffffffu, v, l); }
__device__ __forceinline__ cdouble shfl(cdouble v, int l) { return {shfl(v.re, l), shfl(v.im, l)}; }

}  // namespace

// The tile's sums for step j: dots (rows d_0 .. d_j, then v0.v0 when j = 0, then extra rows)
// into sums, and n_j into nj[c] (shared) and n2[j] (global).
template <class T>
__device__ void fgmres_sums(const double *partial, int nparts, int nrows,
                            const double *norm, int norm_parts, int j, int k, int c0, double *n2,
                            double *red, double *sums, double *nj) {
  constexpr int C = fg<T>::C, ET = fg<T>::ET, CB = fg<T>::CB;
  tile_sum<T>(partial, nparts, nrows, k * C, c0 * C, j > 0 ? norm : nullptr, norm_parts, k, c0, red, sums, nj);
  if (threadIdx.x < CB) {
    const int c = threadIdx.x;
    if (j == 0) nj[c] = sums[ET + c * C];
    if (c0 + c < k) n2[(size_t)j * k + c0 + c] = nj[c];
  }
  __syncthreads();
}

// D[(j * (m + 1) + i) * k + c] = d_ij, coef[i * k + c] = -d_ij / n_i for the multi-AXPY of step j.
template <class T>
__global__ void __launch_bounds__(RT) k_fgmres_mid(const double *__restrict__ partial, int nparts,
                                                   int nrows, const double *__restrict__ norm,
                                                   int norm_parts, int j, int m, int k, double *n2,
                                                   typename acc_of<T>::type *__restrict__ D, T *__restrict__ coef) {
  typedef typename acc_of<T>::type H;
  constexpr int ET = fg<T>::ET, CB = fg<T>::CB;
  __shared__ double red[(TR + 1) * RT];
  __shared__ double sums[fg<T>::MAXROWS * ET], nj[8];
  const int c0 = blockIdx.x * CB;
  // thread (i, c): the norm of u_i is loaded before the sums (at most 32 vectors x 8 columns)
  const int i = threadIdx.x / CB, c = threadIdx.x - (threadIdx.x / CB) * CB;
  const bool mine = i <= j && c0 + c < k;
  double n = mine && i < j ? n2[(size_t)i * k + c0 + c] : 0.0;
  fgmres_sums<T>(partial, nparts, nrows, norm, norm_parts, j, k, c0, n2, red, sums, nj);
  if (!mine) return;
  n = usable(i == j ? nj[c] : n);
  const H d = at(sums + i * ET, c, H());
  D[((size_t)j * (m + 1) + i) * k + c0 + c] = d;
  coef[(size_t)i * k + c0 + c] = cvt<T, H>(rmul(-1.0 / n, d));
}

// The last step, j = its - 1, and the least-squares problem: y[i * k + c], i < its.
// One warp per column; lane q keeps column q of G, and the norm of u_q.
template <class T>
__global__ void __launch_bounds__(RT) k_fgmres_tail(const double *__restrict__ partial, int nparts,
                                                    int nrows, const double *__restrict__ norm,
                                                    int norm_parts, int its, int m, int k, double *n2,
                                                    const typename acc_of<T>::type *__restrict__ D,
                                                    T *__restrict__ y) {
  typedef typename acc_of<T>::type H;
  constexpr int ET = fg<T>::ET, CB = fg<T>::CB, C = fg<T>::C;
  __shared__ double red[(TR + 1) * RT];
  __shared__ double sums[fg<T>::MAXROWS * ET], nj[8];
  extern __shared__ __align__(16) unsigned char tail_smem[];
  const int c0 = blockIdx.x * CB, j = its - 1;
  const int c = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool mine = c < CB && c0 + c < k;
  const size_t cg = c0 + c;
  H *G = (H *)tail_smem + (size_t)c * (its + 1) * its;      // G[i * its + q], used by warp c < CB
  // what earlier steps left is loaded before the sums: norms, and the dots d_iq of the columns q < j
  double n = mine && lane < j ? n2[(size_t)lane * k + cg] : 0.0;
  if (mine && lane < j)
    for (int i = 0; i <= lane; ++i) G[i * its + lane] = D[((size_t)lane * (m + 1) + i) * k + cg];
  fgmres_sums<T>(partial, nparts, nrows, norm, norm_parts, j, k, c0, n2, red, sums, nj);
  if (!mine) return;
  // norms s_q = sqrt(n_q): zero for a vanished vector, whose 1 / s_q is 1
  if (lane == j) n = nj[c];
  const double is = lane < its ? rsqrt(usable(n)) : 0.0;
  const double sq = lane < its && n > 0.0 && isfinite(n) ? n * is : 0.0;
  // n_its = |w|^2 - sum_q |d_q|^2 / n_q
  const H dl = lane < its ? at(sums + lane * ET, c, H()) : zero<H>();
  double part = abs2(rmul(is, dl));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
  const double w2 = sums[(nrows - 1) * ET + c * C];
  const double nl = fmax(w2 - part, w2 * (sizeof(typename real_of<T>::type) == 4 ? 0x1p-24 : 0x1p-53));
  const double sl = nl > 0.0 && isfinite(nl) ? nl * rsqrt(nl) : 0.0;
  const double below = __shfl_down_sync(0xffffffffu, sq, 1);   // s_{q+1}, the subdiagonal of column q
  if (lane == j)
    for (int i = 0; i < its; ++i) G[i * its + lane] = at(sums + i * ET, c, H());
  for (int i = 0; i < its; ++i) {
    const double v = __shfl_sync(0xffffffffu, is, i);
    if (lane >= i && lane < its) G[i * its + lane] = rmul(v, G[i * its + lane]);
  }
  if (lane < its) G[(lane + 1) * its + lane] = make<H>(lane == j ? sl : below, 0.0);
  __syncwarp();
  const double s0 = __shfl_sync(0xffffffffu, sq, 0);
  H g = make<H>(s0, 0.0), gi = zero<H>();                   // lane i keeps entry i of the rotated right-hand side
  double inv = 0.0;                                         // and 1 / R_ii
  bool active = s0 > 0.0;
  int J = 0;
  for (int i = 0; i < its && active; ++i) {
    const H a = G[i * its + i];
    const double b = re(G[(i + 1) * its + i]), r2 = abs2(a) + b * b;
    if (!(r2 > 0.0)) break;
    const double ir = rsqrt(r2);
    const H cc = rmul(ir, a);
    const double ss = b * ir;
    if (lane > i && lane < its) {
      const H u = G[i * its + lane], v = G[(i + 1) * its + lane];
      G[i * its + lane] = conj(cc) * u + rmul(ss, v);
      G[(i + 1) * its + lane] = cc * v - rmul(ss, u);
    }
    if (lane == i) {
      gi = conj(cc) * g;
      inv = ir;
    }
    g = rmul(-ss, g);
    J = i + 1;
    active = b > 0.0;
    __syncwarp();
  }
  for (int l = J - 1; l >= 0; --l) {
    H yl = rmul(inv, gi);
    yl = shfl(yl, l);
    if (lane < l) gi = gi - G[lane * its + l] * yl;
    if (lane == l) gi = yl;
  }
  if (lane < its) y[(size_t)lane * k + cg] = cvt<T, H>(lane < J ? gi : zero<H>());
}

// Step j's partial dots of w against u_0 = b, u_1 .. u_j (V + i * vstride), with b.b on the first
// step and w.w on the last.
int launch_fgmres_dots(DType t, const void *b, const void *V, size_t vstride, int j, int its, const void *w, size_t rows,
                       int k, void *partials, cudaStream_t s) {
  const int extra = (j == 0 ? 2 : 0) | (j == its - 1 ? 1 : 0);
  int passes = 0;
  MLMC_DISPATCH(t, T, passes = dots_partial<T>(b, V, vstride, j + 1, w, rows, k, partials, multidot_parts(t, rows, k),
                                               extra, s));
  return passes;
}

void launch_fgmres_mid(DType t, const void *partials, const void *norm, int j, int m, size_t rows, int k, double *n2,
                       void *D, void *coef, cudaStream_t s) {
  const int nparts = multidot_parts(t, rows, k), nnorm = multiaxpy_norm_parts(t, rows, k);
  MLMC_DISPATCH(t, T, {
    typedef typename acc_of<T>::type H;
    k_fgmres_mid<T><<<(k + fg<T>::CB - 1) / fg<T>::CB, RT, 0, s>>>((const double *)partials, nparts, j + 1 + (j == 0),
                                                                  (const double *)norm, nnorm, j, m, k, n2, (H *)D,
                                                                  (T *)coef);
  });
  MLMC_LAUNCH_CHECK("k_fgmres_mid");
}

void launch_fgmres_tail(DType t, const void *partials, const void *norm, int its, int m, size_t rows, int k,
                        double *n2, const void *D, void *y, cudaStream_t s) {
  const int nparts = multidot_parts(t, rows, k), nnorm = multiaxpy_norm_parts(t, rows, k);
  MLMC_DISPATCH(t, T, {
    typedef typename acc_of<T>::type H;
    auto bytes = [](int n) { return (size_t)fg<T>::CB * (n + 1) * n * sizeof(H); };
    int dev = 0;
    MLMC_CUDA(cudaGetDevice(&dev));
    // the longest solve (32 steps) sets the limit once per device: every later value is smaller
    static std::once_flag once[64];
    std::call_once(once[dev & 63], [&] {
      check_cuda(cudaFuncSetAttribute(k_fgmres_tail<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes(32)),
                 "cudaFuncSetAttribute(k_fgmres_tail)");
    });
    k_fgmres_tail<T><<<(k + fg<T>::CB - 1) / fg<T>::CB, RT, bytes(its), s>>>(
        (const double *)partials, nparts, its + 1 + (its == 1), (const double *)norm, nnorm, its, m, k, n2, (const H *)D, (T *)y);
  });
  MLMC_LAUNCH_CHECK("k_fgmres_tail");
}

// w += sum_v u_v coef[v][c] (u_0 = b, then V + v * vstride), with the partial column norms of the result
int launch_fgmres_axpy(DType t, void *w, const void *b, const void *V, size_t vstride, int nvec, const void *coef,
                       size_t rows, int k, void *norm, cudaStream_t s) {
  int passes = 0;
  MLMC_DISPATCH(t, T, passes = (axpy_all<T, T>(w, b, V, vstride, nvec, coef, 1.0, rows, k, false, norm, s)));
  return passes;
}

// x = sum_v Z_v y[v][c]
int launch_fgmres_update(DType t, void *x, const void *Z, size_t vstride, int nvec, const void *y, size_t rows, int k,
                         cudaStream_t s) {
  int passes = 0;
  MLMC_DISPATCH(t, T, passes = (axpy_all<T, T>(x, Z, Z, vstride, nvec, y, 1.0, rows, k, true, nullptr, s)));
  return passes;
}

}  // namespace mlmc
