// The paper's hierarchy for Example 5.1 (Sec. 5): bilinear interpolation
// between grids N_l = 2 N_{l+1} + 1 (coarse point I on fine point 2I + 1,
// Dirichlet), its adjoint as restriction (full weighting without the 1/4),
// and the 9-point Galerkin operators of the coarse levels with their
// 4-colour Gauss-Seidel smoother.
//
// Layout: a 9-point operator is coef[site][9] with taps 0 self, 1 +x, 2 -x,
// 3 +y, 4 -y, 5 (+x,+y), 6 (-x,+y), 7 (+x,-y), 8 (-x,-y); taps that leave the
// grid are zero and never followed.  Vector blocks are [site][k] (d = 1) with
// the k right-hand sides innermost; one thread handles VEC consecutive
// columns of one site with 16-byte loads, grid.y is the lattice row.
#include <type_traits>

#include "mlmc_internal.cuh"

namespace mlmc {

namespace {

template <class T, int VEC> struct alignas(sizeof(T) * VEC) PackB { T v[VEC]; };

// the taps' offsets, folded into the unrolled loops (arrays in constant memory are loads there)
__host__ __device__ constexpr int tap_dx(int q) { return q == 1 || q == 5 || q == 7 ? 1 : q == 2 || q == 6 || q == 8 ? -1 : 0; }
__host__ __device__ constexpr int tap_dy(int q) { return q == 3 || q == 5 || q == 6 ? 1 : q == 4 || q == 7 || q == 8 ? -1 : 0; }

template <class T>
int vec_of(int k) {
  const int v = 16 / (int)sizeof(T);
  return k % v == 0 ? v : 1;
}

}  // namespace

// y = A x (mode 0) or y = b - A x (mode 1).
template <class T, int VEC>
__global__ void __launch_bounds__(256) k_stencil9(const T *__restrict__ coef, const T *__restrict__ x,
                                                  const T *__restrict__ b, T *__restrict__ y, int nx, int ny, int kv,
                                                  int mode) {
  typedef PackB<T, VEC> V;
  const int j = blockIdx.y;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nx * kv) return;
  const int i = t / kv, c = t - (t / kv) * kv;
  const int s = j * nx + i;
  const V *X = (const V *)x;
  const T *a = coef + (size_t)s * 9;
  T acc[VEC];
#pragma unroll
  for (int u = 0; u < VEC; ++u) acc[u] = T(0);
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    const int ii = i + tap_dx(q), jj = j + tap_dy(q);
    if (ii < 0 || ii >= nx || jj < 0 || jj >= ny) continue;
    const T w = __ldg(a + q);
    const V xn = X[(size_t)(jj * nx + ii) * kv + c];
#pragma unroll
    for (int u = 0; u < VEC; ++u) acc[u] += w * xn.v[u];
  }
  V out;
  if (mode) {
    const V bb = ((const V *)b)[(size_t)s * kv + c];
#pragma unroll
    for (int u = 0; u < VEC; ++u) out.v[u] = bb.v[u] - acc[u];
  } else {
#pragma unroll
    for (int u = 0; u < VEC; ++u) out.v[u] = acc[u];
  }
  ((V *)y)[(size_t)s * kv + c] = out;
}

// One colour of a 4-colour Gauss-Seidel sweep: for the sites with
// (i mod 2) + 2 (j mod 2) == colour, x_s = dinv_s (b_s - sum_{q != 0} a_q x_nb(q)).
// Sites of one colour do not couple in a 9-point stencil, so this is exact
// Gauss-Seidel in colour order.  grid.y runs over the rows of that parity.
template <class T, int VEC>
__global__ void __launch_bounds__(256) k_gs9_colour(const T *__restrict__ coef, const T *__restrict__ dinv,
                                                    T *__restrict__ x, const T *__restrict__ b, int nx, int ny, int kv,
                                                    int colour) {
  typedef PackB<T, VEC> V;
  const int j = 2 * blockIdx.y + (colour >> 1);
  const int i0 = colour & 1;
  const int hx = (nx - i0 + 1) >> 1;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= ny || t >= hx * kv) return;
  const int m = t / kv, c = t - (t / kv) * kv;
  const int i = 2 * m + i0;
  const int s = j * nx + i;
  V *X = (V *)x;
  const T *a = coef + (size_t)s * 9;
  V acc = ((const V *)b)[(size_t)s * kv + c];
#pragma unroll
  for (int q = 1; q < 9; ++q) {
    const int ii = i + tap_dx(q), jj = j + tap_dy(q);
    if (ii < 0 || ii >= nx || jj < 0 || jj >= ny) continue;
    const T w = __ldg(a + q);
    const V xn = X[(size_t)(jj * nx + ii) * kv + c];
#pragma unroll
    for (int u = 0; u < VEC; ++u) acc.v[u] -= w * xn.v[u];
  }
  const T di = __ldg(dinv + s);
#pragma unroll
  for (int u = 0; u < VEC; ++u) acc.v[u] *= di;
  X[(size_t)s * kv + c] = acc;
}

// rc[I, J] = sum_{a, b in {-1, 0, 1}} w_a w_b r[2I+1+a, 2J+1+b], w_0 = 1, w_{+-1} = 1/2
// (R = P^T of bilinear interpolation); every fine index is inside the grid.
template <class T, int VEC>
__global__ void __launch_bounds__(256) k_restrict_bilinear(const T *__restrict__ r, T *__restrict__ rc, int nxc,
                                                           int nyc, int kv) {
  typedef PackB<T, VEC> V;
  const int J = blockIdx.y;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nxc * kv) return;
  const int I = t / kv, c = t - (t / kv) * kv;
  const int nx = 2 * nxc + 1;
  const V *R = (const V *)r;
  T acc[VEC];
#pragma unroll
  for (int u = 0; u < VEC; ++u) acc[u] = T(0);
#pragma unroll
  for (int bb = -1; bb <= 1; ++bb) {
#pragma unroll
    for (int aa = -1; aa <= 1; ++aa) {
      const T w = T((aa == 0 ? 1.0 : 0.5) * (bb == 0 ? 1.0 : 0.5));
      const V v = R[(size_t)((2 * J + 1 + bb) * nx + 2 * I + 1 + aa) * kv + c];
#pragma unroll
      for (int u = 0; u < VEC; ++u) acc[u] += w * v.v[u];
    }
  }
  V out;
#pragma unroll
  for (int u = 0; u < VEC; ++u) out.v[u] = acc[u];
  ((V *)rc)[(size_t)(J * nxc + I) * kv + c] = out;
}

// x[i, j] += (P ec)[i, j]: odd i takes coarse column (i-1)/2 with weight 1, even i
// the columns i/2 - 1 and i/2 with weight 1/2 each (those inside the coarse grid);
// the same in y.
template <class T, int VEC>
__global__ void __launch_bounds__(256) k_prolong_bilinear(const T *__restrict__ ec, T *__restrict__ x, int nx, int ny,
                                                          int kv) {
  typedef PackB<T, VEC> V;
  const int j = blockIdx.y;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nx * kv) return;
  const int i = t / kv, c = t - (t / kv) * kv;
  const int nxc = (nx - 1) / 2, nyc = (ny - 1) / 2;
  // two candidate coarse columns / rows each, weight 0 where one does not exist
  // (its index clamped into the grid, so every load stays in bounds)
  int ia, ib, ja, jb;
  T wa, wb, va, vb;
  if (i & 1) { ia = ib = (i - 1) >> 1; wa = T(1); wb = T(0); }
  else {
    ia = i / 2 - 1; ib = i / 2;
    wa = ia >= 0 ? T(0.5) : T(0); wb = ib < nxc ? T(0.5) : T(0);
    ia = ia < 0 ? 0 : ia; ib = ib >= nxc ? nxc - 1 : ib;
  }
  if (j & 1) { ja = jb = (j - 1) >> 1; va = T(1); vb = T(0); }
  else {
    ja = j / 2 - 1; jb = j / 2;
    va = ja >= 0 ? T(0.5) : T(0); vb = jb < nyc ? T(0.5) : T(0);
    ja = ja < 0 ? 0 : ja; jb = jb >= nyc ? nyc - 1 : jb;
  }
  const V *E = (const V *)ec;
  V *X = (V *)x;
  V acc = X[(size_t)(j * nx + i) * kv + c];
  const V e00 = E[(size_t)(ja * nxc + ia) * kv + c], e01 = E[(size_t)(ja * nxc + ib) * kv + c];
  const V e10 = E[(size_t)(jb * nxc + ia) * kv + c], e11 = E[(size_t)(jb * nxc + ib) * kv + c];
#pragma unroll
  for (int u = 0; u < VEC; ++u)
    acc.v[u] += va * (wa * e00.v[u] + wb * e01.v[u]) + vb * (wa * e10.v[u] + wb * e11.v[u]);
  X[(size_t)(j * nx + i) * kv + c] = acc;
}

namespace {

template <class F>
void real_dispatch(DType t, int k, F &&f) {
  if (t == F64) {
    if (vec_of<double>(k) == 2) f(double(), std::integral_constant<int, 2>());
    else f(double(), std::integral_constant<int, 1>());
  } else if (t == F32) {
    if (vec_of<float>(k) == 4) f(float(), std::integral_constant<int, 4>());
    else f(float(), std::integral_constant<int, 1>());
  } else {
    throw cuda_error{cudaErrorInvalidValue, "the bilinear hierarchy is real (Example 5.1)"};
  }
}

}  // namespace

void launch_stencil9(const StencilView &A, const void *x, const void *b, void *y, int k, int mode, cudaStream_t s) {
  real_dispatch(A.t, k, [&](auto tag, auto vtag) {
    typedef decltype(tag) T;
    constexpr int VEC = decltype(vtag)::value;
    const int kv = k / VEC;
    dim3 g((A.nx * kv + 255) / 256, A.ny);
    k_stencil9<T, VEC><<<g, 256, 0, s>>>((const T *)A.coef, (const T *)x, (const T *)b, (T *)y, A.nx, A.ny, kv, mode);
  });
  MLMC_LAUNCH_CHECK("k_stencil9");
}

void launch_gs9_sweep(const StencilView &A, void *x, const void *b, int k, int order, int x_zero, cudaStream_t s) {
  if (x_zero) MLMC_CUDA(cudaMemsetAsync(x, 0, (size_t)A.nx * A.ny * k * dtype_size(A.t), s));
  real_dispatch(A.t, k, [&](auto tag, auto vtag) {
    typedef decltype(tag) T;
    constexpr int VEC = decltype(vtag)::value;
    const int kv = k / VEC;
    for (int q = 0; q < 4; ++q) {
      const int colour = order == 0 ? q : 3 - q;
      const int hx = (A.nx - (colour & 1) + 1) >> 1;
      const int rows = (A.ny - (colour >> 1) + 1) >> 1;
      if (hx <= 0 || rows <= 0) continue;
      dim3 g((hx * kv + 255) / 256, rows);
      k_gs9_colour<T, VEC><<<g, 256, 0, s>>>((const T *)A.coef, (const T *)A.dinv, (T *)x, (const T *)b, A.nx, A.ny,
                                             kv, colour);
    }
  });
  MLMC_LAUNCH_CHECK("k_gs9_colour");
}

void launch_restrict_bilinear(DType t, const void *r, void *rc, int nxc, int nyc, int k, cudaStream_t s) {
  real_dispatch(t, k, [&](auto tag, auto vtag) {
    typedef decltype(tag) T;
    constexpr int VEC = decltype(vtag)::value;
    const int kv = k / VEC;
    dim3 g((nxc * kv + 255) / 256, nyc);
    k_restrict_bilinear<T, VEC><<<g, 256, 0, s>>>((const T *)r, (T *)rc, nxc, nyc, kv);
  });
  MLMC_LAUNCH_CHECK("k_restrict_bilinear");
}

void launch_prolong_bilinear(DType t, const void *ec, void *x, int nx, int ny, int k, cudaStream_t s) {
  real_dispatch(t, k, [&](auto tag, auto vtag) {
    typedef decltype(tag) T;
    constexpr int VEC = decltype(vtag)::value;
    const int kv = k / VEC;
    dim3 g((nx * kv + 255) / 256, ny);
    k_prolong_bilinear<T, VEC><<<g, 256, 0, s>>>((const T *)ec, (T *)x, nx, ny, kv);
  });
  MLMC_LAUNCH_CHECK("k_prolong_bilinear");
}

// ------------------------------------------------------------------ small levels, one block per column pack
// A cycle on a 9-point level is a dozen launches (four colours per sweep, residual, transfers)
// of 2 - 4 us each, whatever the level's size, and a K-cycle visits the small levels most.
// Columns are independent, so on the smallest levels a block takes one pack of columns, its x in
// shared memory, through everything before the coarse solve in one launch, and through
// everything after it in another, with block barriers between the colours.  The residual is
// not formed: its restriction is R b - (R A) x with the 25-point rows of R A formed at setup.
// Coefficients are read as [tap][site] arrays, so that a warp's consecutive sites are
// coalesced; a thread's next site is loaded while it solves one.
// Vectors are [site][k], so a block touches every site's own cache line for its few columns,
// which takes the load unit a clock each: the time grows with the sites, and from 63^2 on
// (36 us per cycle and one sweep each way, 48 columns) the separate launches (32 us) win;
// 31^2: 15.4 against 32 us.
constexpr int S9_THREADS = 512;

// One site's 4-colour Gauss-Seidel data: the off-diagonal taps, 1 / diagonal and b.
template <class T, int VEC> struct Site9 {
  T w[8], di;
  PackB<T, VEC> b;
  int s;
  unsigned on;       // which of the eight neighbours lie in the grid
};

template <class T, int VEC>
__device__ __forceinline__ bool site9_load(Site9<T, VEC> &o, const T *__restrict__ ct, const T *__restrict__ dinv,
                                           const PackB<T, VEC> *B, int nx, int ny, int kv, int c, int colour, int idx) {
  const int i0 = colour & 1, hx = (nx - i0 + 1) >> 1, hy = (ny - (colour >> 1) + 1) >> 1;
  if (idx >= hx * hy) return false;
  const int m = idx / hx, i = 2 * (idx - m * hx) + i0, j = 2 * m + (colour >> 1), n = nx * ny;
  o.s = j * nx + i;
  o.b = B[(size_t)o.s * kv + c];
  o.di = __ldg(dinv + o.s);
  o.on = 0;
#pragma unroll
  for (int q = 1; q < 9; ++q) {
    const int ii = i + tap_dx(q), jj = j + tap_dy(q);
    o.on |= (unsigned)(ii >= 0 && ii < nx && jj >= 0 && jj < ny) << q;
    o.w[q - 1] = __ldg(ct + q * n + o.s);
  }
  return true;
}

template <class T, int VEC>
__device__ __forceinline__ void site9_solve(const Site9<T, VEC> &o, PackB<T, VEC> *X, int nx) {
  PackB<T, VEC> acc = o.b;
#pragma unroll
  for (int q = 1; q < 9; ++q)
    if (o.on >> q & 1) {
      const PackB<T, VEC> xn = X[o.s + tap_dy(q) * nx + tap_dx(q)];
#pragma unroll
      for (int u = 0; u < VEC; ++u) acc.v[u] -= o.w[q - 1] * xn.v[u];
    }
#pragma unroll
  for (int u = 0; u < VEC; ++u) acc.v[u] *= o.di;
  X[o.s] = acc;
}

// `sweeps` 4-colour sweeps over X in shared memory (order 0: colours 0..3, 1: 3..0).  Starts and
// ends with the block synchronised.
template <class T, int VEC>
__device__ void sweeps9(PackB<T, VEC> *X, const T *ct, const T *dinv, const PackB<T, VEC> *B, int nx, int ny, int kv,
                        int c, int sweeps, int order) {
  auto colour_of = [&](int st) { return order ? 3 - (st & 3) : st & 3; };
  auto rounds_of = [&](int colour) {
    return (((nx - (colour & 1) + 1) >> 1) * ((ny - (colour >> 1) + 1) >> 1) + S9_THREADS - 1) / S9_THREADS;
  };
  Site9<T, VEC> cur, next;
  bool have = site9_load<T, VEC>(cur, ct, dinv, B, nx, ny, kv, c, colour_of(0), threadIdx.x), have_next = false;
  const int steps = sweeps * 4;
  for (int st = 0; st < steps; ++st) {
    const int colour = colour_of(st), rounds = rounds_of(colour);
    for (int rd = 0; rd < rounds; ++rd) {
      // the thread's next site, of this colour or the next, is loaded while this one is solved
      if (rd + 1 < rounds)
        have_next = site9_load<T, VEC>(next, ct, dinv, B, nx, ny, kv, c, colour, threadIdx.x + (rd + 1) * S9_THREADS);
      else
        have_next = st + 1 < steps &&
                    site9_load<T, VEC>(next, ct, dinv, B, nx, ny, kv, c, colour_of(st + 1), threadIdx.x);
      if (have) site9_solve<T, VEC>(cur, X, nx);
      cur = next;
      have = have_next;
    }
    __syncthreads();
  }
}

// x = `sweeps` sweeps from zero, rc = R (b - A x)
template <class T, int VEC>
__global__ void __launch_bounds__(S9_THREADS) k_cycle9_down(const T *__restrict__ ct, const T *__restrict__ dinv,
                                                               const T *__restrict__ ra, const T *b, T *x, T *rc,
                                                               int nx, int ny, int kv, int sweeps) {
  typedef PackB<T, VEC> V;
  extern __shared__ __align__(16) unsigned char s9_smem[];
  V *X = (V *)s9_smem;
  const int c = blockIdx.x, n = nx * ny;
  const V *B = (const V *)b;
  for (int e = threadIdx.x; e < n; e += S9_THREADS) {
    V z;
#pragma unroll
    for (int u = 0; u < VEC; ++u) z.v[u] = T(0);
    X[e] = z;
  }
  __syncthreads();
  sweeps9<T, VEC>(X, ct, dinv, B, nx, ny, kv, c, sweeps, 0);
  for (int e = threadIdx.x; e < n; e += S9_THREADS) ((V *)x)[(size_t)e * kv + c] = X[e];
  const int nxc = (nx - 1) / 2, nyc = (ny - 1) / 2, nc = nxc * nyc;
  for (int e = threadIdx.x; e < nc; e += S9_THREADS) {
    const int J = e / nxc, I = e - J * nxc, p = (2 * J + 1) * nx + 2 * I + 1;
    T acc[VEC];
#pragma unroll
    for (int u = 0; u < VEC; ++u) acc[u] = T(0);
#pragma unroll
    for (int bb = -1; bb <= 1; ++bb)
#pragma unroll
      for (int aa = -1; aa <= 1; ++aa) {
        const T w = T((aa == 0 ? 1.0 : 0.5) * (bb == 0 ? 1.0 : 0.5));
        const V v = B[(size_t)(p + bb * nx + aa) * kv + c];
#pragma unroll
        for (int u = 0; u < VEC; ++u) acc[u] += w * v.v[u];
      }
    // columns 2I - 1 .. 2I + 3 and rows 2J - 1 .. 2J + 3, those in the grid
#pragma unroll
    for (int dy = -2; dy <= 2; ++dy) {
      const int jj = 2 * J + 1 + dy;
      if (jj < 0 || jj >= ny) continue;
#pragma unroll
      for (int dx = -2; dx <= 2; ++dx) {
        const int ii = 2 * I + 1 + dx;
        if (ii < 0 || ii >= nx) continue;
        const T w = __ldg(ra + ((dy + 2) * 5 + dx + 2) * nc + e);
        const V v = X[jj * nx + ii];
#pragma unroll
        for (int u = 0; u < VEC; ++u) acc[u] -= w * v.v[u];
      }
    }
    V out;
#pragma unroll
    for (int u = 0; u < VEC; ++u) out.v[u] = acc[u];
    ((V *)rc)[(size_t)e * kv + c] = out;
  }
}

// x += P ec, then `sweeps` sweeps in reverse colour order
template <class T, int VEC>
__global__ void __launch_bounds__(S9_THREADS) k_cycle9_up(const T *__restrict__ ct, const T *__restrict__ dinv,
                                                             const T *b, const T *ec, T *x, int nx, int ny, int kv,
                                                             int sweeps) {
  typedef PackB<T, VEC> V;
  extern __shared__ __align__(16) unsigned char s9_smem[];
  V *X = (V *)s9_smem;
  const int c = blockIdx.x, n = nx * ny, nxc = (nx - 1) / 2, nyc = (ny - 1) / 2;
  const V *E = (const V *)ec;
  V *xg = (V *)x;
  for (int e = threadIdx.x; e < n; e += S9_THREADS) {
    const int j = e / nx, i = e - j * nx;
    V acc;
#pragma unroll
    for (int u = 0; u < VEC; ++u) acc.v[u] = T(0);
    if (!(i & j & 1)) {                    // colour 3 is overwritten first, without being read
      // odd i: coarse column (i - 1) / 2; even i: the columns i/2 - 1 and i/2, half each
      const int ia = (i + 1) / 2 - 1, ib = i / 2, ja = (j + 1) / 2 - 1, jb = j / 2;
      const T wi = (i & 1) ? T(1) : T(0.5), wj = (j & 1) ? T(1) : T(0.5);
      acc = xg[(size_t)e * kv + c];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int I = q & 1 ? ib : ia, J = q >> 1 ? jb : ja;
        if (((q & 1) && (i & 1)) || ((q >> 1) && (j & 1)) || I < 0 || I >= nxc || J < 0 || J >= nyc) continue;
        const V v = E[(size_t)(J * nxc + I) * kv + c];
#pragma unroll
        for (int u = 0; u < VEC; ++u) acc.v[u] += (wi * wj) * v.v[u];
      }
    }
    X[e] = acc;
  }
  __syncthreads();
  sweeps9<T, VEC>(X, ct, dinv, (const V *)b, nx, ny, kv, c, sweeps, 1);
  for (int e = threadIdx.x; e < n; e += S9_THREADS) xg[(size_t)e * kv + c] = X[e];
}

namespace {

// Columns per block: the narrowest pack that k allows, whose x fits in the shared memory of a
// block and that leaves no more blocks than SMs (a block's shared-memory reads, and its share
// of the SMs' time, grow with its columns); else the widest that fits.  0: none.
int cycle9_pack(const StencilView &A, int k) {
  const size_t n = (size_t)A.nx * A.ny, es = dtype_size(A.t);
  int best = 0;
  for (int v = 1; v * es <= 16; v *= 2) {
    if (k % v || n * v * es > 48 * 1024) continue;
    best = v;
    if (k / v <= 152) break;
  }
  return best;
}

template <class F>
void cycle9_dispatch(const StencilView &A, int k, F &&f) {
  const int v = cycle9_pack(A, k);
  const size_t smem = (size_t)A.nx * A.ny * v * dtype_size(A.t);
  if (A.t == F32) {
    if (v == 4) f(float(), std::integral_constant<int, 4>(), k / 4, smem);
    else if (v == 2) f(float(), std::integral_constant<int, 2>(), k / 2, smem);
    else f(float(), std::integral_constant<int, 1>(), k, smem);
  } else {
    if (v == 2) f(double(), std::integral_constant<int, 2>(), k / 2, smem);
    else f(double(), std::integral_constant<int, 1>(), k, smem);
  }
}

}  // namespace

bool cycle9_ok(const StencilView &A, int k) {
  return A.taps == 9 && A.taps9 && A.ra && (A.t == F32 || A.t == F64) && cycle9_pack(A, k) > 0;
}

void launch_cycle9_down(const StencilView &A, const void *b, void *x, void *rc, int k, int sweeps, cudaStream_t s) {
  cycle9_dispatch(A, k, [&](auto tag, auto vtag, int kv, size_t smem) {
    typedef decltype(tag) T;
    constexpr int VEC = decltype(vtag)::value;
    k_cycle9_down<T, VEC><<<kv, S9_THREADS, smem, s>>>((const T *)A.taps9, (const T *)A.dinv, (const T *)A.ra,
                                                       (const T *)b, (T *)x, (T *)rc, A.nx, A.ny, kv, sweeps);
  });
  MLMC_LAUNCH_CHECK("k_cycle9_down");
}

void launch_cycle9_up(const StencilView &A, const void *b, const void *ec, void *x, int k, int sweeps, cudaStream_t s) {
  cycle9_dispatch(A, k, [&](auto tag, auto vtag, int kv, size_t smem) {
    typedef decltype(tag) T;
    constexpr int VEC = decltype(vtag)::value;
    k_cycle9_up<T, VEC><<<kv, S9_THREADS, smem, s>>>((const T *)A.taps9, (const T *)A.dinv, (const T *)b, (const T *)ec,
                                                     (T *)x, A.nx, A.ny, kv, sweeps);
  });
  MLMC_LAUNCH_CHECK("k_cycle9_up");
}

}  // namespace mlmc
