// Internal header of libmlmc: scalar types, dtype dispatch and the launcher
// declarations shared by the translation units.  Not part of the C ABI.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string>

namespace mlmc {

// ----------------------------------------------------------------- scalars
struct __align__(16) cdouble { double re, im; };
struct __align__(8) cfloat { float re, im; };

// element type of a vector block / operator storage
enum DType : int { F64 = 0, F32 = 1, C64 = 2, C32 = 3 };
inline bool dtype_complex(DType t) { return t == C64 || t == C32; }
inline size_t dtype_size(DType t) { return t == F64 ? 8 : t == F32 ? 4 : t == C64 ? 16 : 8; }
inline DType dtype_lower(DType t) { return t == F64 ? F32 : t == C64 ? C32 : t; }

template <class T> struct real_of { typedef T type; };
template <> struct real_of<cdouble> { typedef double type; };
template <> struct real_of<cfloat> { typedef float type; };

__host__ __device__ inline double re(double a) { return a; }
__host__ __device__ inline float re(float a) { return a; }
__host__ __device__ inline double re(cdouble a) { return a.re; }
__host__ __device__ inline float re(cfloat a) { return a.re; }
__host__ __device__ inline double im(double) { return 0.0; }
__host__ __device__ inline float im(float) { return 0.0f; }
__host__ __device__ inline double im(cdouble a) { return a.im; }
__host__ __device__ inline float im(cfloat a) { return a.im; }

template <class T> __host__ __device__ inline T zero() { return T(0); }
template <> __host__ __device__ inline cdouble zero<cdouble>() { return cdouble{0.0, 0.0}; }
template <> __host__ __device__ inline cfloat zero<cfloat>() { return cfloat{0.0f, 0.0f}; }

template <class T> __host__ __device__ inline T make(double r, double i);
template <> __host__ __device__ inline double make<double>(double r, double) { return r; }
template <> __host__ __device__ inline float make<float>(double r, double) { return (float)r; }
template <> __host__ __device__ inline cdouble make<cdouble>(double r, double i) { return cdouble{r, i}; }
template <> __host__ __device__ inline cfloat make<cfloat>(double r, double i) { return cfloat{(float)r, (float)i}; }

__host__ __device__ inline cdouble operator+(cdouble a, cdouble b) { return {a.re + b.re, a.im + b.im}; }
__host__ __device__ inline cdouble operator-(cdouble a, cdouble b) { return {a.re - b.re, a.im - b.im}; }
__host__ __device__ inline cdouble operator-(cdouble a) { return {-a.re, -a.im}; }
__host__ __device__ inline cdouble operator*(cdouble a, cdouble b) {
  return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
__host__ __device__ inline cdouble operator*(double s, cdouble a) { return {s * a.re, s * a.im}; }
__host__ __device__ inline cfloat operator+(cfloat a, cfloat b) { return {a.re + b.re, a.im + b.im}; }
__host__ __device__ inline cfloat operator-(cfloat a, cfloat b) { return {a.re - b.re, a.im - b.im}; }
__host__ __device__ inline cfloat operator-(cfloat a) { return {-a.re, -a.im}; }
__host__ __device__ inline cfloat operator*(cfloat a, cfloat b) {
  return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
__host__ __device__ inline cfloat operator*(float s, cfloat a) { return {s * a.re, s * a.im}; }

__host__ __device__ inline double conj(double a) { return a; }
__host__ __device__ inline float conj(float a) { return a; }
__host__ __device__ inline cdouble conj(cdouble a) { return {a.re, -a.im}; }
__host__ __device__ inline cfloat conj(cfloat a) { return {a.re, -a.im}; }
__host__ __device__ inline double abs2(double a) { return a * a; }
__host__ __device__ inline float abs2(float a) { return a * a; }
__host__ __device__ inline double abs2(cdouble a) { return a.re * a.re + a.im * a.im; }
__host__ __device__ inline float abs2(cfloat a) { return a.re * a.re + a.im * a.im; }
// a * b with a real scalar
__host__ __device__ inline double rmul(double s, double a) { return s * a; }
__host__ __device__ inline float rmul(float s, float a) { return s * a; }
__host__ __device__ inline cdouble rmul(double s, cdouble a) { return {s * a.re, s * a.im}; }
__host__ __device__ inline cfloat rmul(float s, cfloat a) { return {s * a.re, s * a.im}; }

// acc + a * b and acc - a * b.  Complex FP64: four multiply-adds; acc + (a * b) as written above is
// a product, a multiply-add and an addition per component, six instructions (the compiler keeps
// the order of the sum), which FP64 kernels pay in full (8 x 8 complex FP64 blocks on 32^2 x 128:
// 475 us so, 285 us with four, at 168 M FMA = 268 us of the measured rate).  Four multiply-adds round
// the sum twice per term (40 terms: rms 3.0e-16 of the result against 2.2e-16).  Complex FP32 forms
// the product first: its kernels wait for memory, and a product with the operator, the update of
// a solution and the dense products keep their digits (an inner solve of the Wilson operator stagnates
// at a residual of 3.4e-7, at 4.4e-7 with four multiply-adds; 128^2 estimate 70.5 against 69.2 ms).
__host__ __device__ inline double madd(double c, double a, double b) { return c + a * b; }
__host__ __device__ inline float madd(float c, float a, float b) { return c + a * b; }
__host__ __device__ inline double msub(double c, double a, double b) { return c - a * b; }
__host__ __device__ inline float msub(float c, float a, float b) { return c - a * b; }
__host__ __device__ inline cdouble madd(cdouble c, cdouble a, cdouble b) {
  return {fma(-a.im, b.im, fma(a.re, b.re, c.re)), fma(a.im, b.re, fma(a.re, b.im, c.im))};
}
__host__ __device__ inline cdouble msub(cdouble c, cdouble a, cdouble b) {
  return {fma(a.im, b.im, fma(-a.re, b.re, c.re)), fma(-a.im, b.re, fma(-a.re, b.im, c.im))};
}
__host__ __device__ inline cfloat madd(cfloat c, cfloat a, cfloat b) {
  return {c.re + fmaf(-a.im, b.im, a.re * b.re), c.im + fmaf(a.im, b.re, a.re * b.im)};
}
__host__ __device__ inline cfloat msub(cfloat c, cfloat a, cfloat b) {
  return {c.re - fmaf(-a.im, b.im, a.re * b.re), c.im - fmaf(a.im, b.re, a.re * b.im)};
}
// The same in four multiply-adds for complex FP32 too: for the smoothers, whose result the flexible
// FGMRES takes as it is, so that its rounding does not reach the solution (all kernels with the
// product first: 128^2 Wilson estimate 72.1 ms).
template <class T> __host__ __device__ inline T madd4(T c, T a, T b) { return madd(c, a, b); }
template <class T> __host__ __device__ inline T msub4(T c, T a, T b) { return msub(c, a, b); }
template <> __host__ __device__ inline cfloat madd4(cfloat c, cfloat a, cfloat b) {
  return {fmaf(-a.im, b.im, fmaf(a.re, b.re, c.re)), fmaf(a.im, b.re, fmaf(a.re, b.im, c.im))};
}
template <> __host__ __device__ inline cfloat msub4(cfloat c, cfloat a, cfloat b) {
  return {fmaf(a.im, b.im, fmaf(-a.re, b.re, c.re)), fmaf(-a.im, b.re, fmaf(-a.re, b.im, c.im))};
}

// conversions between precisions of the same field
template <class To, class From> __host__ __device__ inline To cvt(From a);
template <> __host__ __device__ inline double cvt<double, double>(double a) { return a; }
template <> __host__ __device__ inline float cvt<float, float>(float a) { return a; }
template <> __host__ __device__ inline double cvt<double, float>(float a) { return (double)a; }
template <> __host__ __device__ inline float cvt<float, double>(double a) { return (float)a; }
template <> __host__ __device__ inline cdouble cvt<cdouble, cdouble>(cdouble a) { return a; }
template <> __host__ __device__ inline cfloat cvt<cfloat, cfloat>(cfloat a) { return a; }
template <> __host__ __device__ inline cdouble cvt<cdouble, cfloat>(cfloat a) { return {(double)a.re, (double)a.im}; }
template <> __host__ __device__ inline cfloat cvt<cfloat, cdouble>(cdouble a) { return {(float)a.re, (float)a.im}; }
template <> __host__ __device__ inline float cvt<float, cfloat>(cfloat a) { return a.re; }

template <class T> struct dtype_of;
template <> struct dtype_of<double> { static const DType v = F64; };
template <> struct dtype_of<float> { static const DType v = F32; };
template <> struct dtype_of<cdouble> { static const DType v = C64; };
template <> struct dtype_of<cfloat> { static const DType v = C32; };

// run `body` with T bound to the element type of `t`
#define MLMC_DISPATCH(t, T, ...)                                 \
  switch (t) {                                                   \
    case ::mlmc::F64: { typedef double T; __VA_ARGS__; } break;  \
    case ::mlmc::F32: { typedef float T; __VA_ARGS__; } break;   \
    case ::mlmc::C64: { typedef ::mlmc::cdouble T; __VA_ARGS__; } break; \
    case ::mlmc::C32: { typedef ::mlmc::cfloat T; __VA_ARGS__; } break;  \
  }

// ----------------------------------------------------------------- errors
struct cuda_error {
  cudaError_t code;
  std::string where;
};
void check_cuda(cudaError_t e, const char *where);
#define MLMC_CUDA(call) ::mlmc::check_cuda((call), #call)
#define MLMC_LAUNCH_CHECK(name) ::mlmc::check_cuda(cudaGetLastError(), name)

inline unsigned grid_for(size_t work, int block, size_t cap = 152 * 32) {
  size_t g = (work + block - 1) / block;
  if (g < 1) g = 1;
  if (g > cap) g = cap;
  return (unsigned)g;
}

// Grid of a kernel whose blocks stride over `units` work units: `per_sm` blocks per
// SM of the current device (all resident at once when the kernel's resources allow),
// at most `units`, at least 1.
unsigned resident_grid(size_t units, int per_sm);

// Blocks of `kernel` that fit on one SM at once (launch block size, dynamic shared
// memory), at least 1.
template <class F>
int blocks_per_sm(F kernel, int block, size_t smem) {
  int n = 0;
  check_cuda(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, block, smem), "occupancy");
  return n > 0 ? n : 1;
}

// ----------------------------------------------------------------- views
// Nearest-neighbour block stencil on an nx x ny periodic lattice with d dofs
// per site: coef[site][dir][r][c], dir = 0 self, 1 +x, 2 -x, 3 +y, 4 -y.
// Dirichlet boundaries are zero blocks.  Vector blocks are [site][dof][k].
struct StencilView {
  int nx, ny, d;
  DType t;            // element type of coef / dinv
  const void *coef;   // [nsite][5][d][d]
  const void *dinv;   // [nsite][d][d] inverse of the self block (smoother), may be null
  const void *first;  // [nsite][5][d][d] A_{s,dir} D_nb^{-1} on colour 1 (launch_rbgs_first), may be null
  const void *taps9;  // 9-point levels: the operator as [9][nsite], may be null
  const void *ra;     // 9-point levels: R A as [25][coarse sites], offsets -2 .. 2 in x, then in y
  int const_laplace;  // 1: Example 5.1 operator, applied without reading coef
  double diag;        //    its diagonal 4 + shift
  int periodic;       //    0: Dirichlet
  int taps;           // 5: the nearest-neighbour block stencil above; 9: a 9-point scalar
                      //    stencil coef[site][9] (bilinear coarse levels, Dirichlet, d = 1)
};

// Per-aggregate prolongation blocks P[agg][loc*d + a][q] with loc = jj*ax + ii.
struct ProlongView {
  int nx, ny, d;      // fine lattice
  int ax, ay, dc;     // aggregate shape and coarse dofs
  DType t;
  const void *P;
  int bilinear;       // 1: bilinear interpolation from the (nx-1)/2 x (ny-1)/2 grid (no P array)
};

// ----------------------------------------------------------------- launchers
// vector kernels (kernels_vec.cu)
void launch_noise(int kind, uint64_t seed, uint64_t key_hi, uint64_t first_sample, size_t n, int k,
                  DType t, void *out, cudaStream_t s);
void launch_convert(DType to, void *dst, DType from, const void *src, size_t count, cudaStream_t s);
void launch_fill_zero(DType t, void *dst, size_t count, cudaStream_t s);
// blocks x 256 threads, each running 8 FMA (add = 1: addition) chains of `iters` steps (F64 or F32);
// out (blocks x 256 entries) is written only under a condition that never holds
void launch_fma_rate(DType t, int add, void *out, int blocks, int iters, cudaStream_t s);
// `passes` copies a -> b -> a ... of n16 16-byte packs in one launch (bandwidth probe)
void launch_copy16(void *a, void *b, size_t n16, int passes, int blocks, cudaStream_t s);
void launch_fill_one(DType t, void *dst, size_t count, cudaStream_t s);
void launch_sub(DType t, void *out, const void *a, const void *b, size_t count, cudaStream_t s);
// y[i][c] = alpha[c] * x[i][c] (+ y if accumulate)
void launch_scale_cols(DType t, void *y, const void *x, const void *alpha, int alpha_is_inverse_norm,
                       size_t rows, int k, cudaStream_t s);
// out[v][c] = sum_i conj(V_v[i][c]) * w[i][c], v < nvec, FP64 (complex FP64), fixed order
// (kernels_dots.cu).  partials: nparts * nvec * k FP64 (complex FP64) entries, nparts =
// multidot_parts(t, rows, k) <= 304.
void launch_multidot(DType t, const void *V, size_t vstride, int nvec, const void *w, size_t rows,
                     int k, void *partials, int nparts, void *out, cudaStream_t s);
int multidot_parts(DType t, size_t rows, int k);
// w[i][c] = (init ? 0 : w[i][c]) + sign * sum_v V_v[i][c] * h[v][c], h FP64 (complex FP64)
int launch_multiaxpy(DType t, void *w, const void *V, size_t vstride, int nvec, const void *h, double sign,
                     size_t rows, int k, bool init, cudaStream_t s);   // returns its launches

// The fixed-length FGMRES with an unnormalised basis u_0 = b, u_1, ... (V + i * vstride); each
// returns its number of launches where that depends on the length.
// Step j: partial dots of w = A z_j, then the multi-AXPY's coefficients (mid), the multi-AXPY
// itself with the partial norms of u_{j+1} = w; on the last step the solution's weights (tail)
// instead.  partials: multidot_parts * (its + 2) * k, norm: multiaxpy_norm_parts * k FP64
// (complex FP64) entries; n2: its * k; D: its * (m + 1) * k; coef, y: its * k of type t.
int launch_fgmres_dots(DType t, const void *b, const void *V, size_t vstride, int j, int its, const void *w, size_t rows,
                       int k, void *partials, cudaStream_t s);
void launch_fgmres_mid(DType t, const void *partials, const void *norm, int j, int m, size_t rows, int k, double *n2,
                       void *D, void *coef, cudaStream_t s);
void launch_fgmres_tail(DType t, const void *partials, const void *norm, int its, int m, size_t rows, int k,
                        double *n2, const void *D, void *y, cudaStream_t s);
int launch_fgmres_axpy(DType t, void *w, const void *b, const void *V, size_t vstride, int nvec, const void *coef,
                       size_t rows, int k, void *norm, cudaStream_t s);
int launch_fgmres_update(DType t, void *x, const void *Z, size_t vstride, int nvec, const void *y, size_t rows, int k,
                         cudaStream_t s);
int multiaxpy_norm_parts(DType t, size_t rows, int k);

}  // namespace mlmc

namespace mlmc {
// stencil kernels (kernels_stencil.cu)
// mode 0: y = A x;  mode 1: y = b - A x
void launch_stencil(const StencilView &A, const void *x, const void *b, void *y, int k, int mode,
                    cudaStream_t s);
// one red-black block Gauss-Seidel half-sweep over sites of `colour`
void launch_rbgs_half(const StencilView &A, void *x, const void *b, int k, int colour, cudaStream_t s);
// one full red-black sweep (order 0: red then black, 1: black then red).  x_zero = 1
// means x holds zeros on entry (x need not be initialised: the kernels skip it).
void launch_rbgs_sweep(const StencilView &A, void *x, const void *b, int k, int order, int x_zero,
                       cudaStream_t s);
// the first red-black sweep from x = 0 when another follows: sets x on colour 1 only
void launch_rbgs_first(const StencilView &A, void *x, const void *b, int k, cudaStream_t s);
void launch_first_blocks(DType t, const void *coef, const void *dinv, void *first, int nx, int ny, int d,
                         cudaStream_t s);
// rc = P^* r
void launch_restrict(const ProlongView &P, const void *r, void *rc, int k, cudaStream_t s);
// x += P ec
void launch_prolong_add(const ProlongView &P, const void *ec, void *x, int k, cudaStream_t s);
// x += P ec on the sites of one red-black colour only (aggregation levels; all sites otherwise)
void launch_prolong_add_colour(const ProlongView &P, const void *ec, void *x, int k, int colour, cudaStream_t s);
// rc = P^* (b - A x) with the residual taken on the sites of `colour` only (zero on the
// other colour after a red-black Gauss-Seidel sweep that updated it last); aggregation
// levels with d, dc <= 4 and the Example 5.1 fine level
bool residual_restrict_ok(const StencilView &A, const ProlongView &P);
// the levels on which the cycle fuses the two: those, and FP32 levels with dc = 8
bool residual_restrict_fused(const StencilView &A, const ProlongView &P);
void launch_residual_restrict(const StencilView &A, const ProlongView &P, const void *x, const void *b, void *rc,
                              int k, int colour, cudaStream_t s);
// out = base + omega * D^{-1} (rhs - y), D = diagonal entries of the self blocks; base/rhs may be null
// one damped-Jacobi sweep out = x - omega D^-1 A x of the constant-coefficient Laplacian
void launch_laplace_jacobi(const StencilView &A, const void *x, void *out, int k, double omega, cudaStream_t s);
void launch_jacobi_update(const StencilView &A, void *out, const void *base, const void *rhs,
                          const void *y, double omega, int k, cudaStream_t s);
// bilinear hierarchy of Example 5.1 (kernels_bilinear.cu), real data, d = 1
void launch_stencil9(const StencilView &A, const void *x, const void *b, void *y, int k, int mode, cudaStream_t s);
// one 4-colour Gauss-Seidel sweep (order 0: colours 0..3, 1: 3..0); x_zero: x is zeroed first
void launch_gs9_sweep(const StencilView &A, void *x, const void *b, int k, int order, int x_zero, cudaStream_t s);
// small 9-point levels, one launch each: x = `sweeps` sweeps from zero and rc = R (b - A x);
// x += P ec and `sweeps` sweeps in reverse colour order
constexpr size_t CYCLE9_SITES = 48 * 48;         // the largest such level
bool cycle9_ok(const StencilView &A, int k);
void launch_cycle9_down(const StencilView &A, const void *b, void *x, void *rc, int k, int sweeps, cudaStream_t s);
void launch_cycle9_up(const StencilView &A, const void *b, const void *ec, void *x, int k, int sweeps, cudaStream_t s);
// rc = P^T r from the fine (2 nxc + 1) x (2 nyc + 1) grid
void launch_restrict_bilinear(DType t, const void *r, void *rc, int nxc, int nyc, int k, cudaStream_t s);
// x += P ec on the fine nx x ny grid
void launch_prolong_bilinear(DType t, const void *ec, void *x, int nx, int ny, int k, cudaStream_t s);
// setup kernels (kernels_setup.cu)
void launch_block_inverse(DType t, const void *coef, void *dinv, int nsite, int d, int *err,
                          cudaStream_t s);
void launch_mgs(DType t, const void *V, void *P, int nx, int ny, int d, int ax, int ay, int ntv,
                int spin_split, int *err, cudaStream_t s);
void launch_galerkin(const StencilView &fine, const ProlongView &P, void *coarse_coef, cudaStream_t s);
// dense inverse of an n x n matrix (row-major), work = n x 2n elements, scratch of
// gauss_jordan_scratch_bytes(n) bytes; *err = 3 for a singular matrix, MLMC_ERR_TIMEOUT
// when a bounded grid-barrier wait gave up
size_t gauss_jordan_scratch_bytes(int n);
void launch_gauss_jordan(DType t, const void *A, void *Ainv, void *work, int n, int *err, void *scratch,
                         size_t scratch_bytes, cudaStream_t s);
void launch_trace(DType t, const void *A, int n, void *out /* FP64 (complex) */, cudaStream_t s);
// Y = Ainv * B  (n x n times n x k, row-major / [row][k])
// part: scratch of dense_apply_splits(n, k) * n * k elements (or null: no split of j)
void launch_dense_apply(DType t, const void *Ainv, const void *B, void *Y, int n, int k, void *part, cudaStream_t s);
int dense_apply_splits(int n, int k);
// Tensor-core (tcgen05, 3xTF32) variant for FP32 / complex-FP32 data, any n, k >= 1.
// part: dense_apply_tc_part_bytes(t, n, k) bytes of K-slice partials (none needed
// when that is 0); err: device int that receives MLMC_ERR_TIMEOUT if a bounded
// wait gives up.  Pointers 16-byte aligned.  withhold != 0: test mode that
// issues no MMA, so the first bounded wait runs out (about 1 ms).
bool dense_apply_tc_ok(DType t, int n, int k);
size_t dense_apply_tc_part_bytes(DType t, int n, int k);
void launch_dense_apply_tc(DType t, const void *Ainv, const void *B, void *Y, int n, int k, void *part,
                           size_t part_bytes, int *err, cudaStream_t s, int withhold = 0);
}  // namespace mlmc

namespace mlmc {
// per-column Krylov kernels of the restarted FGMRES (kernels_krylov.cu).  `hc` = 1 for complex
// Hessenberg data.  g0[c] holds |r|^2 on entry (from a column dot); sets beta, invnrm and
// active (1 / 0; -1 where the residual norm is not finite: such a column can never converge).
void launch_arnoldi_init(int hc, void *g, double *bnorm, double *invnrm, int *active, int *jdone,
                         int k, double tol, int first, cudaStream_t s);
void launch_arnoldi_step(int hc, void *H, void *cs, void *sn, void *g, int j, int m, int k, int *active,
                         int *jdone, const double *bnorm, double tol, double *invnrm, double *resid, cudaStream_t s);
void launch_trisolve(int hc, const void *H, const void *g, void *y, const int *jdone, int m, int k,
                     cudaStream_t s);
void launch_add_acc(int hc, void *dst, const void *src, int count, cudaStream_t s);
// out[c] = a[c] - b[c] (complex FP64 samples from two column dots)
void launch_sample_combine(int hc, const void *a, const void *b, void *out, int k, cudaStream_t s);
// Welford accumulation of k complex samples into acc = {N, mean.re, mean.im, M2}
void launch_accumulate(const void *samples, int k, double *acc, cudaStream_t s);
// fine block stencils from the operator descriptor
void launch_build_laplace(double *coef, int nx, int ny, double shift, int periodic, cudaStream_t s);
void launch_build_wilson(cdouble *coef, const cdouble *links, int nx, int ny, double mass, cudaStream_t s);
// dense n x n matrix of a block stencil level (row-major)
void launch_stencil_to_dense(const StencilView &A, void *dense, cudaStream_t s);
}  // namespace mlmc

namespace mlmc {
// learned correction (kernels_learned.cu)
void launch_to_channels(DType t, const void *x, float *a, int nsite, int d, int k, cudaStream_t s);
void launch_add_from_channels(DType t, void *x, const float *a, int nsite, int d, int k, cudaStream_t s);
// by_tap: layers with a ReLU add up tap by tap (see k_conv)
void launch_conv_fwd(int ci, int co, const float *in, const float *W, float *out, int nx, int ny, int k,
                     int periodic, cudaStream_t s, bool by_tap = false);
void launch_conv_bwd_data(int ci, int co, const float *gout, const float *W, const float *act, float *gin, int nx,
                          int ny, int k, int periodic, cudaStream_t s);
// the first and last layer reading and writing the vector block itself (real, or complex
// interleaved): out = relu(W x); x = W in, or x += W in
void launch_conv_first(DType t, int ci, const void *x, const float *W, float *out, int nx, int ny, int k, int periodic,
                       cudaStream_t s);
void launch_conv_last(DType t, int co, const float *in, const float *W, void *x, bool add, int nx, int ny, int k,
                      int periodic, cudaStream_t s);
// floats of scratch for the weight gradients' partial sums
size_t conv_weight_scratch();
void launch_conv_bwd_weight(int ci, int co, const float *in, const float *gout, float *partial, float *grad,
                            float scale, int nx, int ny, int k, int periodic, cudaStream_t s);
// tensor-core convolutions (kernels_conv_tc.cu): forward (mirror = 0; W [cout][cin][9]) or
// backward-data (mirror = 1; W [cin][cout][9]), output masked by act > 0 when act is given
bool conv_tc_ok(int nx, int k, int cin, int cout);
void launch_conv_tc(const float *in, const float *W, const float *act, float *out, int nx, int ny, int k, int cin,
                    int cout, int periodic, int mirror, int relu, int *err, cudaStream_t s);
// per-CTA partial weight gradients [conv_wgrad_tc_blocks()][cout][cin][9]; k_weight_reduce adds them
bool conv_wgrad_tc_ok(int k, int cin, int cout);
int conv_wgrad_tc_blocks();
void launch_conv_wgrad_tc(const float *in, const float *gout, float *partial, int nx, int ny, int k, int cin,
                          int cout, int periodic, int *err, cudaStream_t s);
// grad[w] = scale * sum over blocks of partial[block][w], blocks in order
void launch_weight_reduce(const float *partial, int nblocks, int nw, float *grad, float scale, cudaStream_t s);
void launch_adam(float *W, const float *g, float *m, float *v, int n, float lr, int step, cudaStream_t s);
void launch_spin_flip(DType t, void *x, int nsite, int d, int k, cudaStream_t s);
// alpha[c] = scale / |dot[c]| (real part), FP64 per-column factors from a column dot
void launch_col_factor(int hc, const void *dot, double *alpha, double scale, int k, cudaStream_t s);
}  // namespace mlmc
