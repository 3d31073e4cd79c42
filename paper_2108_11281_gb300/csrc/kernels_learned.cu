// Learned correction inside the multigrid cycle: a bias-free 3-layer 3x3
// convolutional network (channels c0 -> 16 -> 16 -> c0, ReLU after the first
// two layers) on the fine lattice, with its training kernels (backward data
// and weight gradients, the loss seed of ||A net(r) - r||^2 / ||r||^2, Adam).
// The paper has no learned component; this is the project's smoother.
//
// Activations are FP32 blocks [site][channel][k] (the k columns innermost, as
// for vectors).  Channel 2a / 2a+1 hold Re / Im of dof a for complex vectors,
// channel a holds dof a for real ones.  Weights are FP32 [c_out][c_in][3][3];
// tap (ty, tx) reads the site (i + tx - 1, j + ty - 1), periodic or zero
// outside a Dirichlet lattice.
#include <type_traits>

#include "mlmc_internal.cuh"

namespace mlmc {

__device__ inline int tap_site(int i, int j, int tx, int ty, int nx, int ny, int periodic) {
  int ii = i + tx - 1, jj = j + ty - 1;
  if (periodic) {
    ii = ii < 0 ? ii + nx : (ii >= nx ? ii - nx : ii);
    jj = jj < 0 ? jj + ny : (jj >= ny ? jj - ny : jj);
    return jj * nx + ii;
  }
  if (ii < 0 || ii >= nx || jj < 0 || jj >= ny) return -1;
  return jj * nx + ii;
}

// ------------------------------------------------------------------ vector <-> channels
template <class T>
__global__ void k_to_channels(const T *x, float *a, int nsite, int d, int k) {
  const int cpd = sizeof(T) == sizeof(double) * 2 || sizeof(T) == sizeof(float) * 2 ? 2 : 1;
  unsigned total = (unsigned)nsite * d * k;
  for (unsigned t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
    unsigned row = t / (unsigned)k;
    int c = (int)(t - row * (unsigned)k);
    int s = (int)(row / (unsigned)d), dof = (int)(row - (unsigned)s * d);
    T v = x[t];
    float* base = a + ((size_t)s * d * cpd) * k + c;
    if (cpd == 2) {
      base[(size_t)(2 * dof) * k] = (float)re(v);
      base[(size_t)(2 * dof + 1) * k] = (float)im(v);
    } else {
      base[(size_t)dof * k] = (float)re(v);
    }
  }
}

// x += from_channels(a)
template <class T>
__global__ void k_add_from_channels(T *x, const float *a, int nsite, int d, int k) {
  const int cpd = sizeof(T) == sizeof(double) * 2 || sizeof(T) == sizeof(float) * 2 ? 2 : 1;
  unsigned total = (unsigned)nsite * d * k;
  for (unsigned t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
    unsigned row = t / (unsigned)k;
    int c = (int)(t - row * (unsigned)k);
    int s = (int)(row / (unsigned)d), dof = (int)(row - (unsigned)s * d);
    const float *base = a + ((size_t)s * d * cpd) * k + c;
    if (cpd == 2) x[t] = x[t] + make<T>(base[(size_t)(2 * dof) * k], base[(size_t)(2 * dof + 1) * k]);
    else x[t] = x[t] + make<T>(base[(size_t)dof * k], 0.0);
  }
}

// ------------------------------------------------------------------ convolutions
// out[s][co][c] = epi(sum_{tap, ci} W[co][ci][tap] in[tap_site(s)][ci][c]).  A thread computes
// PX consecutive sites of a lattice row for one column and at most 8 output channels: with PX = 8 a
// (row, channel) of its inputs is ten loads for three taps, and a 16-byte shared load of weights
// (four clocks of the load unit) serves 32 multiply-adds.  Bound by FP32 arithmetic: the 256^2 x
// 32 network (c0 = 4) takes 14.5 GFLOP, 185 us at the measured 39.2 T FMA/s; 345 us here, 586
// with one site per thread (five load instructions per 16 multiply-adds), 445 with predicates
// and 64-bit address arithmetic on every load, 378 without the packed multiply-adds.  KC is the
// block width where it is one of the usual powers of two, known at compile time so that the
// loads' offsets are immediates (0: any width): the sites between the halo columns are
// contiguous, and only the two halo columns take a wrap or a Dirichlet zero.
// The gradient with respect to the input is the same sum with mirrored taps and exchanged
// channels (mirror = 1, W [CIN][COUT][9]):
// gin[s][ci] = sum_{tap, co} W[co][ci][tap] gout[s - (tap offset)][co].
// A layer may read the complex block itself (XIN: two channels per 8-byte load) and write its
// result there, so that inference needs no layout passes.
// TAPS: the sum runs tap by tap with the channels innermost (eight loads per tap instead of ten
// per three).  The forward pass of a loss gradient takes this order: an activation within rounding
// of zero decides a ReLU's mask by the order of its sum, and one flipped mask changes the gradient
// by up to 1e-4 of its scale, so the order stays what training has always used (16 seeds of 128^2 x
// 32: error against 64 bits as with one site per thread, seed by seed; 581 us per gradient, 531
// with the other order, 2632 with one site per thread).
// a0 += x0 * v, a1 += x1 * v as one packed instruction (each half rounds as fmaf does): half the
// issue slots of two multiply-adds
__device__ __forceinline__ void fma_pair(float &a0, float &a1, float x0, float x1, float v) {
  const float2 r = __ffma2_rn(make_float2(x0, x1), make_float2(v, v), make_float2(a0, a1));
  a0 = r.x;
  a1 = r.y;
}

enum { EPI_NONE = 0, EPI_RELU = 1, EPI_MASK = 2, EPI_STORE_COMPLEX = 3, EPI_ADD_COMPLEX = 4, EPI_ADD = 5 };

template <int CIN, int COUT, int EPI, bool XIN, int KC, int PX, bool TAPS>
__global__ void __launch_bounds__(128, 4) k_conv(const float *__restrict__ in, const float *__restrict__ W, int mirror,
                                                 const float *__restrict__ act, float *__restrict__ out, int nx, int ny,
                                                 int kk, int periodic) {
  constexpr int CS = XIN ? 2 : 1;                              // channels per load
  constexpr int CB = COUT < 8 ? COUT : 8, HALVES = COUT / CB;  // output channels per thread
  const int k = KC ? KC : kk;
  __shared__ __align__(16) float Ws[9 * CIN * COUT];           // [ty][ci][tx][co]
  for (int e = threadIdx.x; e < 9 * CIN * COUT; e += blockDim.x) {
    const int co = e % COUT, tx = e / COUT % 3, ci = e / (COUT * 3) % CIN, ty = e / (COUT * 3 * CIN);
    const int tap = ty * 3 + tx;
    Ws[e] = mirror ? W[(ci * COUT + co) * 9 + 8 - tap] : W[(co * CIN + ci) * 9 + tap];
  }
  __syncthreads();
  const unsigned groups = (nx + PX - 1) / PX, total = groups * ny * k * HALVES;
  for (unsigned t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
    unsigned q = t / (unsigned)k;
    const int c = (int)(t - q * (unsigned)k);
    // neighbouring groups of k threads take the output halves of the same sites (inputs from L1)
    const int cb = (int)(q % HALVES) * CB;
    q /= HALVES;
    const int j = (int)(q / groups);
    // the last group of a row whose length PX does not divide is moved back, and leaves the
    // sites before `first` to the group before it
    const int first = (int)(q - (unsigned)j * groups) * PX;
    const int i0 = max(0, min(first, nx - PX));
    const int n = min(PX, nx);                                 // nx < PX: one short group
    const int il = i0 > 0 ? i0 - 1 : nx - 1, ir = i0 + n < nx ? i0 + n : 0;
    const bool onl = i0 > 0 || periodic, onr = i0 + n < nx || periodic;
    float acc[PX][CB];
#pragma unroll
    for (int p = 0; p < PX; ++p)
#pragma unroll
      for (int co = 0; co < CB; ++co) acc[p][co] = 0.f;
    auto taps = [&](const float *w, const float *v) {
#pragma unroll
      for (int tx = 0; tx < 3; ++tx) {
        float wv[CB];
        if constexpr (CB % 4 == 0) {
#pragma unroll
          for (int co = 0; co < CB; co += 4) {
            const float4 w4 = *reinterpret_cast<const float4 *>(w + tx * COUT + co);
            wv[co] = w4.x; wv[co + 1] = w4.y; wv[co + 2] = w4.z; wv[co + 3] = w4.w;
          }
#pragma unroll
          for (int p = 0; p < PX; ++p)
#pragma unroll
            for (int co = 0; co < CB; co += 2) fma_pair(acc[p][co], acc[p][co + 1], wv[co], wv[co + 1], v[p + tx]);
        } else {
#pragma unroll
          for (int co = 0; co < CB; ++co) wv[co] = w[tx * COUT + co];
#pragma unroll
          for (int p = 0; p < PX; ++p)
#pragma unroll
            for (int co = 0; co < CB; ++co) acc[p][co] = fmaf(wv[co], v[p + tx], acc[p][co]);
        }
      }
    };
#pragma unroll 1
    for (int ty = 0; ty < 3; ++ty) {
      int jj = j + ty - 1;
      if (periodic) jj = jj < 0 ? jj + ny : jj >= ny ? jj - ny : jj;
      if (jj < 0 || jj >= ny) continue;
      const size_t row = (size_t)jj * nx;
      const float *mid = in + (row + i0) * CIN * k + CS * c;
      const float *left = in + (row + il) * CIN * k + CS * c, *right = in + (row + ir) * CIN * k + CS * c;
      const float *w = Ws + ty * CIN * 3 * COUT + cb;
      if constexpr (TAPS) {
#pragma unroll
        for (int tx = 0; tx < 3; ++tx) {
#pragma unroll 2
          for (int ci = 0; ci < CIN; ++ci) {
            const int o = ci * k;
            float v[PX], wv[CB];
#pragma unroll
            for (int u = 0; u < PX; ++u) {
              const int at = u + tx - 1;                       // site i0 + at; n is its right halo
              const float *src = at < 0 ? left : at < n ? mid + (size_t)at * CIN * k : right;
              const bool ok = at < 0 ? onl : at < n || (at == n && onr);
              v[u] = ok ? src[o] : 0.f;
            }
#pragma unroll
            for (int co = 0; co < CB; co += 4) {
              const float4 w4 = *reinterpret_cast<const float4 *>(w + (ci * 3 + tx) * COUT + co);
              wv[co] = w4.x; wv[co + 1] = w4.y; wv[co + 2] = w4.z; wv[co + 3] = w4.w;
            }
#pragma unroll
            for (int p = 0; p < PX; ++p)
#pragma unroll
              for (int co = 0; co < CB; co += 2) fma_pair(acc[p][co], acc[p][co + 1], wv[co], wv[co + 1], v[p]);
          }
        }
        continue;
      }
#pragma unroll 2
      for (int ci = 0; ci < CIN; ci += CS) {
        float v[CS][PX + 2];
        auto load = [&](int u, const float *src, bool ok) {
          if constexpr (XIN) {
            const float2 x = ok ? *reinterpret_cast<const float2 *>(src) : make_float2(0.f, 0.f);
            v[0][u] = x.x;
            v[1][u] = x.y;
          } else {
            v[0][u] = ok ? *src : 0.f;
          }
        };
        load(0, left, onl);
        if (n == PX) {
#pragma unroll
          for (int u = 0; u < PX; ++u) load(u + 1, mid + u * CIN * k, true);
          load(PX + 1, right, onr);
        } else {
          // a lattice narrower than the group: its right halo comes after n sites
#pragma unroll
          for (int u = 0; u <= PX; ++u)
            load(u + 1, u < n ? mid + u * CIN * k : right, u < n || (u == n && onr));
        }
#pragma unroll
        for (int z = 0; z < CS; ++z) taps(w + (ci + z) * 3 * COUT, v[z]);
        left += CS * k;
        mid += CS * k;
        right += CS * k;
      }
    }
#pragma unroll
    for (int p = 0; p < PX; ++p) {
      if (p >= n) break;
      if (i0 + p < first) continue;
      const size_t o = (((size_t)j * nx + i0 + p) * COUT + cb) * k;
      if constexpr (EPI == EPI_STORE_COMPLEX || EPI == EPI_ADD_COMPLEX) {
#pragma unroll
        for (int co = 0; co + 1 < CB; co += 2) {
          float2 *dst = reinterpret_cast<float2 *>(out + o + (size_t)co * k) + c;
          float2 v = make_float2(acc[p][co], acc[p][co + 1]);
          if (EPI == EPI_ADD_COMPLEX) {
            const float2 x = *dst;
            v.x += x.x;
            v.y += x.y;
          }
          *dst = v;
        }
      } else {
#pragma unroll
        for (int co = 0; co < CB; ++co) {
          float *dst = out + o + (size_t)co * k + c;
          float v = acc[p][co];
          if (EPI == EPI_RELU) v = fmaxf(v, 0.f);
          if (EPI == EPI_MASK) v = act[o + (size_t)co * k + c] > 0.f ? v : v * 0.f;
          if (EPI == EPI_ADD) v += *dst;
          *dst = v;
        }
      }
    }
  }
}

// ------------------------------------------------------------------ backward: weights
// partial[part][co][ci][tap] = sum over the part's (site, column) pairs of
// gout[s][co][c] * in[tap_site(s)][ci][c].  Lanes are columns (several lattice rows when k < 32);
// a warp keeps one input channel's nine taps times COG output channels in registers (72 sums)
// and walks lattice rows with a 3 x 3 window, so a site costs COG + 3 coalesced loads for
// 9 COG multiply-adds; the warps of a block walk the same sites for the other channels and
// share the loads in L1.  The loads run ahead of the products (the window by two sites, the
// gradients by one: more spills).  16 -> 16 channels on 128^2 x 32 (2.4 GFLOP, 31 us at the
// measured rate): about 120 us against 1151 us with the pairs staged through shared memory and
// two shared loads per multiply-add.  The lanes meet once at the end (fixed shuffle tree), the
// parts in k_weight_reduce.
constexpr int WG_THREADS = 512, WG_SEG = 16, WG_BLOCKS = 152;

template <int CI, int CO> struct wg {
  static constexpr int COG = CO < 8 ? CO : 8;
  static constexpr int COMBOS = CI * (CO / COG);                     // (input channel, output group) pairs
  static constexpr int CPB = COMBOS < 16 ? COMBOS : 16;              // of one block's 16 warps
  static constexpr int SLICES = 16 / CPB, GY = COMBOS / CPB;
  static constexpr int PARTS = WG_BLOCKS / GY * SLICES;
};

template <int CI, int CO, int KC>
__global__ void __launch_bounds__(WG_THREADS, 1) k_conv_bwd_weight(const float *__restrict__ in,
                                                                   const float *__restrict__ gout,
                                                                   float *__restrict__ partial, int nx, int ny, int kk,
                                                                   int periodic) {
  typedef wg<CI, CO> G;
  constexpr int COG = G::COG;
  const int k = KC ? KC : kk;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int combo = blockIdx.y * G::CPB + warp % G::CPB, ci = combo % CI, co0 = combo / CI * COG;
  const int part = blockIdx.x * G::SLICES + warp / G::CPB;
  const int rpu = k >= 32 ? 1 : 32 / k;                       // lattice rows per unit
  const int chunks = (k + 31) / 32, segs = (nx + WG_SEG - 1) / WG_SEG;
  const int units = (ny + rpu - 1) / rpu * chunks * segs;
  float acc[COG][9];
#pragma unroll
  for (int q = 0; q < COG; ++q)
#pragma unroll
    for (int p = 0; p < 9; ++p) acc[q][p] = 0.f;
  const float *X = in + (size_t)ci * k, *Gp = gout + (size_t)co0 * k;
  for (int u = part; u < units; u += G::PARTS) {
    const int seg = u % segs, v = u / segs;
    const int c = k >= 32 ? v % chunks * 32 + lane : lane % k;
    const int j = k >= 32 ? v / chunks : v * rpu + lane / k;
    const bool live = c < k && j < ny && (k >= 32 || lane / k < rpu);
    const int i0 = seg * WG_SEG, i1 = min(i0 + WG_SEG, nx);
    // the window's rows: which exist (an idle lane has none) and where they start
    const float *row[3];
    bool on[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      int jj = j + r - 1;
      if (periodic) jj = jj < 0 ? jj + ny : jj >= ny ? jj - ny : jj;
      on[r] = live && jj >= 0 && jj < ny;
      row[r] = X + (on[r] ? (size_t)jj * nx * CI * k + c : 0);
    }
    const float *g = Gp + (live ? ((size_t)j * nx + i0) * CO * k + c : 0);
    auto column = [&](int i, float w[3]) {                   // window column i, -1 <= i <= nx + 1
      const bool in_row = (unsigned)i < (unsigned)nx;
      const int ii = in_row ? i : i < 0 ? i + nx : i - nx;
      const bool ok = in_row || periodic;
      const size_t o = (size_t)(unsigned)ii * (unsigned)(CI * k);
#pragma unroll
      for (int r = 0; r < 3; ++r) w[r] = ok && on[r] && ii < nx ? row[r][o] : 0.f;
    };
    auto grads = [&](float w[COG], bool ok) {                // the next site's gradients
#pragma unroll
      for (int q = 0; q < COG; ++q) w[q] = live && ok ? g[q * k] : 0.f;
      g += CO * k;
    };
    float a[3], b[3], d[3], e[3], g0[COG];
    column(i0 - 1, a);
    column(i0, b);
    column(i0 + 1, d);
    column(min(i0 + 2, nx + 1), e);
    grads(g0, true);
#pragma unroll 4
    for (int i = i0; i < i1; ++i) {
      float en[3], gn[COG];
      column(min(i + 3, nx + 1), en);                        // used two sites on, if at all
      grads(gn, i + 1 < i1);
      auto taps3 = [&](int r, int tx, float x) {
        if constexpr (COG % 2 == 0) {
#pragma unroll
          for (int q = 0; q < COG; q += 2)
            fma_pair(acc[q][r * 3 + tx], acc[q + 1][r * 3 + tx], g0[q], g0[q + 1], x);
        } else {
#pragma unroll
          for (int q = 0; q < COG; ++q) acc[q][r * 3 + tx] = fmaf(g0[q], x, acc[q][r * 3 + tx]);
        }
      };
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        taps3(r, 0, a[r]);
        taps3(r, 1, b[r]);
        taps3(r, 2, d[r]);
      }
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        a[r] = b[r];
        b[r] = d[r];
        d[r] = e[r];
        e[r] = en[r];
      }
#pragma unroll
      for (int q = 0; q < COG; ++q) g0[q] = gn[q];
    }
  }
  float *dst = partial + (size_t)part * CO * CI * 9;
#pragma unroll
  for (int q = 0; q < COG; ++q)
#pragma unroll
    for (int p = 0; p < 9; ++p) {
      float v = acc[q][p];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == (q * 9 + p) % 32) dst[((size_t)(co0 + q) * CI + ci) * 9 + p] = v;
    }
}

// grad[w] = scale * sum over parts of partial[part][w] in FP64: a block takes eight weights (one
// sector per part), 32 threads each adding every 32nd part (up to 1216 parts of a narrow layer; with 32
// weights per block their FP64 additions would take one SM 12 us), met in fixed order.
__global__ void __launch_bounds__(256) k_weight_reduce(const float *partial, int nparts, int nw, float *grad,
                                                       float scale) {
  __shared__ double red[32][8];
  const int lane = threadIdx.x & 7, sl = threadIdx.x >> 3, w = blockIdx.x * 8 + lane;
  double a = 0.0;
  if (w < nw) {
#pragma unroll 4
    for (int p = sl; p < nparts; p += 32) a += (double)partial[(size_t)p * nw + w];
  }
  red[sl][lane] = a;
  __syncthreads();
  if (sl < 4) {
    for (int q = sl + 4; q < 32; q += 4) a += red[q][lane];
    red[sl][lane] = a;               // read by this thread alone in this step
  }
  __syncthreads();
  if (sl == 0 && w < nw) grad[w] = (float)(((a + red[1][lane]) + (red[2][lane] + red[3][lane])) * scale);
}

// ------------------------------------------------------------------ Adam
__global__ void k_adam(float *W, const float *g, float *m, float *v, int n, float lr, float b1, float b2, float eps,
                       float c1, float c2) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float mi = b1 * m[i] + (1.f - b1) * g[i];
  float vi = b2 * v[i] + (1.f - b2) * g[i] * g[i];
  m[i] = mi;
  v[i] = vi;
  W[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// ------------------------------------------------------------------ launchers
static unsigned cgrid(unsigned total) {
  unsigned g = (total + 255) / 256;
  return g < 152 * 16 ? (g ? g : 1) : 152 * 16;
}

void launch_to_channels(DType t, const void *x, float *a, int nsite, int d, int k, cudaStream_t s) {
  unsigned g = cgrid((unsigned)nsite * d * k);
  MLMC_DISPATCH(t, T, k_to_channels<T><<<g, 256, 0, s>>>((const T *)x, a, nsite, d, k));
  MLMC_LAUNCH_CHECK("k_to_channels");
}

void launch_add_from_channels(DType t, void *x, const float *a, int nsite, int d, int k, cudaStream_t s) {
  unsigned g = cgrid((unsigned)nsite * d * k);
  MLMC_DISPATCH(t, T, k_add_from_channels<T><<<g, 256, 0, s>>>((T *)x, a, nsite, d, k));
  MLMC_LAUNCH_CHECK("k_add_from_channels");
}

// The usual block widths are compile-time constants of the kernels, any other is not (network forward
// with k = 32 at compile time and at run time: 256^2 340 / 391 us, 128^2 114 / 128; k = 16 on 256^2
// 191 / 217, k = 64 on 128^2 190 / 214; loss gradients 1.13 - 1.19 times as long).
template <class F>
static void by_width(int k, F f) {
  switch (k) {
    case 16: f(std::integral_constant<int, 16>()); break;
    case 32: f(std::integral_constant<int, 32>()); break;
    case 64: f(std::integral_constant<int, 64>()); break;
    default: f(std::integral_constant<int, 0>()); break;
  }
}

template <int CIN, int COUT, int EPI, bool XIN, bool TAPS = false>
static void conv_go(const float *in, const float *W, int mirror, const float *act, float *out, int nx, int ny, int k,
                    int periodic, cudaStream_t s) {
  auto go = [&](auto px, auto kc) {
    constexpr int PX = decltype(px)::value;
    const size_t threads = (size_t)((nx + PX - 1) / PX) * ny * k * (COUT > 8 ? COUT / 8 : 1);
    k_conv<CIN, COUT, EPI, XIN, decltype(kc)::value, PX, TAPS><<<resident_grid((threads + 127) / 128, 4), 128, 0, s>>>(
        in, W, mirror, act, out, nx, ny, k, periodic);
  };
  // Sites per thread: eight need the fewest loads, but below some 768 (site, column) pairs per SM
  // they leave fewer than six warps per SM, each a long serial chain; four or two then give
  // more, shorter ones (any block width: the offsets' arithmetic hides in the latency).  Network
  // forward with 8 / 4 / 2 sites: 64^2 x 8 50 / 42.8 / 41.0 us, 96^2 x 8 51 / 46.3 / 47.2, 64^2 x 24
  // 61 / 53.5 / 56.4, 64^2 x 32 56.6 / 59.1 / 64.9, 128^2 x 8 57.1 / 56.9 / 62.8.
  const size_t pairs = (size_t)nx * ny * k;
  if (pairs < (size_t)152 * 384) go(std::integral_constant<int, 2>(), std::integral_constant<int, 0>());
  else if (pairs < (size_t)152 * 768) go(std::integral_constant<int, 4>(), std::integral_constant<int, 0>());
  else by_width(k, [&](auto kc) { go(std::integral_constant<int, 8>(), kc); });
  MLMC_LAUNCH_CHECK("k_conv");
}

// Layers in channel layout: c0 -> 16 and 16 -> 16, both with a ReLU; c0 = 1 (real, one dof per site) or
// 4 (two complex ones).
void launch_conv_fwd(int ci, int co, const float *in, const float *W, float *out, int nx, int ny, int k, int periodic,
                     cudaStream_t s, bool by_tap) {
#define MLMC_TAPS(A) \
  if (by_tap && ci == A && co == 16) \
    return conv_go<A, 16, EPI_RELU, false, true>(in, W, 0, nullptr, out, nx, ny, k, periodic, s);
  MLMC_TAPS(1) MLMC_TAPS(4) MLMC_TAPS(16)
#undef MLMC_TAPS
#define MLMC_FWD(A) \
  if (ci == A && co == 16) return conv_go<A, 16, EPI_RELU, false>(in, W, 0, nullptr, out, nx, ny, k, periodic, s);
  MLMC_FWD(1) MLMC_FWD(4) MLMC_FWD(16)
#undef MLMC_FWD
  throw cuda_error{cudaErrorInvalidValue, "conv: unsupported channel counts"};
}

void launch_conv_first(DType t, int ci, const void *x, const float *W, float *out, int nx, int ny, int k, int periodic,
                       cudaStream_t s) {
  const float *in = (const float *)x;
  if (t == C32 && ci == 4) conv_go<4, 16, EPI_RELU, true>(in, W, 0, nullptr, out, nx, ny, k, periodic, s);
  else if (t == F32) launch_conv_fwd(ci, 16, in, W, out, nx, ny, k, periodic, s);
  else throw cuda_error{cudaErrorInvalidValue, "conv: unsupported block"};
}

void launch_conv_last(DType t, int co, const float *in, const float *W, void *x, bool add, int nx, int ny, int k,
                      int periodic, cudaStream_t s) {
  float *out = (float *)x;
#define MLMC_LAST(TT, B, ADD, E) \
  if (t == TT && co == B && add == ADD) return conv_go<16, B, E, false>(in, W, 0, nullptr, out, nx, ny, k, periodic, s);
  MLMC_LAST(C32, 4, true, EPI_ADD_COMPLEX) MLMC_LAST(C32, 4, false, EPI_STORE_COMPLEX)
  MLMC_LAST(F32, 1, true, EPI_ADD) MLMC_LAST(F32, 1, false, EPI_NONE)
#undef MLMC_LAST
  throw cuda_error{cudaErrorInvalidValue, "conv: unsupported block"};
}

// gradient wrt the input of a layer 16 -> co, masked by act > 0
void launch_conv_bwd_data(int ci, int co, const float *gout, const float *W, const float *act, float *gin, int nx,
                          int ny, int k, int periodic, cudaStream_t s) {
#define MLMC_BWD(B) \
  if (ci == 16 && co == B) return conv_go<B, 16, EPI_MASK, false>(gout, W, 1, act, gin, nx, ny, k, periodic, s);
  MLMC_BWD(1) MLMC_BWD(4) MLMC_BWD(16)
#undef MLMC_BWD
  throw cuda_error{cudaErrorInvalidValue, "conv: unsupported channel counts"};
}

size_t conv_weight_scratch() {
  // floats of partial sums of the widest layer in either family of kernels
  return (size_t)304 * 16 * 16 * 9;
}

void launch_conv_bwd_weight(int ci, int co, const float *in, const float *gout, float *partial, float *grad,
                            float scale, int nx, int ny, int k, int periodic, cudaStream_t s) {
#define MLMC_BWW(A, B)                                                                                        \
  if (ci == A && co == B) {                                                                                   \
    static_assert((size_t)wg<A, B>::PARTS * A * B * 9 <= (size_t)304 * 16 * 16 * 9, "partial sums");          \
    by_width(k, [&](auto kc) {                                                                                \
      k_conv_bwd_weight<A, B, decltype(kc)::value>                                                            \
          <<<dim3(WG_BLOCKS / wg<A, B>::GY, wg<A, B>::GY), WG_THREADS, 0, s>>>(in, gout, partial, nx, ny, k, periodic); \
    });                                                                                                       \
    MLMC_LAUNCH_CHECK("k_conv_bwd_weight");                                                                   \
    launch_weight_reduce(partial, wg<A, B>::PARTS, A * B * 9, grad, scale, s);                                \
    return;                                                                                                   \
  }
  MLMC_BWW(1, 16) MLMC_BWW(4, 16) MLMC_BWW(16, 16) MLMC_BWW(16, 1) MLMC_BWW(16, 4)
#undef MLMC_BWW
  throw cuda_error{cudaErrorInvalidValue, "conv: unsupported channel counts"};
}

void launch_weight_reduce(const float *partial, int nparts, int nw, float *grad, float scale, cudaStream_t s) {
  k_weight_reduce<<<(nw + 7) / 8, 256, 0, s>>>(partial, nparts, nw, grad, scale);
  MLMC_LAUNCH_CHECK("k_weight_reduce");
}

void launch_adam(float *W, const float *g, float *m, float *v, int n, float lr, int step, cudaStream_t s) {
  const float b1 = 0.9f, b2 = 0.999f;
  float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
  k_adam<<<(n + 255) / 256, 256, 0, s>>>(W, g, m, v, n, lr, b1, b2, 1e-8f, c1, c2);
  MLMC_LAUNCH_CHECK("k_adam");
}

// J v: negate the second half of each site's dofs (spin parity of Example 5.3)
template <class T>
__global__ void k_spin_flip(T *x, int nsite, int d, int k) {
  unsigned total = (unsigned)nsite * d * k;
  for (unsigned t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
    unsigned row = t / (unsigned)k;
    int dof = (int)(row % (unsigned)d);
    if (dof >= d / 2) x[t] = -x[t];
  }
}

void launch_spin_flip(DType t, void *x, int nsite, int d, int k, cudaStream_t s) {
  unsigned g = cgrid((unsigned)nsite * d * k);
  MLMC_DISPATCH(t, T, k_spin_flip<T><<<g, 256, 0, s>>>((T *)x, nsite, d, k));
  MLMC_LAUNCH_CHECK("k_spin_flip");
}

}  // namespace mlmc
