// Learned per-patch threshold (the paper uses one uniform constant c,
// Sec. 2.2; the per-patch choice is this library's addition): features and
// labels of patches, a small MLP (in -> 64 -> 64 -> 1, GELU) trained with
// these kernels, and its inference into the per-patch eps of a simulation.
//
//  * features: detail nodes grouped by (l, S), l = the largest per-axis
//    class of the node, S = the axes of that class (x, y, both); per group,
//    over all fields: log10(mean d^2 + 1e-30) and log10(max |d| + 1e-30) of
//    the forward-transformed patch, groups ordered l = 1..L then S = x, y,
//    xy -> 6L inputs.
//  * label: log10 of the largest eps = 10^(-7 + k/8), k = 0..40, whose
//    thresholding (constant rule, no quantisation) changes the patch by at
//    most delta * ||patch||_2 after the inverse transform, refined by four
//    bisections in log eps towards the next grid value (steps under 2%);
//    -7 when no eps of the grid passes, -2 when all do.
// Reductions are in a fixed order, so repeated runs give the same bits.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <type_traits>
#include <vector>

#include "../../include/wcsim.h"
#include "common.cuh"

namespace {

constexpr int MLP_NH = 64;
constexpr int MLP_MAXIN = 64;
constexpr int EPS_N = 41;
__constant__ double c_eps_grid[EPS_N];  // 10^(-7 + k/8), filled on the host

__host__ __device__ inline int nparam(int nin) { return MLP_NH * nin + MLP_NH + MLP_NH * MLP_NH + MLP_NH + MLP_NH + 1; }

// ------------------------------------------------ in-smem lifting (FP64)
template <typename T> __device__ void lift_line_smem(T* u, int stride, int P, int L, int wavelet, bool inverse) {
  auto at = [&](int k, int st) -> T& { return u[k * st * stride]; };
  if (!inverse) {
    for (int lev = 1; lev <= L; ++lev) {
      const int st = 1 << (lev - 1), K = (P / st) / 2;
      if (wavelet == WCS_BL53) {
        for (int k = 0; k < K; ++k) at(2 * k + 1, st) = wcs::fma_rn(T(-0.5), at(2 * k, st) + at(2 * k + 2, st), at(2 * k + 1, st));
        for (int k = 1; k < K; ++k) {
          const T e = wcs::fma_rn(wcs::bl53_alpha<T>(k - 1, K), at(2 * k - 1, st), at(2 * k, st));
          at(2 * k, st) = wcs::fma_rn(wcs::bl53_alpha<T>(k, K), at(2 * k + 1, st), e);
        }
      } else {
        for (int k = 0; k < K; ++k) {
          const T a = at(2 * k, st), b = at(2 * k + 1, st), d = b - a;
          at(2 * k, st) = wcs::fma_rn(T(0.5), d, a);
          at(2 * k + 1, st) = d;
        }
      }
    }
  } else {
    for (int lev = L; lev >= 1; --lev) {
      const int st = 1 << (lev - 1), K = (P / st) / 2;
      if (wavelet == WCS_BL53) {
        for (int k = 1; k < K; ++k) {
          const T e = wcs::fma_rn(-wcs::bl53_alpha<T>(k - 1, K), at(2 * k - 1, st), at(2 * k, st));
          at(2 * k, st) = wcs::fma_rn(-wcs::bl53_alpha<T>(k, K), at(2 * k + 1, st), e);
        }
        for (int k = 0; k < K; ++k) at(2 * k + 1, st) = wcs::fma_rn(T(0.5), at(2 * k, st) + at(2 * k + 2, st), at(2 * k + 1, st));
      } else {
        for (int k = 0; k < K; ++k) {
          const T s = at(2 * k, st), d = at(2 * k + 1, st);
          const T a = wcs::fma_rn(T(-0.5), d, s);
          at(2 * k, st) = a;
          at(2 * k + 1, st) = a + d;
        }
      }
    }
  }
}

__device__ inline int cls(int k, int L) {
  if ((k & ((1 << L) - 1)) == 0) return 0;
  return __ffs(k);
}
// Feature group of node (kx, ky): -1 for a coarse node, else 3 (l - 1) + S - 1.
__device__ inline int group_of(int kx, int ky, int L) {
  const int cx = cls(kx, L), cy = cls(ky, L), l = cx > cy ? cx : cy;
  if (l == 0) return -1;
  return 3 * (l - 1) + (cx == l ? 1 : 0) + (cy == l ? 2 : 0) - 1;
}

// Block sum of a double in a fixed order (power-of-two tree over threads).
__device__ double block_sum(double v, double* red) {
  const int t = threadIdx.x;
  red[t] = v;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (t < o) red[t] = red[t] + red[t + o];
    __syncthreads();
  }
  const double r = red[0];
  __syncthreads();
  return r;
}
__device__ double block_max(double v, double* red) {
  const int t = threadIdx.x;
  red[t] = v;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (t < o) red[t] = red[t] > red[t + o] ? red[t] : red[t + o];
    __syncthreads();
  }
  const double r = red[0];
  __syncthreads();
  return r;
}

// Squared L2 error, summed over all fields, of thresholding patch (px, py)
// at eps: per field load, forward, threshold, inverse, compare.  Every
// thread returns the same value.
__device__ double patch_err2(const float* __restrict__ dense, int F, int G0, int G1, int px, int py, int P, int L,
                             int wavelet, double eps, double* u, double* c, double* red) {
  const int E = wavelet == WCS_BL53 ? P + 1 : P, n = E * E, tid = threadIdx.x;
  double err2 = 0;
  for (int f = 0; f < F; ++f) {
    for (int i = tid; i < n; i += blockDim.x) {
      const int y = i / E, x = i - y * E;
      const int gx = (px * P + x) % G0, gy = (py * P + y) % G1;
      u[i] = double(dense[(size_t(f) * G1 + gy) * G0 + gx]);
      c[i] = u[i];
    }
    __syncthreads();
    for (int y = tid; y < E; y += blockDim.x) lift_line_smem<double>(c + y * E, 1, P, L, wavelet, false);
    __syncthreads();
    for (int x = tid; x < E; x += blockDim.x) lift_line_smem<double>(c + x, E, P, L, wavelet, false);
    __syncthreads();
    for (int i = tid; i < n; i += blockDim.x) {
      const int y = i / E, x = i - y * E;
      if (group_of(x, y, L) >= 0 && !(fabs(c[i]) >= eps)) c[i] = 0.0;
    }
    __syncthreads();
    for (int x = tid; x < E; x += blockDim.x) lift_line_smem<double>(c + x, E, P, L, wavelet, true);
    __syncthreads();
    for (int y = tid; y < E; y += blockDim.x) lift_line_smem<double>(c + y * E, 1, P, L, wavelet, true);
    __syncthreads();
    double my = 0;
    for (int i = tid; i < n; i += blockDim.x) my += (c[i] - u[i]) * (c[i] - u[i]);
    err2 += block_sum(my, red);
  }
  return err2;
}

// One CTA per patch of a dense FP32 state [F][G1][G0] (periodic BL5/3 or
// Haar grids), 256 threads, FP64 arithmetic.
__global__ void __launch_bounds__(256) features_labels(const float* __restrict__ dense, int F, int G0, int G1, int npx,
                                                        int P, int L, int wavelet, double delta, float* feat,
                                                        float* label) {
  extern __shared__ double sm[];
  const int E = wavelet == WCS_BL53 ? P + 1 : P;
  const int n = E * E;
  double* u = sm;          // original nodes of one field
  double* c = u + n;       // its coefficients
  double* t = c + n;       // a trial
  double* red = t + n;     // 256 doubles
  const int pid = blockIdx.x, px = pid % npx, py = pid / npx;
  const int tid = threadIdx.x;
  const int G = 3 * L;
  double e2[24], mx[24], err2[EPS_N];
  for (int g = 0; g < 24; ++g) { e2[g] = 0; mx[g] = 0; }
  for (int k = 0; k < EPS_N; ++k) err2[k] = 0;
  double norm2 = 0;
  for (int f = 0; f < F; ++f) {
    for (int i = tid; i < n; i += blockDim.x) {
      const int y = i / E, x = i - y * E;
      const int gx = (px * P + x) % G0, gy = (py * P + y) % G1;
      const double v = double(dense[(size_t(f) * G1 + gy) * G0 + gx]);
      u[i] = v;
      c[i] = v;
    }
    __syncthreads();
    for (int y = tid; y < E; y += blockDim.x) lift_line_smem<double>(c + y * E, 1, P, L, wavelet, false);
    __syncthreads();
    for (int x = tid; x < E; x += blockDim.x) lift_line_smem<double>(c + x, E, P, L, wavelet, false);
    __syncthreads();
    double my_n2 = 0, my_e2[24], my_mx[24];
    for (int g = 0; g < 24; ++g) { my_e2[g] = 0; my_mx[g] = 0; }
    for (int i = tid; i < n; i += blockDim.x) {
      const int y = i / E, x = i - y * E;
      my_n2 += u[i] * u[i];
      const int g = group_of(x, y, L);
      if (g >= 0) {
        my_e2[g] += c[i] * c[i];
        my_mx[g] = fmax(my_mx[g], fabs(c[i]));
      }
    }
    norm2 += block_sum(my_n2, red);
    for (int g = 0; g < G; ++g) {
      e2[g] += block_sum(my_e2[g], red);
      mx[g] = fmax(mx[g], block_max(my_mx[g], red));
    }
    for (int k = 0; k < EPS_N; ++k) {
      const double eps = c_eps_grid[k];
      for (int i = tid; i < n; i += blockDim.x) {
        const int y = i / E, x = i - y * E;
        const double v = c[i];
        t[i] = (group_of(x, y, L) >= 0 && !(fabs(v) >= eps)) ? 0.0 : v;
      }
      __syncthreads();
      for (int x = tid; x < E; x += blockDim.x) lift_line_smem<double>(t + x, E, P, L, wavelet, true);
      __syncthreads();
      for (int y = tid; y < E; y += blockDim.x) lift_line_smem<double>(t + y * E, 1, P, L, wavelet, true);
      __syncthreads();
      double my = 0;
      for (int i = tid; i < n; i += blockDim.x) my += (t[i] - u[i]) * (t[i] - u[i]);
      err2[k] += block_sum(my, red);
    }
  }
  if (tid == 0) {
    for (int g = 0; g < G; ++g) {
      long long cnt = 0;
      for (int y = 0; y < E; ++y)
        for (int x = 0; x < E; ++x) cnt += group_of(x, y, L) == g;
      feat[size_t(pid) * 2 * G + 2 * g] = float(log10(e2[g] / double(cnt * F) + 1e-30));
      feat[size_t(pid) * 2 * G + 2 * g + 1] = float(log10(mx[g] + 1e-30));
    }
  }
  const double bound = delta * sqrt(norm2);
  int best = -1;
  for (int k = 0; k < EPS_N; ++k)
    if (sqrt(err2[k]) <= bound) best = k;
  double lab;
  if (best < 0) {
    lab = -7.0;
  } else if (best == EPS_N - 1) {
    lab = -2.0;
  } else {
    double lo = c_eps_grid[best], hi = c_eps_grid[best + 1];
    for (int it = 0; it < 4; ++it) {
      const double mid = sqrt(lo * hi);
      if (sqrt(patch_err2(dense, F, G0, G1, px, py, P, L, wavelet, mid, u, c, red)) <= bound) lo = mid;
      else hi = mid;
    }
    lab = log10(lo);
  }
  if (tid == 0) label[pid] = float(lab);
}

// Features and labels of BL5/3 patches of P cells and L levels with their
// lines in registers, for the sizes the step kernels use (others, and Haar:
// features_labels above).  One CTA of 256 threads per patch.
//
// What bounds it is FP64: an SM does two FP64 operations per cycle, so the
// forward transform of nine 65^2 fields alone takes 87 us.  The label needs
// the error of many thresholds, and takes it from FP32 where that decides:
//  - the fields' coefficients stay in shared memory rounded to FP32; a node
//    is dropped at eps iff |c| < eps, and rounding is monotonic, so the FP32
//    comparison is the FP64 one unless both round to the same number;
//  - the lifting is linear, so the error is the inverse transform of the
//    dropped coefficients c alone, however small it is beside the patch's
//    norm.  Every lifting step rounds twice per node that it changes; with the
//    2-norms of the steps before (rows of those nodes) and behind (columns of
//    those nodes) it, all roundings in FP32 together, c's own among them, add
//    up to at most ERR |c| (FlCfg: the sums for both sizes, and a little), and
//    the norm from FP32 sums of squares (40 roundings on any way) is within 2^-19;
//  - the FP64 error has the rounding of both FP64 transforms in it, by the same
//    sums at most ROUND times the patch's norm;
//  - so a threshold fails where the norm of some fields less these passes the
//    bound, and passes where the norm with them stays below; in between (some
//    1e-4 of the bound), or with a node on the rounding boundary, FP64 decides
//    (err2_exact) as features_labels decides all of them.
// The label is the largest grid value that passes, so the grid is walked from
// the top and the walk ends at the first pass.  64 patches of 64 cells, nine
// fields: 16.1 ms before (41 inverse transforms of every field in FP64, a line
// in shared memory per thread), 0.45 to 0.6 ms now (a decision in FP64: 0.15 ms).
template <int P, int L> struct FlCfg {
  static constexpr int E = P + 1, N = E * E, NT = 256, NW = NT / 32;
  static constexpr double ERR = P == 64 ? 2.7e-5 : 1.1e-5, ROUND = P == 64 ? 4e-13 : 2e-13;
  static_assert((P == 64 && L == 4) || (P == 32 && L == 3), "the error bounds are of these sizes");
  static constexpr int FG = 2;  // FP64 tiles: fields transformed together
  static constexpr int TG = FG * 2;  // FP32 trial tiles in the same place
  static constexpr size_t OFF_RED = size_t(FG) * N * 8;
  static constexpr size_t OFF_C = OFF_RED + (2 * NW + 2 * NW * 3 * L + 8) * 8;
  static constexpr size_t smem(int F) { return OFF_C + size_t(F) * N * 4; }
};

template <int P, int L>
__global__ void __launch_bounds__(256) features_labels_reg(const float* __restrict__ dense, int F, int G0, int G1, int npx,
                                                            double delta, float* feat, float* label) {
  typedef FlCfg<P, L> C;
  constexpr int E = C::E, N = C::N, NT = C::NT, NW = C::NW, FG = C::FG, TG = C::TG, G = 3 * L;
  extern __shared__ __align__(16) unsigned char fsm[];
  double* tile = reinterpret_cast<double*>(fsm);
  float* trial = reinterpret_cast<float*>(fsm);
  double* red = reinterpret_cast<double*>(fsm + C::OFF_RED);  // warp partials
  double* ge = red + 2 * NW;                                  // [warp][G] energies, then maxima
  int* verdict = reinterpret_cast<int*>(ge + 2 * NW * G);
  float* c32 = reinterpret_cast<float*>(fsm + C::OFF_C);      // [F][N] coefficients
  const int pid = blockIdx.x, px = pid % npx, py = pid / npx;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  auto load = [&](int f, double* t) {  // nodes of field f
    for (int i = tid; i < N; i += NT) {
      const int y = i / E, x = i - y * E;
      const int gx = px * P + x < G0 ? px * P + x : 0, gy = py * P + y < G1 ? py * P + y : 0;
      t[i] = double(dense[(size_t(f) * G1 + gy) * G0 + gx]);
    }
  };
  // sum over the block, the same in every thread (fixed order)
  auto block_sum_w = [&](double v) -> double {
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) red[warp] = v;
    __syncthreads();
    double r = 0.0;
#pragma unroll
    for (int w = 0; w < NW; ++w) r += red[w];
    __syncthreads();
    return r;
  };
  // lines of FG tiles, one per thread at a time
  auto lines = [&](int nf, auto fn) {
    for (int t = tid; t < nf * E; t += NT) fn(t / E, t % E);
    __syncthreads();
  };

  // ---- forward transforms in FP64, features, FP32 copies
  double n2 = 0.0;
  for (int g = tid; g < NW * G * 2; g += NT) ge[g] = 0.0;
  __syncthreads();
  for (int f0 = 0; f0 < F; f0 += FG) {
    const int nf = F - f0 < FG ? F - f0 : FG;
    for (int q = 0; q < nf; ++q) load(f0 + q, tile + q * N);
    __syncthreads();
    lines(nf, [&](int q, int y) {
      double v[E];
      double* p = tile + q * N + y * E;
#pragma unroll
      for (int i = 0; i < E; ++i) {
        v[i] = p[i];
        n2 = wcs::fma_rn(v[i], v[i], n2);
      }
      wcs::fwd_levels<wcs::WV_BL53, P, 1, L, double>(v);
#pragma unroll
      for (int i = 0; i < E; ++i) p[i] = v[i];
    });
    // columns: whole warps take part (the group sums are shuffled)
    for (int t0 = 0; t0 < nf * E; t0 += NT) {
      const int t = t0 + tid, q = t / E, x = t - q * E;
      const bool on = t < nf * E;
      double acc[L + 1], mx[L + 1];
#pragma unroll
      for (int c = 0; c <= L; ++c) acc[c] = mx[c] = 0.0;
      if (on) {
        double v[E];
        const double* p = tile + q * N + x;
        float* cf = c32 + (f0 + q) * N + x;
#pragma unroll
        for (int i = 0; i < E; ++i) v[i] = p[i * E];
        wcs::fwd_levels<wcs::WV_BL53, P, 1, L, double>(v);
#pragma unroll
        for (int i = 0; i < E; ++i) {
          const int cy = wcs::node_class<L>(i);
          acc[cy] = wcs::fma_rn(v[i], v[i], acc[cy]);
          mx[cy] = fmax(mx[cy], fabs(v[i]));
          cf[i * E] = float(v[i]);
        }
      }
      const int cx = on ? wcs::node_class_rt<L>(x) : 0;
      // group (l, x): cx == l, rows below l; (l, y): cx < l, rows of l; (l, xy)
      double below = 0.0, bmx = 0.0;
#pragma unroll
      for (int l = 1; l <= L; ++l) {
        below += acc[l - 1];
        bmx = fmax(bmx, mx[l - 1]);
        const double e[3] = {on && cx == l ? below : 0.0, on && cx < l ? acc[l] : 0.0, on && cx == l ? acc[l] : 0.0};
        const double m[3] = {on && cx == l ? bmx : 0.0, on && cx < l ? mx[l] : 0.0, on && cx == l ? mx[l] : 0.0};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          double se = e[k], sm = m[k];
#pragma unroll
          for (int o = 16; o >= 1; o >>= 1) {
            se += __shfl_down_sync(0xffffffffu, se, o);
            sm = fmax(sm, __shfl_down_sync(0xffffffffu, sm, o));
          }
          if (lane == 0) {
            const int g = 3 * (l - 1) + k;
            ge[warp * G + g] += se;
            ge[(NW + warp) * G + g] = fmax(ge[(NW + warp) * G + g], sm);
          }
        }
      }
    }
    __syncthreads();
  }
  const double norm2 = block_sum_w(n2);
  if (tid < G) {
    double e = 0.0, m = 0.0;
    for (int w = 0; w < NW; ++w) {
      e += ge[w * G + tid];
      m = fmax(m, ge[(NW + w) * G + tid]);
    }
    // nodes of the group: nc(c) nodes of class c on a line
    const int l = tid / 3 + 1, k = tid % 3;
    auto nc = [](int c) { return c == 0 ? (P >> L) + 1 : P >> c; };
    int lower = 0;  // nodes of a class below l
    for (int c = 0; c < l; ++c) lower += nc(c);
    const int cnt = k == 2 ? nc(l) * nc(l) : nc(l) * lower;
    feat[size_t(pid) * 2 * G + 2 * tid] = float(log10(e / (double(cnt) * F) + 1e-30));
    feat[size_t(pid) * 2 * G + 2 * tid + 1] = float(log10(m + 1e-30));
  }

  // ---- label
  const double bound = delta * sqrt(norm2), bound2 = bound * bound;
  const double rnd = C::ROUND * sqrt(norm2);
  const bool fp32 = bound2 > 1e-24 && bound2 < 1e24;  // far from the ends of FP32's range
  auto err2_exact = [&](double eps) -> double {  // FP64, field by field
    double err2 = 0.0;
    for (int f = 0; f < F; ++f) {
      __syncthreads();
      load(f, tile);
      load(f, tile + N);
      __syncthreads();
      lines(1, [&](int, int y) { wcs::line_transform<wcs::WV_BL53, P, L, false, double>(tile + y * E, 1); });
      lines(1, [&](int, int x) {
        double v[E];
#pragma unroll
        for (int i = 0; i < E; ++i) v[i] = tile[i * E + x];
        wcs::fwd_levels<wcs::WV_BL53, P, 1, L, double>(v);
        const bool xc = (x & ((1 << L) - 1)) == 0;
#pragma unroll
        for (int i = 0; i < E; ++i)
          if (!(xc && (i & ((1 << L) - 1)) == 0) && !(fabs(v[i]) >= eps)) v[i] = 0.0;
        wcs::inv_levels<wcs::WV_BL53, P, L, double>(v);
#pragma unroll
        for (int i = 0; i < E; ++i) tile[i * E + x] = v[i];
      });
      double my = 0.0;
      lines(1, [&](int, int y) {
        double v[E];
#pragma unroll
        for (int i = 0; i < E; ++i) v[i] = tile[y * E + i];
        wcs::inv_levels<wcs::WV_BL53, P, L, double>(v);
#pragma unroll
        for (int i = 0; i < E; ++i) {
          const double d = v[i] - tile[N + y * E + i];
          my += d * d;
        }
      });
      err2 += block_sum_w(my);
      if (sqrt(err2) > bound) return err2;  // more fields only add to it
    }
    return err2;
  };
  auto passes = [&](double eps) -> bool {
    const float e32 = float(eps);
    float s = 0.0f, c2 = 0.0f;  // thread 0: squared norms of the error and of c so far
    int said = 0;               // 1: the threshold fails, 2: it passes
    bool tie = !fp32;
    for (int f0 = 0; f0 < F && fp32; f0 += TG) {
      const int nf = F - f0 < TG ? F - f0 : TG;
      float mc = 0.0f, my = 0.0f;
      lines(nf, [&](int q, int x) {
        const float* c = c32 + (f0 + q) * N + x;
        const bool xc = (x & ((1 << L) - 1)) == 0;
        float v[E], part[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int i = 0; i < E; ++i) {
          v[i] = c[i * E];
          const bool coarse = xc && (i & ((1 << L) - 1)) == 0;
          tie = tie || (!coarse && fabsf(v[i]) == e32);
          if (coarse || fabsf(v[i]) >= e32) v[i] = 0.0f;
          part[i & 3] = __fmaf_rn(v[i], v[i], part[i & 3]);
        }
        mc += (part[0] + part[1]) + (part[2] + part[3]);
        wcs::inv_levels<wcs::WV_BL53, P, L, float>(v);
#pragma unroll
        for (int i = 0; i < E; ++i) trial[q * N + i * E + x] = v[i];
      });
      lines(nf, [&](int q, int y) {
        float v[E];
#pragma unroll
        for (int i = 0; i < E; ++i) v[i] = trial[q * N + y * E + i];
        wcs::inv_levels<wcs::WV_BL53, P, L, float>(v);
        float part[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int i = 0; i < E; ++i) part[i & 3] = __fmaf_rn(v[i], v[i], part[i & 3]);
        my += (part[0] + part[1]) + (part[2] + part[3]);
      });
#pragma unroll
      for (int o = 16; o >= 1; o >>= 1) {
        my += __shfl_down_sync(0xffffffffu, my, o);
        mc += __shfl_down_sync(0xffffffffu, mc, o);
      }
      float* fred = reinterpret_cast<float*>(red);
      if (lane == 0) {
        fred[warp] = my;
        fred[NW + warp] = mc;
      }
      __syncthreads();
      if (tid == 0) {  // (the FP64 operations once: in every thread they took 4 us a threshold)
#pragma unroll
        for (int k = 0; k < NW; ++k) {
          s += fred[k];
          c2 += fred[NW + k];
        }
        const double e = sqrtf(s), off = C::ERR * sqrtf(c2) + e * 0x1p-19 + rnd;
        *verdict = e - off > bound ? 1 : (f0 + TG >= F && e + off < bound ? 2 : 0);
      }
      __syncthreads();
      said = *verdict;
      if (said == 1) break;
    }
    tie = __syncthreads_or(tie);
    if (!tie && said) return said == 2;
    return sqrt(err2_exact(eps)) <= bound;
  };
  int best = EPS_N - 1;
  while (best >= 0 && !passes(c_eps_grid[best])) --best;
  double lab;
  if (best < 0) {
    lab = -7.0;
  } else if (best == EPS_N - 1) {
    lab = -2.0;
  } else {
    double lo = c_eps_grid[best], hi = c_eps_grid[best + 1];
    for (int it = 0; it < 4; ++it) {
      const double mid = sqrt(lo * hi);
      if (passes(mid)) lo = mid;
      else hi = mid;
    }
    lab = log10(lo);
  }
  if (tid == 0) label[pid] = float(lab);
}

template <int P, int L>
cudaError_t run_features_labels_reg(const float* dense, int F, int64_t nx, int64_t ny, double delta, float* feat,
                                    float* label, cudaStream_t st) {
  const size_t smem = FlCfg<P, L>::smem(F);
  cudaError_t e = cudaFuncSetAttribute(features_labels_reg<P, L>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
  if (e != cudaSuccess) return e;
  const int npx = int(nx / P), npy = int(ny / P);
  features_labels_reg<P, L><<<npx * npy, 256, smem, st>>>(dense, F, int(nx), int(ny), npx, delta, feat, label);
  return cudaGetLastError();
}

// ------------------------------------------------ 3-D features and labels
// Cubic BL5/3 patches of P cells (the D3Q19 path): FP32 lifting in a shared
// tile (the precision of the 3-D step), a CTA per patch in a stride, the
// forward-transformed fields kept in a global scratch slot of F (P+1)^3
// floats per CTA.  Features: energy (FP64) and max per band, summed per z
// line and then over the band's lines in order; groups (l, S) over the 7 axis
// sets.  Labels as in 2-D: the grid is walked from the top, and a threshold
// ends at the field whose error passes the bound.  The error of a threshold
// is that of the FP32 inverse transform, so the transform stays as it is; the
// differences t - u are taken and squared in FP32 and added eight at a time in
// FP32, then in FP64: a difference is within 2^-24 of itself, its square within
// 3 x 2^-24, a sum of eight squares within 11 x 2^-24 = 7e-7, at any delta (t
// and u are the same FP32 numbers either way); only where the sum lies within
// FL3_MARGIN of the bound is it taken again in FP64.  What bounded
// the kernel was that sum (five FP64 operations per node, two per cycle and
// SM), run-time modulos per node, and a thread walking a whole band: 132 ms
// for 48 patches of 32 cells (every threshold in full), now 13.5 ms
// (82 ms with the early ends alone).
constexpr double FL3_MARGIN = 1e-5;
template <int P, int L> struct Fl3Cfg {
  static constexpr int E = P + 1, E2 = E * E, E3 = E2 * E;
  static constexpr int NT = P >= 32 ? 576 : 320, NWARP = NT / 32, MINB = P >= 32 ? 1 : 3;
  static constexpr int NB = (L + 1) * (L + 1) * (L + 1);
  static constexpr size_t OFF_LE = (size_t(E3) * 4 + 15) / 16 * 16;         // per z line and z class: energy
  static constexpr size_t OFF_LM = OFF_LE + size_t(E2) * (L + 1) * 8;       //   and maximum
  static constexpr size_t OFF_RED = (OFF_LM + size_t(E2) * (L + 1) * 4 + 15) / 16 * 16;  // NWARP partial sums
  static constexpr size_t OFF_BE = OFF_RED + size_t(NWARP) * 8;             // band energy (all fields)
  static constexpr size_t OFF_BM = OFF_BE + size_t(NB) * 8;                 // band max
  static constexpr size_t SMEM = OFF_BM + size_t(NB) * 4;
};
template <int P, int L>
__global__ void __launch_bounds__(Fl3Cfg<P, L>::NT, Fl3Cfg<P, L>::MINB)
    features_labels3(const float* __restrict__ dense, int F, int G0, int G1, int G2, int npx, int npy, int npz,
                     double delta, float* __restrict__ cscr, unsigned long long slot, float* feat, float* label) {
  typedef Fl3Cfg<P, L> K;
  constexpr int E = K::E, E2 = K::E2, E3 = K::E3, NT = K::NT, NWARP = K::NWARP, G = 7 * L, NB = K::NB;
  extern __shared__ __align__(16) unsigned char sm3[];
  float* tile = reinterpret_cast<float*>(sm3);
  double* le = reinterpret_cast<double*>(sm3 + K::OFF_LE);
  float* lm = reinterpret_cast<float*>(sm3 + K::OFF_LM);
  double* wred = reinterpret_cast<double*>(sm3 + K::OFF_RED);
  double* be = reinterpret_cast<double*>(sm3 + K::OFF_BE);
  float* bmx = reinterpret_cast<float*>(sm3 + K::OFF_BM);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float* C = cscr + size_t(blockIdx.x) * slot;
  const size_t vol = size_t(G0) * G1 * G2;
  // lines along x (0) or y (1): thread per line
  auto lines = [&](int axis, bool inverse) {
    for (int l = tid; l < E2; l += NT) {
      const int u = l % E, v = l / E;
      float* q = axis == 0 ? tile + v * E2 + u * E : tile + v * E2 + u;
      const int st = axis == 0 ? 1 : E;
      if (inverse) wcs::line_transform<wcs::WV_BL53, P, L, true, float>(q, st);
      else wcs::line_transform<wcs::WV_BL53, P, L, false, float>(q, st);
    }
    __syncthreads();
  };
  auto block_sum = [&](double v) -> double {  // fixed order: shuffle tree, then warps in order
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) wred[warp] = v;
    __syncthreads();
    double r = 0.0;
    for (int w = 0; w < NWARP; ++w) r += wred[w];
    __syncthreads();
    return r;
  };
  const int np = npx * npy * npz;
  for (int pid = blockIdx.x; pid < np; pid += gridDim.x) {
    const int px = pid % npx, py = (pid / npx) % npy, pz = pid / (npx * npy);
    // a warp per row (y, z): fn(index in the tile, global index, lane's node exists)
    auto rows = [&](auto fn) {
#pragma unroll 4
      for (int r = warp; r < E2; r += NWARP) {
        const int z = r / E, y = r - z * E;
        const int gy = py * P + y < G1 ? py * P + y : 0, gz = pz * P + z < G2 ? pz * P + z : 0;
        const size_t row = (size_t(gz) * G1 + gy) * G0;
        if (E <= 32) {
          if (lane < E) fn(r * E + lane, row + (px * P + lane < G0 ? px * P + lane : 0));
        } else {
          fn(r * E + lane, row + px * P + lane);
          if (lane == 0) fn(r * E + P, row + (px * P + P < G0 ? px * P + P : 0));
        }
      }
    };
    if (tid < NB) {
      be[tid] = 0.0;
      bmx[tid] = 0.0f;
    }
    double n2 = 0.0;
    for (int f = 0; f < F; ++f) {
      const float* uf = dense + size_t(f) * vol;
      float* Cf = C + size_t(f) * E3;
      rows([&](int i, size_t g) {
        const float v = uf[g];
        tile[i] = v;
        n2 += double(v) * double(v);
      });
      __syncthreads();
      lines(0, false);
      lines(1, false);
      for (int l = tid; l < E2; l += NT) {  // z lines (x, y): coefficients out, their sums per z class
        float v[E];
#pragma unroll
        for (int z = 0; z < E; ++z) v[z] = tile[z * E2 + l];
        wcs::fwd_levels<wcs::WV_BL53, P, 1, L, float>(v);
        double e[L + 1];
        float m[L + 1];
#pragma unroll
        for (int c = 0; c <= L; ++c) {
          e[c] = 0.0;
          m[c] = 0.0f;
        }
#pragma unroll
        for (int z = 0; z < E; ++z) {
          const int c = wcs::node_class<L>(z);
          e[c] = wcs::fma_rn(double(v[z]), double(v[z]), e[c]);
          m[c] = fmaxf(m[c], fabsf(v[z]));
          Cf[z * E2 + l] = v[z];
        }
#pragma unroll
        for (int c = 0; c <= L; ++c) {
          le[c * E2 + l] = e[c];
          lm[c * E2 + l] = m[c];
        }
      }
      __syncthreads();
      if (tid > 0 && tid < NB) {  // band b: its lines in order
        const int b = tid, cx = b / ((L + 1) * (L + 1)), cy = (b / (L + 1)) % (L + 1), cz = b % (L + 1);
        const int sx = cx ? 1 << cx : 1 << L, sy = cy ? 1 << cy : 1 << L;  // nodes of a class: a stride, from half of it on (coarse: from 0)
        double e = 0.0;
        float m = 0.0f;
        for (int y = cy ? sy / 2 : 0; y < E; y += sy)
          for (int x = cx ? sx / 2 : 0; x < E; x += sx) {
            e += le[cz * E2 + y * E + x];
            m = fmaxf(m, lm[cz * E2 + y * E + x]);
          }
        be[b] += e;
        bmx[b] = fmaxf(bmx[b], m);
      }
      __syncthreads();
    }
    const double norm2 = block_sum(n2);
    if (tid < G) {  // group g: level l, axes S; bands of the group in band order
      const int g = tid, l = g / 7 + 1, S = g % 7 + 1;
      double e = 0.0;
      float m = 0.0f;
      long long cnt = 0;
      for (int b = 1; b < NB; ++b) {
        const int c[3] = {b / ((L + 1) * (L + 1)), (b / (L + 1)) % (L + 1), b % (L + 1)};
        const int bl = max(c[0], max(c[1], c[2]));
        const int bs = (c[0] == bl ? 1 : 0) | (c[1] == bl ? 2 : 0) | (c[2] == bl ? 4 : 0);
        if (bl != l || bs != S) continue;
        e += be[b];
        m = fmaxf(m, bmx[b]);
        long long nb = 1;
        for (int a = 0; a < 3; ++a) nb *= c[a] ? P >> c[a] : (P >> L) + 1;
        cnt += nb;
      }
      feat[size_t(pid) * 2 * G + 2 * g] = float(log10(e / double(cnt * F) + 1e-30));
      feat[size_t(pid) * 2 * G + 2 * g + 1] = float(log10(double(m) + 1e-30));
    }
    const double bound = delta * sqrt(norm2), bound2 = bound * bound;
    const bool fp32 = bound > 0.0 && bound2 > 1e-24 && bound2 < 1e24;  // far from the ends of FP32's range
    // squared error of thresholding at eps, up to the field that passes the
    // bound (a partial sum only grows); exact: squares and sums in FP64
    auto err2_of = [&](double eps, auto exact) -> double {
      constexpr bool X = decltype(exact)::value;
      double acc = 0.0, sum = 0.0;
      for (int f = 0; f < F; ++f) {
        const float* Cf = C + size_t(f) * E3;
        for (int l = tid; l < E2; l += NT) {  // threshold and inverse z lifting
          const bool xy = ((l % E) | (l / E)) & ((1 << L) - 1);
          float v[E];
#pragma unroll
          for (int z = 0; z < E; ++z) v[z] = Cf[z * E2 + l];
#pragma unroll
          for (int z = 0; z < E; ++z)
            if ((xy || (z & ((1 << L) - 1))) && !(fabs(double(v[z])) >= eps)) v[z] = 0.0f;
          wcs::inv_levels<wcs::WV_BL53, P, L, float>(v);
#pragma unroll
          for (int z = 0; z < E; ++z) tile[z * E2 + l] = v[z];
        }
        __syncthreads();
        lines(1, true);
        lines(0, true);
        const float* uf = dense + size_t(f) * vol;
        float part = 0.0f;
        int k = 0;
        rows([&](int i, size_t g) {
          if constexpr (X) {
            const double d = double(tile[i]) - double(uf[g]);
            acc += d * d;
          } else {
            const float d = tile[i] - uf[g];
            part = __fmaf_rn(d, d, part);
            if ((++k & 7) == 0) {  // eight squares in FP32, then FP64
              acc += double(part);
              part = 0.0f;
            }
          }
        });
        acc += double(part);
        __syncthreads();
        sum = block_sum(acc);
        if (X ? sqrt(sum) > bound : sum > bound2 * (1.0 + FL3_MARGIN)) break;
      }
      return sum;
    };
    auto passes = [&](double eps) -> bool {
      if (fp32) {
        const double s = err2_of(eps, std::false_type());
        if (s > bound2 * (1.0 + FL3_MARGIN)) return false;
        if (s < bound2 * (1.0 - FL3_MARGIN)) return true;
      }
      return sqrt(err2_of(eps, std::true_type())) <= bound;
    };
    int best = EPS_N - 1;
    while (best >= 0 && !passes(c_eps_grid[best])) --best;
    double lab;
    if (best < 0) {
      lab = -7.0;
    } else if (best == EPS_N - 1) {
      lab = -2.0;
    } else {
      double lo = c_eps_grid[best], hi = c_eps_grid[best + 1];
      for (int it = 0; it < 4; ++it) {
        const double mid = sqrt(lo * hi);
        if (passes(mid)) lo = mid;
        else hi = mid;
      }
      lab = log10(lo);
    }
    if (tid == 0) label[pid] = float(lab);
    __syncthreads();
  }
}

template <int P, int L>
wcs_status run_features_labels3(const float* dense, int nfields, int64_t nx, int64_t ny, int64_t nz, double delta,
                                float* feat, float* label, cudaStream_t st) {
  const size_t smem = Fl3Cfg<P, L>::SMEM;
  if (cudaFuncSetAttribute(features_labels3<P, L>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)) != cudaSuccess)
    return WCS_E_CUDA;
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const int npx = int(nx / P), npy = int(ny / P), npz = int(nz / P), np = npx * npy * npz;
  int grid = std::min(np, nsm * Fl3Cfg<P, L>::MINB);
  const unsigned long long slot = (unsigned long long)nfields * (P + 1) * (P + 1) * (P + 1);
  float* cscr = nullptr;
  while (cudaMalloc(&cscr, size_t(grid) * slot * 4) != cudaSuccess) {  // little memory left: fewer CTAs
    cudaGetLastError();
    if (grid == 1) return WCS_E_OOM;
    grid = (grid + 1) / 2;
  }
  features_labels3<P, L><<<grid, Fl3Cfg<P, L>::NT, smem, st>>>(dense, nfields, int(nx), int(ny), int(nz), npx, npy,
                                                               npz, delta, cscr, slot, feat, label);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFree(cscr);
  return e == cudaSuccess ? WCS_OK : WCS_E_CUDA;
}

// ------------------------------------------------------------------ MLP
__device__ inline float gelu(float x) { return wcs::gelu_f(x); }
__device__ inline float gelu_grad(float x) {
  return 0.5f * (1.0f + erff(x * 0.70710678118654752f)) + x * expf(-0.5f * x * x) * 0.39894228040143268f;
}

// Block per slice of a minibatch: CTA b takes samples [b S, b S + S) (S =
// MLP_SPB), stages the weights, the inputs and every activation of its
// samples in shared memory, and writes its partial gradient (the sum over
// its samples, in sample order) to gpart[b][p] and its summed squared error
// to lpart[b].  Per sample: z1 = b1 + W1 x and z2 = b2 + W2 gelu(z1) (sums
// in input order), y = b3 + W3 gelu(z2), error r = y - t, loss r^2,
// dy = 2 r / B, d2 = dy W3 gelu'(z2), d1 = (W2^T d2) gelu'(z1); the
// gradients are the outer products of these with the layer inputs.
// Threads take (sample, unit) pairs in the forward pass and parameters in
// the backward pass.
constexpr int MLP_SPB = 16;
__host__ __device__ inline size_t block_grads_smem(int nin) {
  return (size_t(nparam(nin)) + size_t(MLP_SPB) * (nin + 5 * MLP_NH + 2)) * 4;
}
__global__ void __launch_bounds__(256) mlp_block_grads(const float* __restrict__ w, int nin,
                                                       const float* __restrict__ X, const float* __restrict__ t,
                                                       const int* __restrict__ idx, int B, float* __restrict__ gpart,
                                                       float* __restrict__ lpart) {
  extern __shared__ float msm[];
  constexpr int S = MLP_SPB, H = MLP_NH;
  const int np = nparam(nin), tid = threadIdx.x, NT = blockDim.x;
  const int s0 = blockIdx.x * S, ns = min(S, B - s0);
  float* W = msm;
  float* x = W + np;
  float* z1 = x + S * nin;
  float* a1 = z1 + S * H;
  float* z2 = a1 + S * H;
  float* d2 = z2 + S * H;
  float* d1 = d2 + S * H;
  float* dy = d1 + S * H;
  float* ls = dy + S;
  const float* W1 = W;
  const float* b1 = W1 + H * nin;
  const float* W2 = b1 + H;
  const float* b2 = W2 + H * H;
  const float* W3 = b2 + H;
  const float* b3 = W3 + H;
  for (int p = tid; p < np; p += NT) W[p] = w[p];
  for (int q = tid; q < ns * nin; q += NT) {
    const int sl = q / nin, i = q - sl * nin, g = s0 + sl;
    x[q] = X[size_t(idx ? idx[g] : g) * nin + i];
  }
  __syncthreads();
  for (int q = tid; q < ns * H; q += NT) {  // first layer
    const int sl = q / H, j = q - sl * H;
    float a = b1[j];
    for (int i = 0; i < nin; ++i) a += W1[j * nin + i] * x[sl * nin + i];
    z1[q] = a;
    a1[q] = gelu(a);
  }
  __syncthreads();
  for (int q = tid; q < ns * H; q += NT) {  // second layer
    const int sl = q / H, j = q - sl * H;
    float a = b2[j];
    for (int i = 0; i < H; ++i) a += W2[j * H + i] * a1[sl * H + i];
    z2[q] = a;
  }
  __syncthreads();
  if (tid < ns) {  // output, error and its derivative
    float y = b3[0];
    for (int j = 0; j < H; ++j) y += W3[j] * gelu(z2[tid * H + j]);
    const int g = s0 + tid;
    const float r = y - t[idx ? idx[g] : g];
    ls[tid] = r * r;
    dy[tid] = 2.0f * r / float(B);
  }
  __syncthreads();
  for (int q = tid; q < ns * H; q += NT) {
    const int sl = q / H, j = q - sl * H;
    d2[q] = dy[sl] * W3[j] * gelu_grad(z2[q]);
  }
  __syncthreads();
  for (int q = tid; q < ns * H; q += NT) {
    const int sl = q / H, i = q - sl * H;
    float a = 0.0f;
    for (int j = 0; j < H; ++j) a += d2[sl * H + j] * W2[j * H + i];
    d1[q] = a * gelu_grad(z1[q]);
  }
  __syncthreads();
  float* gp = gpart + size_t(blockIdx.x) * np;
  for (int p = tid; p < np; p += NT) {  // every parameter: its sum over the slice's samples
    float a = 0.0f;
    if (p < H * nin) {
      const int j = p / nin, k = p - j * nin;
      for (int sl = 0; sl < ns; ++sl) a += d1[sl * H + j] * x[sl * nin + k];
    } else if (p < H * nin + H) {
      const int j = p - H * nin;
      for (int sl = 0; sl < ns; ++sl) a += d1[sl * H + j];
    } else if (p < H * nin + H + H * H) {
      const int r = p - H * nin - H, j = r / H, i = r - j * H;
      for (int sl = 0; sl < ns; ++sl) a += d2[sl * H + j] * a1[sl * H + i];
    } else if (p < H * nin + 2 * H + H * H) {
      const int j = p - H * nin - H - H * H;
      for (int sl = 0; sl < ns; ++sl) a += d2[sl * H + j];
    } else if (p < np - 1) {
      const int j = p - H * nin - 2 * H - H * H;
      for (int sl = 0; sl < ns; ++sl) a += dy[sl] * gelu(z2[sl * H + j]);
    } else {
      for (int sl = 0; sl < ns; ++sl) a += dy[sl];
    }
    gp[p] = a;
  }
  if (tid == 0) {
    float a = 0.0f;
    for (int sl = 0; sl < ns; ++sl) a += ls[sl];
    lpart[blockIdx.x] = a;
  }
}

// A whole training run in one launch, for minibatches of up to 8 slices: one
// cluster of eight CTAs, CTA r takes slice r of every minibatch.  The steps are
// a chain (each needs the weights of the one before), so the latency of one
// step is the time; as a launch of a few CTAs plus a launch for the sums it
// was 38 us a step for 128 samples and 24 inputs (weights re-read, 32-way bank
// conflicts on the weight rows, 64 erff one after the other per sample, two
// launches), now 10.9 us.  The weights stay in every CTA's shared memory, each CTA
// owns an eighth of the parameters with their Adam state: partial gradients
// are read from the other CTAs' shared memory, the new weights written to it.
// Every sum runs in the order of mlp_block_grads and mlp_reduce_partials, so
// the weights are the same bits.  A thread holds two samples times two units
// (lane and lane + 32) in both layers and keeps their activations'
// derivatives in registers; the next minibatch's inputs are fetched meanwhile.
constexpr int TC_CTAS = 8, TC_NT = 256, TC_S2 = MLP_NH + 4;  // row pitch of W2: float4 reads without conflicts
constexpr int TC_XMAX = (MLP_SPB * MLP_MAXIN + TC_NT - 1) / TC_NT;
__host__ __device__ inline int tc_s1(int nin) { return nin | 1; }
__host__ __device__ inline int tc_chunk(int nin) { return (nparam(nin) + TC_CTAS - 1) / TC_CTAS; }
__host__ __device__ inline size_t tc_smem(int nin) {
  return (size_t(MLP_NH) * TC_S2 + 4 * size_t(MLP_SPB) * MLP_NH + size_t(MLP_NH) * tc_s1(nin) + 3 * MLP_NH + 4 +
          size_t(nparam(nin)) + 2 * size_t(tc_chunk(nin)) + size_t(MLP_SPB) * nin + 3 * MLP_SPB + 8) * 4;
}
__global__ void __cluster_dims__(TC_CTAS, 1, 1) __launch_bounds__(TC_NT)
    mlp_train_cluster(float* __restrict__ w, float* __restrict__ gm1, float* __restrict__ gm2, int nin,
                      const float* __restrict__ X, const float* __restrict__ t, const int* __restrict__ idx, int nsteps,
                      int nb, int B, float lr, float b1c, float b2c, const float2* __restrict__ bt,
                      float* __restrict__ loss) {
  extern __shared__ __align__(16) float tsm[];
  constexpr int H = MLP_NH, S = MLP_SPB, NT = TC_NT;
  cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
  const int r = int(cl.block_rank()), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int np = nparam(nin), S1 = tc_s1(nin), chunk = tc_chunk(nin), G = (B + S - 1) / S;
  float* W2 = tsm;                 // [H][TC_S2]
  float* a1 = W2 + H * TC_S2;      // [S][H]
  float* pw = a1 + S * H;          // [S][H] W3 a2, then a2
  float* d2 = pw + S * H;          // [S][H]
  float* d1 = d2 + S * H;          // [S][H]
  float* W1 = d1 + S * H;          // [H][S1]
  float* b1 = W1 + H * S1;
  float* b2 = b1 + H;
  float* W3 = b2 + H;
  float* b3 = W3 + H;              // 1 (+ 3)
  float* gp = b3 + 4;              // this CTA's partial gradient
  float* m1 = gp + np;             // Adam state of the owned parameters
  float* m2 = m1 + chunk;
  float* x = m2 + chunk;           // [S][nin]
  float* ts = x + S * nin;         // targets
  float* dy = ts + S;
  float* ls = dy + S;              // squared errors, then their sum in ls[S]
  // where parameter p lives in the padded layout
  auto slot = [&](int p) -> float* {
    if (p < H * nin) return W1 + (p / nin) * S1 + p % nin;
    p -= H * nin;
    if (p < H) return b1 + p;
    p -= H;
    if (p < H * H) return W2 + (p / H) * TC_S2 + p % H;
    p -= H * H;
    return p < H ? b2 + p : (p < 2 * H ? W3 + (p - H) : b3);
  };
  const int p0 = r * chunk, p1 = min(np, p0 + chunk);
  for (int p = tid; p < np; p += NT) *slot(p) = w[p];
  for (int p = p0 + tid; p < p1; p += NT) {
    m1[p - p0] = gm1[p];
    m2[p - p0] = gm2[p];
  }
  const int s0 = r * S, ns = max(0, min(S, B - s0));  // this CTA's samples of a minibatch
  // inputs of a step: element q = tid + k NT of [ns][nin], and the targets
  int xi[TC_XMAX], ti = 0;
  float xv[TC_XMAX], tv = 0.0f;
  auto fetch_index = [&](int st) {
#pragma unroll
    for (int k = 0; k < TC_XMAX; ++k) {
      const int q = tid + k * NT;
      xi[k] = q < ns * nin ? idx[size_t(st) * B + s0 + q / nin] : 0;
    }
    if (tid < ns) ti = idx[size_t(st) * B + s0 + tid];
  };
  auto fetch_values = [&]() {
#pragma unroll
    for (int k = 0; k < TC_XMAX; ++k) {
      const int q = tid + k * NT;
      if (q < ns * nin) xv[k] = X[size_t(xi[k]) * nin + q % nin];
    }
    if (tid < ns) tv = t[ti];
  };
  auto store_values = [&]() {
#pragma unroll
    for (int k = 0; k < TC_XMAX; ++k) {
      const int q = tid + k * NT;
      if (q < ns * nin) x[q] = xv[k];
    }
    if (tid < ns) ts[tid] = tv;
  };
  fetch_index(0);
  fetch_values();
  store_values();
  cl.sync();
  const int sa = 2 * warp, sb = sa + 1;  // this thread's samples; its units: lane, lane + 32
  static_assert(S == 2 * (NT / 32) && H == 64, "two samples per warp, two units per lane");
  for (int st = 0; st < nsteps; ++st) {
    if (st + 1 < nsteps) fetch_index(st + 1);
    float g1[2][2], g2[2][2];
    {  // first layer
      float z[2][2] = {{b1[lane], b1[lane + 32]}, {b1[lane], b1[lane + 32]}};
      const float *wa = W1 + lane * S1, *wb = W1 + (lane + 32) * S1;
#pragma unroll 4
      for (int i = 0; i < nin; ++i) {
        const float xa = x[sa * nin + i], xb = x[sb * nin + i], u = wa[i], v = wb[i];
        z[0][0] += u * xa;
        z[0][1] += v * xa;
        z[1][0] += u * xb;
        z[1][1] += v * xb;
      }
#pragma unroll
      for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          a1[(sa + s) * H + lane + 32 * j] = gelu(z[s][j]);
          g1[s][j] = gelu_grad(z[s][j]);
        }
    }
    __syncthreads();
    if (st + 1 < nsteps) fetch_values();
    float a2[2][2];
    {  // second layer
      float z[2][2] = {{b2[lane], b2[lane + 32]}, {b2[lane], b2[lane + 32]}};
      const float4 *wa = reinterpret_cast<const float4*>(W2 + lane * TC_S2), *wb = reinterpret_cast<const float4*>(W2 + (lane + 32) * TC_S2);
      const float4 *aa = reinterpret_cast<const float4*>(a1 + sa * H), *ab = reinterpret_cast<const float4*>(a1 + sb * H);
#pragma unroll 4
      for (int i = 0; i < H / 4; ++i) {
        const float4 u4 = wa[i], v4 = wb[i], x4 = aa[i], y4 = ab[i];
        const float u[4] = {u4.x, u4.y, u4.z, u4.w}, v[4] = {v4.x, v4.y, v4.z, v4.w};
        const float xa[4] = {x4.x, x4.y, x4.z, x4.w}, xb[4] = {y4.x, y4.y, y4.z, y4.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          z[0][0] += u[k] * xa[k];
          z[0][1] += v[k] * xa[k];
          z[1][0] += u[k] * xb[k];
          z[1][1] += v[k] * xb[k];
        }
      }
#pragma unroll
      for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          a2[s][j] = gelu(z[s][j]);
          g2[s][j] = gelu_grad(z[s][j]);
          pw[(sa + s) * H + lane + 32 * j] = W3[lane + 32 * j] * a2[s][j];
        }
    }
    __syncthreads();
    if (tid < ns) {  // output, error and its derivative
      float y = b3[0];
#pragma unroll 8
      for (int j = 0; j < H; ++j) y += pw[tid * H + j];
      const float e = y - ts[tid];
      ls[tid] = e * e;
      dy[tid] = 2.0f * e / float(B);
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int u = lane + 32 * j;
        if (sa + s < ns) d2[(sa + s) * H + u] = dy[sa + s] * W3[u] * g2[s][j];
        pw[(sa + s) * H + u] = a2[s][j];
      }
    __syncthreads();
    {  // d1 = (W2^T d2) gelu'(z1)
      float q[2][2] = {{0.0f, 0.0f}, {0.0f, 0.0f}};
#pragma unroll 8
      for (int j = 0; j < H; ++j) {
        const float da = d2[sa * H + j], db = d2[sb * H + j], u = W2[j * TC_S2 + lane], v = W2[j * TC_S2 + lane + 32];
        q[0][0] += da * u;
        q[0][1] += da * v;
        q[1][0] += db * u;
        q[1][1] += db * v;
      }
#pragma unroll
      for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int j = 0; j < 2; ++j)
          if (sa + s < ns) d1[(sa + s) * H + lane + 32 * j] = q[s][j] * g1[s][j];
    }
    if (r < G) {  // gradients that need no d1: W2 (8 rows per warp, 2 columns per lane), b2, W3, b3, the loss
      float q[8][2];
#pragma unroll
      for (int k = 0; k < 8; ++k) q[k][0] = q[k][1] = 0.0f;
      for (int sl = 0; sl < ns; ++sl) {
        const float u = a1[sl * H + lane], v = a1[sl * H + lane + 32];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const float d = d2[sl * H + 8 * warp + k];
          q[k][0] += d * u;
          q[k][1] += d * v;
        }
      }
      float* o = gp + H * nin + H;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        o[(8 * warp + k) * H + lane] = q[k][0];
        o[(8 * warp + k) * H + lane + 32] = q[k][1];
      }
      o += H * H;
      if (tid < H) {
        float a = 0.0f;
        for (int sl = 0; sl < ns; ++sl) a += d2[sl * H + tid];
        o[tid] = a;
      } else if (tid < 2 * H) {
        const int j = tid - H;
        float a = 0.0f;
        for (int sl = 0; sl < ns; ++sl) a += dy[sl] * pw[sl * H + j];
        o[H + j] = a;
      } else if (tid == 2 * H) {
        float a = 0.0f;
        for (int sl = 0; sl < ns; ++sl) a += dy[sl];
        o[2 * H] = a;
      } else if (tid == 2 * H + 32) {
        float a = 0.0f;
        for (int sl = 0; sl < ns; ++sl) a += ls[sl];
        ls[S] = a;
      }
    }
    __syncthreads();
    if (r < G) {  // W1, b1
      for (int p = tid; p < H * nin; p += NT) {
        const int j = p / nin, k = p - j * nin;
        float a = 0.0f;
        for (int sl = 0; sl < ns; ++sl) a += d1[sl * H + j] * x[sl * nin + k];
        gp[p] = a;
      }
      if (tid < H) {
        float a = 0.0f;
        for (int sl = 0; sl < ns; ++sl) a += d1[sl * H + tid];
        gp[H * nin + tid] = a;
      }
    }
    cl.sync();
    if (st + 1 < nsteps) store_values();
    const float2 pt = bt[st];
    for (int p = p0 + tid; p < p1; p += NT) {  // the owned parameters: sum over the slices in order, Adam, new weight to all
      float v[TC_CTAS];
#pragma unroll
      for (int b = 0; b < TC_CTAS; ++b) v[b] = b < G ? cl.map_shared_rank(gp, b)[p] : 0.0f;
      float a = 0.0f;
#pragma unroll
      for (int b = 0; b < TC_CTAS; ++b)
        if (b < G) a += v[b];
      const float n1 = b1c * m1[p - p0] + (1.0f - b1c) * a, n2 = b2c * m2[p - p0] + (1.0f - b2c) * a * a;
      m1[p - p0] = n1;
      m2[p - p0] = n2;
      const float mh = n1 / (1.0f - pt.x), vh = n2 / (1.0f - pt.y);
      float* at = slot(p);
      const float wn = *at - lr * mh / (sqrtf(vh) + 1e-8f);
#pragma unroll
      for (int b = 0; b < TC_CTAS; ++b) *cl.map_shared_rank(at, b) = wn;
    }
    if (r == 0 && tid == 0 && (st + 1) % nb == 0) {
      float a = 0.0f;
      for (int b = 0; b < G; ++b) a += cl.map_shared_rank(ls, b)[S];
      loss[st / nb] = a / float(B);
    }
    cl.sync();
  }
  for (int p = p0 + tid; p < p1; p += NT) {
    w[p] = *slot(p);
    gm1[p] = m1[p - p0];
    gm2[p] = m2[p - p0];
  }
}

// Sum of the G partial gradients in block order (thread per parameter),
// then, if adam, the Adam update of that parameter in the same thread.
__global__ void mlp_reduce_partials(const float* __restrict__ gpart, int G, int np, int B, const float* lpart,
                                    float* g, float* loss, bool adam, float* w, float* m1, float* m2, float lr,
                                    float b1, float b2, float b1t, float b2t) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < np) {
    float a = 0.0f;
    for (int b = 0; b < G; ++b) a += gpart[size_t(b) * np + p];
    g[p] = a;
    if (adam) {
      m1[p] = b1 * m1[p] + (1.0f - b1) * a;
      m2[p] = b2 * m2[p] + (1.0f - b2) * a * a;
      const float mh = m1[p] / (1.0f - b1t), vh = m2[p] / (1.0f - b2t);
      w[p] -= lr * mh / (sqrtf(vh) + 1e-8f);
    }
  }
  if (p == 0) {
    float a = 0.0f;
    for (int b = 0; b < G; ++b) a += lpart[b];
    *loss = a / float(B);
  }
}

// Per-column mean and sample deviation of X (n x ncol, row-major) in FP64,
// one block per column; column ncol of the output is the target vector t
// (its mean only).  stats[2c] = mean, stats[2c+1] = deviation.
__global__ void __launch_bounds__(256) column_stats(const float* __restrict__ X, int n, int ncol,
                                                    const float* __restrict__ t, double* stats) {
  const int c = blockIdx.x;
  double s = 0, s2 = 0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const double v = c < ncol ? double(X[size_t(i) * ncol + c]) : double(t[i]);
    s += v;
    s2 += v * v;
  }
  __shared__ double rs[256], rs2[256];
  rs[threadIdx.x] = s;
  rs2[threadIdx.x] = s2;
  __syncthreads();
  for (int h = blockDim.x / 2; h > 0; h >>= 1) {
    if (threadIdx.x < h) {
      rs[threadIdx.x] += rs[threadIdx.x + h];
      rs2[threadIdx.x] += rs2[threadIdx.x + h];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double mean = rs[0] / n;
    const double var = n > 1 ? fmax(rs2[0] - n * mean * mean, 0.0) / (n - 1) : 0.0;
    stats[2 * c] = mean;
    stats[2 * c + 1] = sqrt(var);
  }
}

// Xs = (X - mean) / max(deviation, floor), column by column.
__global__ void standardise(const float* __restrict__ X, int n, int ncol, const double* __restrict__ stats,
                            double floor_sd, float* __restrict__ Xs) {
  const size_t k = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (k >= size_t(n) * ncol) return;
  const int c = int(k % ncol);
  Xs[k] = float((double(X[k]) - stats[2 * c]) / fmax(stats[2 * c + 1], floor_sd));
}

// Inference: a block of 256 threads takes four samples at a time, one
// thread per hidden unit; the weights are staged in shared memory with W1
// and W2 transposed and rows padded to 65 floats, so that staging writes and
// the per-unit reads are free of bank conflicts.  Output y (if y) and
// eps = clamp(10^y, lo, hi), non-finite -> fallback (if eps).
constexpr int MLP_HP = MLP_NH + 1;
__host__ __device__ inline size_t infer_smem(int nin) {
  return size_t(nin * MLP_HP + MLP_NH * MLP_HP + 3 * MLP_NH + 1 + 4 * nin + 4 * MLP_NH + 8) * 4;
}
__global__ void __launch_bounds__(256) mlp_infer(const float* __restrict__ w, int nin, const float* __restrict__ X, int n,
                                                 float* y, double lo, double hi, double fallback, double* eps) {
  extern __shared__ float sw[];
  constexpr int H = MLP_NH, HP = MLP_HP;
  float* W1T = sw;              // [nin][HP]
  float* W2T = W1T + nin * HP;  // [H][HP]
  float* bb = W2T + H * HP;     // b1[H], b2[H], W3[H], b3
  float* xs = bb + 3 * H + 1;   // [4][nin]
  float* a1 = xs + 4 * nin;     // [4][H]
  float* part = a1 + 4 * H;     // [4][2]
  const float* gW1 = w;
  const float* gb1 = gW1 + H * nin;
  const float* gW2 = gb1 + H;
  const float* gb2 = gW2 + H * H;
  const float* gW3 = gb2 + H;
  const float* gb3 = gW3 + H;
  const int t = threadIdx.x;
  for (int q = t; q < H * nin; q += blockDim.x) {
    const int j = q / nin, i = q - j * nin;
    W1T[i * HP + j] = gW1[q];
  }
  for (int q = t; q < H * H; q += blockDim.x) {
    const int j = q / H, i = q - j * H;
    W2T[i * HP + j] = gW2[q];
  }
  for (int q = t; q < H; q += blockDim.x) {
    bb[q] = gb1[q];
    bb[H + q] = gb2[q];
    bb[2 * H + q] = gW3[q];
  }
  if (t == 0) bb[3 * H] = gb3[0];
  const int g = t / H, j = t - g * H;
  for (int s0 = blockIdx.x * 4; s0 < n; s0 += gridDim.x * 4) {
    __syncthreads();
    for (int q = t; q < 4 * nin; q += blockDim.x) {
      const int gg = q / nin;
      xs[q] = s0 + gg < n ? X[size_t(s0 + gg) * nin + (q - gg * nin)] : 0.0f;
    }
    __syncthreads();
    float h1 = bb[j];
    for (int i = 0; i < nin; ++i) h1 += W1T[i * HP + j] * xs[g * nin + i];
    a1[g * H + j] = gelu(h1);
    __syncthreads();
    float h2 = bb[H + j];
    for (int i = 0; i < H; ++i) h2 += W2T[i * HP + j] * a1[g * H + i];
    float c = bb[2 * H + j] * gelu(h2);
    for (int o = 16; o >= 1; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
    if ((t & 31) == 0) part[t >> 5] = c;
    __syncthreads();
    const int s = s0 + g;
    if (j == 0 && s < n) {
      const float out = bb[3 * H] + (part[2 * g] + part[2 * g + 1]);
      if (y) y[s] = out;
      if (eps) {
        double e = pow(10.0, double(out));
        if (!isfinite(e)) e = fallback;
        eps[s] = e < lo ? lo : (e > hi ? hi : e);
      }
    }
  }
}

cudaError_t launch_infer(const float* w, int nin, const float* X, int n, float* y, double lo, double hi,
                         double fallback, double* eps, cudaStream_t st) {
  const int blocks = std::min((n + 3) / 4, 304);
  mlp_infer<<<blocks, 256, infer_smem(nin), st>>>(w, nin, X, n, y, lo, hi, fallback, eps);
  return cudaGetLastError();
}

}  // namespace

struct wcs_mlp {
  int nin = 8;
  float* w = nullptr;
  float* wt = nullptr;  // the step kernel's layout: W1 and W2 transposed
  float* m1 = nullptr;
  float* m2 = nullptr;
  float* g = nullptr;
  float* loss = nullptr;
  int64_t adam_t = 0;
  std::string err;
};

namespace {
// Rebuilds the kernel-layout copy from host weights w (parameter order).
cudaError_t upload_kernel_layout(wcs_mlp* m, const float* w) {
  const int H = MLP_NH, nin = m->nin;
  std::vector<float> t(nparam(nin));
  for (int j = 0; j < H; ++j)
    for (int i = 0; i < nin; ++i) t[i * H + j] = w[j * nin + i];
  const float* b1 = w + H * nin;
  const float* W2 = b1 + H;
  float* tb1 = t.data() + H * nin;
  float* tW2 = tb1 + H;
  for (int j = 0; j < H; ++j) tb1[j] = b1[j];
  for (int j = 0; j < H; ++j)
    for (int i = 0; i < H; ++i) tW2[i * H + j] = W2[j * H + i];
  const int rest = H + H + 1;  // b2, W3, b3 unchanged
  std::memcpy(tW2 + H * H, W2 + H * H, rest * sizeof(float));
  return cudaMemcpy(m->wt, t.data(), t.size() * 4, cudaMemcpyHostToDevice);
}
}  // namespace

namespace wcs {
const float* mlp_kernel_weights(const wcs_mlp* m) { return m ? m->wt : nullptr; }
int mlp_nin(const wcs_mlp* m) { return m ? m->nin : 0; }
}  // namespace wcs

extern "C" {

wcs_status wcs_features_labels(const float* dense_dev, int nfields, int64_t nx, int64_t ny, int wavelet, int patch,
                               int levels, double delta, float* feat_dev, float* label_dev, void* stream) {
  if (!dense_dev || nfields <= 0 || patch <= 0 || levels <= 0 || levels > 8 || nx % patch || ny % patch || !feat_dev ||
      !label_dev)
    return WCS_E_ARG;
  if (wavelet != WCS_BL53 && wavelet != WCS_HAAR) return WCS_E_UNSUPPORTED;  // features of BL5/3 and Haar patches
  const int E = wavelet == WCS_BL53 ? patch + 1 : patch;
  const size_t smem = (3 * size_t(E) * E + 256) * sizeof(double);
  double grid[EPS_N];
  for (int k = 0; k < EPS_N; ++k) grid[k] = std::pow(10.0, -7.0 + k / 8.0);
  if (cudaMemcpyToSymbol(c_eps_grid, grid, sizeof(grid)) != cudaSuccess) return WCS_E_CUDA;
  if (smem > 232448) return WCS_E_UNSUPPORTED;
  if (cudaFuncSetAttribute(features_labels, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)) != cudaSuccess)
    return WCS_E_CUDA;
  // lines in registers for the step kernels' sizes, when the fields'
  // coefficients fit beside the work space (nine 65^2 fields do)
  if (wavelet == WCS_BL53 && nx > 0 && ny > 0) {
    const cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (patch == 64 && levels == 4 && FlCfg<64, 4>::smem(nfields) <= 232448)
      return run_features_labels_reg<64, 4>(dense_dev, nfields, nx, ny, delta, feat_dev, label_dev, st) == cudaSuccess
                 ? WCS_OK : WCS_E_CUDA;
    if (patch == 32 && levels == 3 && FlCfg<32, 3>::smem(nfields) <= 232448)
      return run_features_labels_reg<32, 3>(dense_dev, nfields, nx, ny, delta, feat_dev, label_dev, st) == cudaSuccess
                 ? WCS_OK : WCS_E_CUDA;
  }
  const int npx = int(nx / patch), npy = int(ny / patch);
  features_labels<<<npx * npy, 256, smem, static_cast<cudaStream_t>(stream)>>>(
      dense_dev, nfields, int(nx), int(ny), npx, patch, levels, wavelet, delta, feat_dev, label_dev);
  return cudaGetLastError() == cudaSuccess ? WCS_OK : WCS_E_CUDA;
}

wcs_status wcs_features_labels3(const float* dense_dev, int nfields, int64_t nx, int64_t ny, int64_t nz, int patch,
                                int levels, double delta, float* feat_dev, float* label_dev, void* stream) {
  if (!dense_dev || nfields <= 0 || !feat_dev || !label_dev || patch <= 0 || nx <= 0 || ny <= 0 || nz <= 0 ||
      nx % patch || ny % patch || nz % patch)
    return WCS_E_ARG;
  double grid[EPS_N];
  for (int k = 0; k < EPS_N; ++k) grid[k] = std::pow(10.0, -7.0 + k / 8.0);
  if (cudaMemcpyToSymbol(c_eps_grid, grid, sizeof(grid)) != cudaSuccess) return WCS_E_CUDA;
  const cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (patch == 32 && levels == 3) return run_features_labels3<32, 3>(dense_dev, nfields, nx, ny, nz, delta, feat_dev, label_dev, st);
  if (patch == 16 && levels == 3) return run_features_labels3<16, 3>(dense_dev, nfields, nx, ny, nz, delta, feat_dev, label_dev, st);
  return WCS_E_UNSUPPORTED;
}

wcs_status wcs_mlp_create(int nin, wcs_mlp** out) {
  if (!out || nin <= 0 || nin > MLP_MAXIN) return WCS_E_ARG;
  wcs_mlp* m = new wcs_mlp();
  m->nin = nin;
  const int np = nparam(nin);
  if (cudaMalloc(&m->w, np * 4) != cudaSuccess || cudaMalloc(&m->wt, np * 4) != cudaSuccess ||
      cudaMalloc(&m->m1, np * 4) != cudaSuccess ||
      cudaMalloc(&m->m2, np * 4) != cudaSuccess || cudaMalloc(&m->g, np * 4) != cudaSuccess ||
      cudaMalloc(&m->loss, 4) != cudaSuccess) {
    cudaGetLastError();
    wcs_mlp_destroy(m);
    return WCS_E_OOM;
  }
  cudaMemset(m->w, 0, np * 4);
  cudaMemset(m->wt, 0, np * 4);
  cudaMemset(m->m1, 0, np * 4);
  cudaMemset(m->m2, 0, np * 4);
  *out = m;
  return WCS_OK;
}

void wcs_mlp_destroy(wcs_mlp* m) {
  if (!m) return;
  cudaDeviceSynchronize();
  cudaFree(m->w);
  cudaFree(m->wt);
  cudaFree(m->m1);
  cudaFree(m->m2);
  cudaFree(m->g);
  cudaFree(m->loss);
  delete m;
}

int wcs_mlp_nparam(const wcs_mlp* m) { return m ? nparam(m->nin) : -1; }

wcs_status wcs_mlp_set_weights(wcs_mlp* m, const float* w_host) {
  if (!m || !w_host) return WCS_E_ARG;
  m->adam_t = 0;
  const int np = nparam(m->nin);
  cudaMemset(m->m1, 0, np * 4);
  cudaMemset(m->m2, 0, np * 4);
  if (cudaMemcpy(m->w, w_host, np * 4, cudaMemcpyHostToDevice) != cudaSuccess) return WCS_E_CUDA;
  return upload_kernel_layout(m, w_host) == cudaSuccess ? WCS_OK : WCS_E_CUDA;
}

wcs_status wcs_mlp_get_weights(const wcs_mlp* m, float* w_host) {
  if (!m || !w_host) return WCS_E_ARG;
  return cudaMemcpy(w_host, m->w, nparam(m->nin) * 4, cudaMemcpyDeviceToHost) == cudaSuccess ? WCS_OK : WCS_E_CUDA;
}

// Loss and gradient of the mean squared error on n samples (device X [n][nin]
// and t [n]); gradient to host.
wcs_status wcs_mlp_grad(wcs_mlp* m, const float* X_dev, const float* t_dev, int n, float* grad_host, float* loss_host) {
  if (!m || !X_dev || !t_dev || n <= 0) return WCS_E_ARG;
  const int np = nparam(m->nin), G = (n + MLP_SPB - 1) / MLP_SPB;
  float *gp = nullptr, *lp = nullptr;
  if (cudaMalloc(&gp, size_t(G) * np * 4) != cudaSuccess || cudaMalloc(&lp, size_t(G) * 4) != cudaSuccess) {
    cudaGetLastError();
    cudaFree(gp);
    return WCS_E_OOM;
  }
  const size_t sm = block_grads_smem(m->nin);
  cudaError_t e = cudaFuncSetAttribute(mlp_block_grads, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sm));
  if (e == cudaSuccess) {
    mlp_block_grads<<<G, 256, sm>>>(m->w, m->nin, X_dev, t_dev, nullptr, n, gp, lp);
    mlp_reduce_partials<<<(np + 255) / 256, 256>>>(gp, G, np, n, lp, m->g, m->loss, false, nullptr, nullptr, nullptr,
                                                   0.f, 0.f, 0.f, 0.f, 0.f);
    e = cudaDeviceSynchronize();
  }
  if (e == cudaSuccess && grad_host) e = cudaMemcpy(grad_host, m->g, np * 4, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess && loss_host) e = cudaMemcpy(loss_host, m->loss, 4, cudaMemcpyDeviceToHost);
  cudaFree(gp);
  cudaFree(lp);
  return e == cudaSuccess ? WCS_OK : WCS_E_CUDA;
}

// Training of minibatches of up to TC_CTAS slices (see mlp_train_cluster).
static wcs_status train_in_cluster(wcs_mlp* m, const float* X_dev, const float* t_dev, int nb, const int* batches_host,
                                   int epochs, int batch, float lr, float* loss_history_host) {
  const int np = nparam(m->nin), steps = epochs * nb;
  const float b1 = 0.9f, b2 = 0.999f;
  std::vector<float2> bt(steps);
  for (int k = 0; k < steps; ++k) bt[k] = make_float2(powf(b1, float(m->adam_t + k + 1)), powf(b2, float(m->adam_t + k + 1)));
  // one allocation: the steps' bias corrections, the minibatches, the losses
  const size_t o_idx = size_t(steps) * 8, o_loss = o_idx + size_t(steps) * batch * 4;
  unsigned char* buf = nullptr;
  if (cudaMalloc(&buf, o_loss + size_t(epochs) * 4) != cudaSuccess) {
    cudaGetLastError();
    return WCS_E_OOM;
  }
  float* loss = reinterpret_cast<float*>(buf + o_loss);
  const size_t sm = tc_smem(m->nin);
  cudaError_t e = cudaMemcpy(buf, bt.data(), size_t(steps) * 8, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(buf + o_idx, batches_host, size_t(steps) * batch * 4, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(mlp_train_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sm));
  if (e == cudaSuccess) {
    mlp_train_cluster<<<TC_CTAS, TC_NT, sm>>>(m->w, m->m1, m->m2, m->nin, X_dev, t_dev, reinterpret_cast<const int*>(buf + o_idx),
                                              steps, nb, batch, lr, b1, b2, reinterpret_cast<const float2*>(buf), loss);
    e = cudaGetLastError();
  }
  m->adam_t += steps;
  std::vector<float> w(np);
  if (e == cudaSuccess) e = cudaMemcpy(w.data(), m->w, size_t(np) * 4, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess && loss_history_host) e = cudaMemcpy(loss_history_host, loss, size_t(epochs) * 4, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = upload_kernel_layout(m, w.data());
  cudaFree(buf);
  return e == cudaSuccess ? WCS_OK : WCS_E_CUDA;
}

// Adam on minibatches; batches[e*nb + b] lists minibatch b of epoch e as
// indices into X / t (host array of epochs * n_batches * batch ints).
wcs_status wcs_mlp_train(wcs_mlp* m, const float* X_dev, const float* t_dev, int n, const int* batches_host, int epochs,
                         int batch, float lr, float* loss_history_host) {
  if (!m || !X_dev || !t_dev || n <= 0 || batch <= 0 || batch > n || epochs <= 0 || !batches_host) return WCS_E_ARG;
  const int np = nparam(m->nin);
  const int nb = n / batch, G = (batch + MLP_SPB - 1) / MLP_SPB;
  const size_t tsm = tc_smem(m->nin);
  // up to eight slices: the whole run in one launch (beyond that a minibatch
  // fills the chip better as a launch of its own)
  if (G <= TC_CTAS && tsm <= 232448 && int64_t(epochs) * nb < (1 << 30)) return train_in_cluster(m, X_dev, t_dev, nb, batches_host, epochs, batch, lr, loss_history_host);
  float *gp = nullptr, *lp = nullptr;
  int* idx = nullptr;
  if (cudaMalloc(&gp, size_t(G) * np * 4) != cudaSuccess || cudaMalloc(&lp, size_t(G) * 4) != cudaSuccess ||
      cudaMalloc(&idx, size_t(epochs) * nb * batch * 4) != cudaSuccess) {
    cudaGetLastError();
    cudaFree(gp);
    cudaFree(lp);
    return WCS_E_OOM;
  }
  cudaError_t e = cudaMemcpy(idx, batches_host, size_t(epochs) * nb * batch * 4, cudaMemcpyHostToDevice);
  const size_t sm = block_grads_smem(m->nin);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(mlp_block_grads, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sm));
  const float b1 = 0.9f, b2 = 0.999f;
  for (int ep = 0; ep < epochs && e == cudaSuccess; ++ep) {
    for (int b = 0; b < nb && e == cudaSuccess; ++b) {
      mlp_block_grads<<<G, 256, sm>>>(m->w, m->nin, X_dev, t_dev, idx + (size_t(ep) * nb + b) * batch, batch, gp, lp);
      ++m->adam_t;
      mlp_reduce_partials<<<(np + 255) / 256, 256>>>(gp, G, np, batch, lp, m->g, m->loss, true, m->w, m->m1, m->m2, lr,
                                                     b1, b2, powf(b1, float(m->adam_t)), powf(b2, float(m->adam_t)));
      e = cudaGetLastError();
    }
    if (e == cudaSuccess && loss_history_host) e = cudaMemcpy(loss_history_host + ep, m->loss, 4, cudaMemcpyDeviceToHost);
  }
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e == cudaSuccess) {
    std::vector<float> w(np);
    e = cudaMemcpy(w.data(), m->w, np * 4, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = upload_kernel_layout(m, w.data());
  }
  cudaFree(gp);
  cudaFree(lp);
  cudaFree(idx);
  return e == cudaSuccess ? WCS_OK : WCS_E_CUDA;
}

wcs_status wcs_mlp_fit(wcs_mlp* m, const float* X_dev, const float* t_dev, int n, const int* batches_host, int epochs,
                       int batch, float lr, double sd_floor, float* loss_history_host, double* stats_host) {
  if (!m || !X_dev || !t_dev || n <= 1 || batch <= 0 || batch > n || epochs <= 0 || !batches_host || !(sd_floor > 0))
    return WCS_E_ARG;
  const int nin = m->nin, np = nparam(nin);
  double* st = nullptr;
  float* Xs = nullptr;
  if (cudaMalloc(&st, size_t(2) * (nin + 1) * 8) != cudaSuccess ||
      cudaMalloc(&Xs, size_t(n) * nin * 4) != cudaSuccess) {
    cudaGetLastError();
    cudaFree(st);
    return WCS_E_OOM;
  }
  column_stats<<<nin + 1, 256>>>(X_dev, n, nin, t_dev, st);
  const size_t tot = size_t(n) * nin;
  standardise<<<unsigned((tot + 255) / 256), 256>>>(X_dev, n, nin, st, sd_floor, Xs);
  std::vector<double> s(2 * (nin + 1));
  std::vector<float> w(np);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpy(s.data(), st, s.size() * 8, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(w.data(), m->w, np * 4, cudaMemcpyDeviceToHost);
  wcs_status r = WCS_E_CUDA;
  if (e == cudaSuccess) {
    w[np - 1] = float(s[2 * nin]);  // the output bias starts at the mean target
    if (wcs_mlp_set_weights(m, w.data()) == WCS_OK)  // also restarts Adam
      r = wcs_mlp_train(m, Xs, t_dev, n, batches_host, epochs, batch, lr, loss_history_host);
  }
  if (r == WCS_OK && cudaMemcpy(w.data(), m->w, np * 4, cudaMemcpyDeviceToHost) == cudaSuccess) {
    // fold the standardisation into the first layer: W1 x' + b1 with
    // x' = (x - mean) / sd equals (W1 / sd) x + (b1 - (W1 / sd) mean)
    for (int h = 0; h < MLP_NH; ++h) {
      double b = w[MLP_NH * nin + h];
      for (int c = 0; c < nin; ++c) {
        const double wf = double(w[h * nin + c]) / std::max(s[2 * c + 1], sd_floor);
        b -= wf * s[2 * c];
        w[h * nin + c] = float(wf);
      }
      w[MLP_NH * nin + h] = float(b);
    }
    r = wcs_mlp_set_weights(m, w.data());
  } else if (r == WCS_OK) {
    r = WCS_E_CUDA;
  }
  if (stats_host) std::copy(s.begin(), s.end(), stats_host);
  cudaFree(st);
  cudaFree(Xs);
  return r;
}

wcs_status wcs_mlp_forward(wcs_mlp* m, const float* X_dev, int n, float* y_dev) {
  if (!m || !X_dev || !y_dev || n <= 0) return WCS_E_ARG;
  return launch_infer(m->w, m->nin, X_dev, n, y_dev, 0, 0, 0, nullptr, nullptr) == cudaSuccess ? WCS_OK : WCS_E_CUDA;
}

// Used by the simulation: per-patch eps from per-patch features.
wcs_status wcs_mlp_eps(wcs_mlp* m, const float* feat_dev, int n, double lo, double hi, double fallback, double* eps_dev,
                       void* stream) {
  if (!m || !feat_dev || !eps_dev || n <= 0) return WCS_E_ARG;
  return launch_infer(m->w, m->nin, feat_dev, n, nullptr, lo, hi, fallback, eps_dev, static_cast<cudaStream_t>(stream)) ==
                 cudaSuccess
             ? WCS_OK
             : WCS_E_CUDA;
}

}  // extern "C"
