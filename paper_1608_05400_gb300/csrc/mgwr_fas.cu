// Waveform relaxation FAS for the 1-D nonlinear problem of Sec. 7
// (Eq. anomalous_diffusion): D_t^alpha u = d/dx(D(u) du/dx) + c du/dx + f on
// (0,1) x (0,T], zero boundary and initial values, discretised with the L1
// scheme (Eq. L1_scheme2), the conservative flux difference of
// Eq. spatial_discretization (a_{n+-1/2} the mean of D at the two nodes) and
// upwind convection (forward difference for c >= 0, backward for c < 0).
//
// Kernels (FP64):
//   k_fas_line   the nonlinear red-black waveform smoother: one warp per time line
//                of one colour; the line is marched in time, each step a scalar
//                Newton solve (the step's equation is strictly increasing in the
//                unknown), the history sum of the L1 matrix shared by the warp's
//                lanes from a shared-memory copy of the line;
//   k_fas_apply  out = base + sign * N_h(u), N_h the discrete operator (time term
//                T_M u by direct sums from shared memory, flux and upwind
//                differences), with its max-norm: the defect f - N_h(u) and the
//                FAS coarse right-hand side N_2h(R u) + R r;
//   k_fas_restrict2, k_fas_correct   full weighting of the iterate and the
//                defect, and u += P (u_c - R u).
// The history sums are direct (O(M^2) per line, as the scheme is written):
// the paper's nonlinear tables use M <= 256, and M is limited to 1024 here, so
// both kernels stay within the default 48 KB of dynamic shared memory.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <cfloat>
#include <cmath>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "mgwr.h"
#include "mgwr_common.cuh"

namespace mgwr {
namespace {

constexpr int kFasMaxM = 1024;
constexpr int kLineWarps = 4;     // time lines per block of k_fas_line
constexpr int kApplyThreads = 256;
constexpr int kNewtonMax = 100;   // Newton iterations per time step before giving up

__device__ __forceinline__ double coef_D(int kind, double v) {
  return kind == MGWR_FAS_D_POROUS ? 1.0 + v * v : 1.0;
}


// Lines of one colour: points i = 2k + parity (k < count), or every point when
// all_points (the one-point grid).  Dynamic shared memory: (1 + kLineWarps) * M
// doubles.  status bit 0 is set when Newton's method did not settle in a step.
__global__ void __launch_bounds__(32 * kLineWarps)
    k_fas_line(double* __restrict__ u, const double* __restrict__ f,
               const double* __restrict__ r, int n, int M, double h, double c, int coef,
               int parity, int all_points, int* __restrict__ status) {
  extern __shared__ double sm[];
  double* rs = sm;  // r_1..r_M of T_M
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double* line = sm + M + (size_t)warp * M;
  for (int j = threadIdx.x; j < M; j += blockDim.x) rs[j] = r[j];
  const int count = all_points ? n : (parity ? n / 2 : (n + 1) / 2);
  const int k = blockIdx.x * kLineWarps + warp;
  const bool active = k < count;
  const int i = all_points ? k : 2 * k + parity;
  if (active)
    for (int j = lane; j < M; j += 32) line[j] = u[(size_t)i * M + j];
  __syncthreads();
  if (!active) return;
  const double* up = (i + 1 < n) ? u + (size_t)(i + 1) * M : nullptr;
  const double* um = (i > 0) ? u + (size_t)(i - 1) * M : nullptr;
  const double* fi = f + (size_t)i * M;
  const double r1 = rs[0], h2 = h * h, half_h2 = 0.5 / h2, c_h = c / h, ac_h = fabs(c_h);
  const double kappa = coef == MGWR_FAS_D_POROUS ? 1.0 : 0.0;  // D(v) = 1 + kappa v^2
  // per-line constants (no FP64 division inside the time loop)
  const double a3 = kappa / h2, a3x3 = 3.0 * a3;
  bool ok = true;
  for (int m = 0; m < M; ++m) {
    // sum_{j<m} (T_M)_{mj} u_j, (T_M)_{mj} = r_{m-j+1}
    double part = 0.0;
    for (int j = lane; j < m; j += 32) part = fma(rs[m - j], line[j], part);
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    const double hist = __shfl_sync(0xffffffffu, part, 0);
    const double P = up ? up[m] : 0.0, Q = um ? um[m] : 0.0;
    const double Dp = 1.0 + kappa * P * P, Dm = 1.0 + kappa * Q * Q, fm = fi[m];
    // The step's equation g(v) = r_1 v + hist - diffusion(v) - convection(v) - f = 0
    // as the cubic a0 + a1 v + a2 v^2 + a3 v^3: with D(v) = 1 + kappa v^2,
    //   2 h^2 diffusion = (Dp+1) P + (Dm+1) Q - (Dp+Dm+2) v + kappa (P+Q) v^2 - 2 kappa v^3.
    const double flux0 = ((Dp + 1.0) * P + (Dm + 1.0) * Q) * half_h2;
    const double conv0 = c >= 0.0 ? c_h * P : -c_h * Q;
    const double a2 = -kappa * (P + Q) * half_h2, a2x2 = 2.0 * a2;
    const double a1 = r1 + (Dp + Dm + 2.0) * half_h2 + ac_h;
    const double a0 = hist - fm - flux0 - conv0;
    // the size of the equation's terms, in units of v (a tolerance scale only, so the
    // FP32 reciprocal of a1 is accurate enough)
    const double s0 =
        (fabs(hist) + fabs(fm) + fabs(flux0) + fabs(conv0)) * (double)(1.0f / (float)a1);
    // Newton's method in FP32 to about 1e-6, then two FP64 Newton steps with the
    // FP32 reciprocal of g' (each contracts the error by about 1e-7)
    const float b0 = (float)a0, b1 = (float)a1, b2 = (float)a2, b3 = (float)a3;
    const float s0f = (float)s0;
    float vf = (float)line[m];
    for (int it = 0; it < 30; ++it) {
      const float gf = fmaf(fmaf(fmaf(b3, vf, b2), vf, b1), vf, b0);
      const float dgf = fmaf(fmaf(3.0f * b3, vf, 2.0f * b2), vf, b1);
      const float sf = gf / dgf;
      vf -= sf;
      if (fabsf(sf) <= 1e-6f * (fabsf(vf) + s0f)) break;
    }
    double v = isfinite(vf) ? (double)vf : line[m];
    double step = 0.0;
    for (int k = 0; k < 2; ++k) {
      const double g = fma(fma(fma(a3, v, a2), v, a1), v, a0);
      const double dg = fma(fma(a3x3, v, a2x2), v, a1);
      const float dgs = fabsf((float)dg);
      if (!(dgs >= FLT_MIN && dgs <= FLT_MAX)) {
        // g' outside FP32's normal range: its FP32 reciprocal would be 0 or inf,
        // so leave the step to the plain FP64 Newton solve below
        step = NAN;
        break;
      }
      step = g * (double)(1.0f / (float)dg);
      v -= step;
    }
    if (!(fabs(step) <= 1e-12 * (fabs(v) + s0) + 1e-300)) {
      // not settled (extreme or non-finite data): plain FP64 Newton from the start
      v = line[m];
      bool done = false, settled = false;
      for (int it = 0; it < kNewtonMax; ++it) {
        const double g = fma(fma(fma(a3, v, a2), v, a1), v, a0);
        const double dg = fma(fma(a3x3, v, a2x2), v, a1);
        step = g / dg;
        v -= step;
        if (done) {
          settled = true;
          break;
        }
        done = fabs(step) <= 1e-13 * (fabs(v) + s0) + 1e-300;
      }
      if (!settled) ok = false;
    }
    __syncwarp();
    if (lane == 0) line[m] = v;
    __syncwarp();
  }
  for (int j = lane; j < M; j += 32) u[(size_t)i * M + j] = line[j];
  if (!ok && lane == 0) atomicOr(status, 1);
}

// The same half-sweep as k_fas_line by a whole-line fixed point instead of a
// march in time: with the splitting N(v) = (T_M + sigma I) v - (sigma v - phi(v)),
// phi the point's spatial term (flux difference and upwind convection with its
// neighbours' lines fixed), sigma = 2/h^2 + |c|/h the spatial term's slope at
// D = 1, every iteration is
//     v <- (T_M + sigma I)^{-1} (f + sigma v - phi(v)),
// one causal convolution per line with the inverse column of T_M + sigma I
// (spectrum kspec) on the FFT engine, two lines per thread group.  For D = 1
// it is the linear smoother (one iteration); otherwise it contracts by about
// max |1 - phi'(v) / sigma| and runs until the largest change of the pair is at
// the convolution's rounding level (4e-15 of its largest value), or stops
// falling below 1e-12 of it, at most max_it times (status bit 1 set when
// neither is reached).  One line pair per block of L/8 threads (E = 1).
template <int BLOCK>
__global__ void __launch_bounds__(BLOCK)
    k_fas_fixed(double* __restrict__ u, const double* __restrict__ f,
                const Cx<double>* __restrict__ kspec, const Cx<double>* __restrict__ tw, int n,
                int M, int logL, double hinv, double hinv2, double c, double sigma, int coef,
                int parity, int all_points, int max_it, int* __restrict__ status,
                unsigned long long* __restrict__ iterations) {
  extern __shared__ unsigned char smem_raw[];
  __shared__ double red[2][BLOCK / 32 > 0 ? BLOCK / 32 : 1];
  __shared__ int done_flag;
  Cx<double>* buf = reinterpret_cast<Cx<double>*>(smem_raw);
  const FftShape sh(logL);
  const int t = threadIdx.x;
  const GroupSync sync(BLOCK, BLOCK, 0);
  const int count = all_points ? n : (parity ? n / 2 : (n + 1) / 2);
  const int kA = 2 * blockIdx.x, kB = kA + 1;
  const bool hasB = kB < count;
  const int iA = all_points ? kA : 2 * kA + parity;
  const int iB = all_points ? kB : 2 * kB + parity;
  double* uA = u + (size_t)iA * M;
  double* uB = u + (size_t)(hasB ? iB : iA) * M;
  const double* fA = f + (size_t)iA * M;
  const double* fB = f + (size_t)(hasB ? iB : iA) * M;
  // neighbour lines (the other colour, fixed in this half-sweep); none on the one-point grid
  const double* pA = (!all_points && iA + 1 < n) ? u + (size_t)(iA + 1) * M : nullptr;
  const double* qA = (!all_points && iA > 0) ? u + (size_t)(iA - 1) * M : nullptr;
  const double* pB = (!all_points && iB + 1 < n) ? u + (size_t)(iB + 1) * M : nullptr;
  const double* qB = (!all_points && iB > 0) ? u + (size_t)(iB - 1) * M : nullptr;
  // f + sigma v - phi(v) at one point: phi(v) = -(diffusion + convection)
  auto rhs = [&](double fm, double v, double P, double Q) {
    const double D0 = coef_D(coef, v);
    const double a_plus = 0.5 * (coef_D(coef, P) + D0);
    const double a_minus = 0.5 * (coef_D(coef, Q) + D0);
    const double diffusion = (a_plus * (P - v) - a_minus * (v - Q)) * hinv2;
    const double convection = c >= 0.0 ? c * (P - v) * hinv : c * (v - Q) * hinv;
    return fm + sigma * v + (diffusion + convection);
  };
  auto load = [&](int m) -> Cx<double> {
    const double bA = rhs(fA[m], uA[m], pA ? pA[m] : 0.0, qA ? qA[m] : 0.0);
    const double bB = hasB ? rhs(fB[m], uB[m], pB ? pB[m] : 0.0, qB ? qB[m] : 0.0) : 0.0;
    return Cx<double>{bA, bB};
  };
  bool settled = false;
  int it = 0;
  double d_prev = 0.0;  // the last iteration's largest change (thread 0)
  for (; it < max_it; ++it) {
    double dmax = 0.0, vmax = 0.0;
    auto store = [&](int m, Cx<double> y) {
      dmax = fmax(dmax, fabs(y.x - uA[m]));
      vmax = fmax(vmax, fabs(y.x));
      uA[m] = y.x;
      if (hasB) {
        dmax = fmax(dmax, fabs(y.y - uB[m]));
        vmax = fmax(vmax, fabs(y.y));
        uB[m] = y.y;
      }
    };
    Cx<double> v[1][8];
    fft_forward<1>(buf, t, sh, tw, load, v, sync);
#pragma unroll
    for (int q = 0; q < 8; ++q) v[0][q] = cmul(v[0][q], kspec[8 * t + q]);
    fft_inverse<1>(buf, t, sh, tw, v, store, sync);
    // the pair's largest change and value (non-finite values count as not settled)
    for (int o = 16; o > 0; o >>= 1) {
      dmax = fmax(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
      vmax = fmax(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
    }
    if (BLOCK >= 32 && (t & 31) == 0) {
      red[0][t >> 5] = dmax;
      red[1][t >> 5] = vmax;
    }
    __syncthreads();
    if (t == 0) {
      double d = 0.0, w = 0.0;
      for (int k = 0; k < (BLOCK >= 32 ? BLOCK / 32 : 1); ++k) {
        d = fmax(d, BLOCK >= 32 ? red[0][k] : dmax);
        w = fmax(w, BLOCK >= 32 ? red[1][k] : vmax);
      }
      // settled: the change is at the level of the convolution's rounding (the
      // right-hand side holds sigma v, so v carries about log2(L) eps of itself),
      // or it has stopped falling within 1e-12 of the line
      done_flag = (w <= DBL_MAX && (d <= 4e-15 * w || (d <= 1e-12 * w && d >= 0.5 * d_prev))) ? 1 : 0;
      d_prev = d;
    }
    __syncthreads();  // also orders this iteration's stores before the next loads
    if (done_flag) {
      settled = true;
      ++it;
      break;
    }
  }
  if (t == 0) {
    if (!settled) atomicOr(status, 2);
    atomicAdd(iterations, (unsigned long long)it * (hasB ? 2 : 1));  // line iterations
  }
}

// k_fas_fixed's iteration with the convolution as FP64 sums, one line per cluster
// of C blocks of M threads.  The transform of a pair costs about 78 M clocks of one
// SM's FP64 pipe and runs on as many SMs as there are pairs (coarse levels: a few);
// the sums cost M^2 / 4 clocks of it and spread over the cluster, M^2 / (4 C).
// Block `rank` owns the steps t = rank mod C (equal shares of the triangle): it forms
// their right-hand sides and hands them to the cluster's other blocks through
// distributed shared memory (two buffers, one cluster barrier an iteration, one before
// the first store, split so that it spans the loads), then sums its outputs with C
// threads each.  Settled per line by k_fas_fixed's rule; the
// largest change and value travel with the next iteration's right-hand sides, so
// that all blocks decide alike.  With the neighbours fixed the right-hand side
// f + sigma v - phi(v) is a cubic in v whose sigma terms cancel: three operations.
// M = 256, one half-sweep of the 255-point grid: 59 us
// against 106; the coarser levels 41 .. 25 us.
template <int C>
__global__ void __cluster_dims__(C, 1, 1) __launch_bounds__(1024)
    k_fas_fixed_sums(double* __restrict__ u, const double* __restrict__ f,
                     const double* __restrict__ kcol, int n, int M, double hinv, double hinv2,
                     double c, int coef, int parity, int all_points, int max_it,
                     int* __restrict__ status, unsigned long long* __restrict__ iterations) {
  namespace cg = cooperative_groups;
  extern __shared__ double sums_sm[];
  // per buffer and rank: largest change, largest value (bits of non-negative doubles,
  // which order like them; compared as integers, off the FP64 pipe)
  __shared__ unsigned long long most[2][C][2];
  __shared__ unsigned long long red[2][32];
  const cg::cluster_group cluster = cg::this_cluster();
  // Another block's shared memory may be written only once that block runs: every
  // block arrives here, and waits for the others before its first such store.
  if (C > 1) cluster.barrier_arrive();
  const int rank = C == 1 ? 0 : (int)cluster.block_rank();
  double* const sk = sums_sm;          // the inverse column
  double* const sb = sums_sm + M;      // two buffers of right-hand sides
  double* const sv = sums_sm + 3 * M;  // this block's outputs
  const int tid = threadIdx.x;
  const int k = blockIdx.x / C;
  const int i = all_points ? k : 2 * k + parity;
  const int own = M / C;
  const bool owner = tid < own;
  const int t = tid * C + rank;
  double* const line = u + (size_t)i * M;
  double v = 0.0, fm = 0.0, P = 0.0, Q = 0.0;
  if (owner) {
    v = line[t];
    fm = f[(size_t)i * M + t];
    if (!all_points && i + 1 < n) P = line[M + t];
    if (!all_points && i > 0) Q = line[t - M];
  }
  sk[tid] = kcol[tid];
  // b = b0 + b1 v + b2 v^2 + b3 v^3 for D(v) = 1 + kappa v^2
  const double kappa = coef == MGWR_FAS_D_POROUS ? 1.0 : 0.0;
  const double b3 = -kappa * hinv2, b2 = 0.5 * kappa * hinv2 * (P + Q);
  const double b1 = -0.5 * kappa * hinv2 * (P * P + Q * Q);
  const double b0 = fm + (c >= 0.0 ? c * P : -c * Q) * hinv +
                    0.5 * hinv2 * ((2.0 + kappa * P * P) * P + (2.0 + kappa * Q * Q) * Q);
  // magnitude bits, 0 for NaN (as fmax ignores it)
  auto mag = [](double x) {
    const unsigned long long m = (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
    return m > 0x7FF0000000000000ull ? 0ull : m;
  };
  // the output this thread helps to sum
  const int o = tid / C, lane = tid % C, to = o * C + rank;
  bool settled = false;
  double d_prev = 0.0;
  if (C > 1) cluster.barrier_wait();
  int it = 0;
  for (;; ++it) {
    const int buf = it & 1;
    if (owner) {
      const double b = fma(fma(fma(b3, v, b2), v, b1), v, b0);
      for (int r = 0; r < C; ++r)
        (C == 1 ? sb : cluster.map_shared_rank(sb, r))[buf * M + t] = b;
    }
    if (C == 1)
      __syncthreads();
    else
      cluster.sync();
    if (it > 0) {
      unsigned long long dm = 0, wm = 0;
      for (int r = 0; r < C; ++r) {
        dm = max(dm, most[buf][r][0]);
        wm = max(wm, most[buf][r][1]);
      }
      const double d = __longlong_as_double((long long)dm), w = __longlong_as_double((long long)wm);
      settled = w <= DBL_MAX && (d <= 4e-15 * w || (d <= 1e-12 * w && d >= 0.5 * d_prev));
      d_prev = d;
      if (settled || it == max_it) break;
    }
    const double* const b = sb + buf * M;
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    for (int s = lane; s < to; s += 4 * C) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (s + q * C < to) a[q] = fma(sk[to - s - q * C], b[s + q * C], a[q]);
    }
    double y = (a[0] + a[1]) + (a[2] + a[3]);
#pragma unroll
    for (int x = C / 2; x > 0; x >>= 1) y += __shfl_xor_sync(0xffffffffu, y, x);
    y = fma(sk[0], b[to], y);  // the largest product last
    if (lane == 0) sv[o] = y;
    __syncthreads();
    unsigned long long d = 0, w = 0;
    if (owner) {
      const double next = sv[tid];
      d = mag(next - v);
      w = mag(next);
      v = next;
    }
    for (int x = 16; x > 0; x >>= 1) {
      d = max(d, __shfl_xor_sync(0xffffffffu, d, x));
      w = max(w, __shfl_xor_sync(0xffffffffu, w, x));
    }
    if ((tid & 31) == 0) {
      red[0][tid >> 5] = d;
      red[1][tid >> 5] = w;
    }
    __syncthreads();
    if (tid < C) {  // thread r tells rank r
      d = w = 0;
      for (int x = 0; x < (own + 31) / 32; ++x) {
        d = max(d, red[0][x]);
        w = max(w, red[1][x]);
      }
      unsigned long long* const to_rank =
          C == 1 ? &most[0][0][0] : cluster.map_shared_rank(&most[0][0][0], tid);
      to_rank[((buf ^ 1) * C + rank) * 2] = d;
      to_rank[((buf ^ 1) * C + rank) * 2 + 1] = w;
    }
  }
  if (owner) line[t] = v;
  if (tid == 0 && rank == 0) {
    if (!settled) atomicOr(status, 2);
    atomicAdd(iterations, (unsigned long long)it);  // line iterations
  }
}

// out = base + sign * N_h(u) on every point (gridDim.y blocks per line, block y the
// steps y mod gridDim.y: coarse levels have fewer lines than SMs), and the
// max-norm of out into *norm_bits (the bits of a non-negative double; a
// non-finite value counts as +inf).  Eight threads share a history sum; the
// spatial terms are formed by whole warps afterwards.  Dynamic shared memory: 3 * M
// doubles.  h is a power of two, so its reciprocals are exact.  M = 256, mean over the levels: 13 us, 20.7 with
// one block per line and one thread per sum.
__global__ void __launch_bounds__(kApplyThreads)
    k_fas_apply(const double* __restrict__ u, const double* __restrict__ r,
                const double* __restrict__ base, double* __restrict__ out, int n, int M,
                double h, double c, int coef, double sign,
                unsigned long long* __restrict__ norm_bits) {
  extern __shared__ double sm[];
  __shared__ double wmax[kApplyThreads / 32];
  constexpr int kLanes = 8;
  double* rs = sm;
  double* line = sm + M;
  const int i = blockIdx.x;
  const size_t row = (size_t)i * M;
  for (int j = threadIdx.x; j < M; j += blockDim.x) {
    rs[j] = r[j];
    line[j] = u[row + j];
  }
  __syncthreads();
  double* const sums = sm + 2 * M;
  const double hinv = 1.0 / h, hinv2 = hinv * hinv;
  const int lane = threadIdx.x % kLanes;
  const int share = (M - (int)blockIdx.y + (int)gridDim.y - 1) / (int)gridDim.y;
  // whole warps run each pass (the sums end in shuffles)
  for (int o0 = 0; o0 < share; o0 += kApplyThreads / kLanes) {
    const int o = o0 + threadIdx.x / kLanes;
    const int m = o < share ? o * (int)gridDim.y + (int)blockIdx.y : -1;
    double t0 = 0.0, t1 = 0.0;
    for (int j = lane; j <= m; j += 2 * kLanes) {
      t0 = fma(rs[m - j], line[j], t0);
      if (j + kLanes <= m) t1 = fma(rs[m - j - kLanes], line[j + kLanes], t1);
    }
    double t = t0 + t1;
#pragma unroll
    for (int x = kLanes / 2; x > 0; x >>= 1) t += __shfl_xor_sync(0xffffffffu, t, x);
    if (m >= 0 && lane == 0) sums[o] = t;
  }
  __syncthreads();
  double local = 0.0;
  for (int o = threadIdx.x; o < share; o += kApplyThreads) {
    const int m = o * (int)gridDim.y + (int)blockIdx.y;
    const double t = sums[o];
    const double w0 = line[m];
    const double wp = i + 1 < n ? u[row + M + m] : 0.0;
    const double wm = i > 0 ? u[row - M + m] : 0.0;
    const double D0 = coef_D(coef, w0);
    const double a_plus = 0.5 * (coef_D(coef, wp) + D0);
    const double a_minus = 0.5 * (coef_D(coef, wm) + D0);
    const double diffusion = (a_plus * (wp - w0) - a_minus * (w0 - wm)) * hinv2;
    const double convection = c >= 0.0 ? c * (wp - w0) * hinv : c * (w0 - wm) * hinv;
    const double val = base[row + m] + sign * (t - (diffusion + convection));
    out[row + m] = val;
    const double a = fabs(val);
    local = fmax(local, a <= DBL_MAX ? a : (double)INFINITY);
  }
  for (int o = 16; o > 0; o >>= 1) local = fmax(local, __shfl_xor_sync(0xffffffffu, local, o));
  if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = local;
  __syncthreads();
  if (threadIdx.x == 0 && norm_bits != nullptr) {
    double mx = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) mx = fmax(mx, wmax[w]);
    atomicMax(norm_bits, (unsigned long long)__double_as_longlong(mx));
  }
}

// Full weighting (1/4)[1 2 1] of two fine fields (n = 2 nc + 1 lines) at once, the
// first to two places (R u and the coarse iterate that starts from it).
__global__ void k_fas_restrict2(const double* __restrict__ a, double* __restrict__ ac,
                                double* __restrict__ ac2, const double* __restrict__ b,
                                double* __restrict__ bc, int nc, int M) {
  const size_t total = (size_t)nc * M;
  for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total;
       idx += (size_t)gridDim.x * blockDim.x) {
    const size_t J = idx / M, m = idx % M;
    const size_t f0 = 2 * J * M + m;  // fine line 2J, then 2J+1 and 2J+2
    const double x = 0.25 * ((a[f0] + 2.0 * a[f0 + M]) + a[f0 + 2 * M]);
    ac[idx] = x;
    ac2[idx] = x;
    bc[idx] = 0.25 * ((b[f0] + 2.0 * b[f0 + M]) + b[f0 + 2 * M]);
  }
}

// u (n = 2 nc + 1 lines) += P (uc - ubar): fine line 2J+1 takes coarse J, fine
// line 2J the mean of coarse J-1 and J (zero beyond the boundary).
__global__ void k_fas_correct(double* __restrict__ u, const double* __restrict__ uc,
                              const double* __restrict__ ubar, int nc, int M) {
  const int n = 2 * nc + 1;
  const size_t total = (size_t)n * M;
  for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total;
       idx += (size_t)gridDim.x * blockDim.x) {
    const int I = (int)(idx / M);
    const size_t m = idx % M;
    double p;
    if (I & 1) {
      const size_t cj = (size_t)((I - 1) / 2) * M + m;
      p = uc[cj] - ubar[cj];
    } else {
      const int J = I / 2;
      p = 0.0;
      if (J >= 1) p += 0.5 * (uc[(size_t)(J - 1) * M + m] - ubar[(size_t)(J - 1) * M + m]);
      if (J < nc) p += 0.5 * (uc[(size_t)J * M + m] - ubar[(size_t)J * M + m]);
    }
    u[idx] += p;
  }
}

}  // namespace
}  // namespace mgwr

// ---- handle -------------------------------------------------------------------------

using mgwr::Cx;

struct mgwr_fas {
  int n = 0, M = 0, nlev = 0, coef = 0, order = MGWR_ORDER_TEXT;
  double T = 0.0, alpha = 0.0, c = 0.0;
  cudaStream_t stream = nullptr;  // the stream every launch and copy goes to
  cudaStream_t own = nullptr;     // the stream the handle created
  double* r = nullptr;       // r_1..r_M of T_M
  double* dk = nullptr;      // d_0..d_M (written by the coefficient kernel)
  double* params = nullptr;  // alpha, tau^-alpha / Gamma(2 - alpha)
  std::vector<double*> u, f, rr, ubar;  // per level, coarsest first
  unsigned long long* flags = nullptr;  // [0] max-norm bits, [1] line-solve status,
                                        // [2] fixed-point line iterations so far
  // whole-line fixed-point smoother (k_fas_fixed): twiddles, per-level inverse
  // columns of T_M + sigma_l I and their spectra; null when M is not a power of
  // two in 128 .. 1024, where the time march serves
  int smoother = MGWR_FAS_SMOOTHER_AUTO;
  Cx<double>* tw = nullptr;
  double* kcol = nullptr;
  Cx<double>* kspec = nullptr;
  std::vector<double> sigma;
  size_t line_smem = 0, apply_smem = 0;
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;
  // one cycle and the norm of its defect as a CUDA graph (about 45 launches at 255
  // points), captured by the second cycle of a solve, for one set of settings
  cudaGraphExec_t graph = nullptr;
  long long graph_key = -1, graph_kernels = 0;
  std::string err;
};

namespace {

int fas_fail(mgwr_fas_t h, int code, const std::string& msg) {
  if (h != nullptr) h->err = msg;
  return code;
}

int fas_cuda(mgwr_fas_t h, cudaError_t e, const char* what) {
  if (e == cudaSuccess) return MGWR_OK;
  cudaGetLastError();
  return fas_fail(h, MGWR_E_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

inline int level_n(int l) { return (1 << (l + 1)) - 1; }
inline double level_h(int l) { return 1.0 / (double)(level_n(l) + 1); }
inline size_t field_bytes(const mgwr_fas* h, int l) {
  return sizeof(double) * (size_t)level_n(l) * h->M;
}

// red = the colour visited first: 1-D text order odd i, table order even i
inline int colour_parity(const mgwr_fas* h, int colour) {
  const int red = h->order == MGWR_ORDER_TEXT ? 1 : 0;
  return colour == MGWR_RED ? red : 1 - red;
}

bool fixed_point(const mgwr_fas* h) {
  return h->kspec != nullptr && h->smoother != MGWR_FAS_SMOOTHER_MARCH;
}

constexpr int kFixedMaxIt = 200;  // fixed-point iterations per half-sweep before giving up

cudaError_t launch_line(mgwr_fas* h, int l, int parity, int all_points) {
  const int n = level_n(l);
  const int count = all_points ? n : (parity ? n / 2 : (n + 1) / 2);
  if (count == 0) return cudaSuccess;
  if (fixed_point(h)) {
    const int L = 2 * h->M, logL = mgwr::ilog2(L);
    const double hl = level_h(l);
    int* st = reinterpret_cast<int*>(h->flags + 1);
    // blocks per line: as many as keep one line's cluster per SM group
    const int sms = mgwr::sm_count();
    const int C = count * 8 <= sms ? 8 : count * 4 <= sms ? 4 : count * 2 <= sms ? 2 : 1;
    // clocks an iteration takes an SM's FP64 pipe: the sums (and about 3000 of
    // right-hand sides and barriers) against the transform of one pair
    const long long M = h->M;
    const long long sums = (M * M / (4 * C) + 3000) * ((count * C + sms - 1) / sms);
    const long long transform = 78 * M * ((((long long)count + 1) / 2 + sms - 1) / sms);
    if (sums < transform) {
      const size_t smem = sizeof(double) * (size_t)(3 * M + M / C);
#define MGWR_SUMS_LAUNCH(CC)                                                                      \
  mgwr::k_fas_fixed_sums<CC><<<(unsigned)(count * CC), (unsigned)M, smem, h->stream>>>(           \
      h->u[l], h->f[l], h->kcol + (size_t)l * M, n, (int)M, 1.0 / hl, 1.0 / (hl * hl), h->c,      \
      h->coef, parity, all_points, kFixedMaxIt, st, h->flags + 2)
      switch (C) {
        case 8: MGWR_SUMS_LAUNCH(8); break;
        case 4: MGWR_SUMS_LAUNCH(4); break;
        case 2: MGWR_SUMS_LAUNCH(2); break;
        default: MGWR_SUMS_LAUNCH(1); break;
      }
#undef MGWR_SUMS_LAUNCH
      return mgwr::counted(cudaGetLastError());
    }
    const unsigned grid = (unsigned)((count + 1) / 2);
    const size_t smem = mgwr::Pad<double>::len(L) * sizeof(Cx<double>);
    const Cx<double>* ks = h->kspec + (size_t)l * L;
#define MGWR_FIXED_LAUNCH(B)                                                                    \
  mgwr::k_fas_fixed<B><<<grid, B, smem, h->stream>>>(h->u[l], h->f[l], ks, h->tw, n, h->M, logL, \
                                                     1.0 / hl, 1.0 / (hl * hl), h->c,           \
                                                     h->sigma[l], h->coef, parity, all_points,   \
                                                     kFixedMaxIt, st, h->flags + 2)
    switch (L / 8) {
      case 32: MGWR_FIXED_LAUNCH(32); break;
      case 64: MGWR_FIXED_LAUNCH(64); break;
      case 128: MGWR_FIXED_LAUNCH(128); break;
      default: MGWR_FIXED_LAUNCH(256); break;
    }
#undef MGWR_FIXED_LAUNCH
    return mgwr::counted(cudaGetLastError());
  }
  const int blocks = (count + mgwr::kLineWarps - 1) / mgwr::kLineWarps;
  mgwr::k_fas_line<<<blocks, 32 * mgwr::kLineWarps, h->line_smem, h->stream>>>(
      h->u[l], h->f[l], h->r, n, h->M, level_h(l), h->c, h->coef, parity, all_points,
      reinterpret_cast<int*>(h->flags + 1));
  return mgwr::counted(cudaGetLastError());
}

cudaError_t launch_apply(mgwr_fas* h, int l, const double* u, const double* base, double* out,
                         double sign, bool norm) {
  // blocks per line: two blocks per SM where the lines are fewer, at least 16 steps each
  const int lines = level_n(l);
  int split = 2 * mgwr::sm_count() / lines;
  if (split > h->M / 16) split = h->M / 16;
  if (split > 16) split = 16;
  if (split < 1) split = 1;
  const dim3 grid((unsigned)lines, (unsigned)split);
  mgwr::k_fas_apply<<<grid, mgwr::kApplyThreads, h->apply_smem, h->stream>>>(
      u, h->r, base, out, level_n(l), h->M, level_h(l), h->c, h->coef, sign,
      norm ? h->flags : nullptr);
  return mgwr::counted(cudaGetLastError());
}

inline int grid_for(size_t total) {
  const size_t b = (total + 255) / 256;
  return (int)(b < 4096 ? (b > 0 ? b : 1) : 4096);
}

cudaError_t smooth_steps(mgwr_fas* h, int l, int steps) {
  cudaError_t e = cudaSuccess;
  for (int s = 0; s < steps && e == cudaSuccess; ++s) {
    e = launch_line(h, l, colour_parity(h, MGWR_RED), 0);
    if (e == cudaSuccess) e = launch_line(h, l, colour_parity(h, MGWR_BLACK), 0);
  }
  return e;
}

// One FAS cycle at level l on the handle's stream (no synchronisation).
cudaError_t fas_cycle(mgwr_fas* h, int l, int nu1, int nu2, int gamma) {
  if (l == 0) return launch_line(h, 0, 0, 1);
  cudaError_t e = smooth_steps(h, l, nu1);
  if (e != cudaSuccess) return e;
  // r = f - N_h(u)
  if ((e = launch_apply(h, l, h->u[l], h->f[l], h->rr[l], -1.0, false)) != cudaSuccess) return e;
  const int nc = level_n(l - 1);
  // ubar = R u, R r (into the coarse defect field, free until the coarse cycle)
  mgwr::k_fas_restrict2<<<grid_for((size_t)nc * h->M), 256, 0, h->stream>>>(
      h->u[l], h->ubar[l - 1], h->u[l - 1], h->rr[l], h->rr[l - 1], nc, h->M);
  if ((e = mgwr::counted(cudaGetLastError())) != cudaSuccess) return e;
  // f_c = N_2h(ubar) + R r; the coarse iterate starts from ubar
  if ((e = launch_apply(h, l - 1, h->ubar[l - 1], h->rr[l - 1], h->f[l - 1], 1.0, false)) !=
      cudaSuccess)
    return e;
  for (int g = 0; g < gamma; ++g)
    if ((e = fas_cycle(h, l - 1, nu1, nu2, gamma)) != cudaSuccess) return e;
  // u += P (u_c - ubar)
  mgwr::k_fas_correct<<<grid_for((size_t)level_n(l) * h->M), 256, 0, h->stream>>>(
      h->u[l], h->u[l - 1], h->ubar[l - 1], nc, h->M);
  if ((e = mgwr::counted(cudaGetLastError())) != cudaSuccess) return e;
  return smooth_steps(h, l, nu2);
}

// Reads the max-norm and Newton status written since the last clear (synchronises).
int read_flags(mgwr_fas* h, double* norm, bool* newton_failed) {
  unsigned long long host[2] = {0, 0};
  int s = fas_cuda(h, cudaMemcpyAsync(host, h->flags, sizeof(host), cudaMemcpyDeviceToHost,
                                      h->stream), "read flags");
  if (s == MGWR_OK) s = fas_cuda(h, cudaStreamSynchronize(h->stream), "synchronize");
  if (s != MGWR_OK) return s;
  if (norm) {
    double v;
    std::memcpy(&v, &host[0], sizeof(v));
    *norm = v;
  }
  if (newton_failed) *newton_failed = (host[1] & 3ull) != 0;
  return MGWR_OK;
}

cudaError_t clear_norm(mgwr_fas* h) {
  return cudaMemsetAsync(h->flags, 0, sizeof(unsigned long long), h->stream);
}

// The max-norm a defect left, and the failure of a line solve since the last clear.
int read_norm(mgwr_fas* h, double* norm) {
  bool failed = false;
  int s = read_flags(h, norm, &failed);
  if (s == MGWR_OK && failed)
    s = fas_fail(h, MGWR_E_NUMERIC, "a line solve did not settle (Newton's method or the whole-line fixed point)");
  return s;
}

int defect_norm(mgwr_fas* h, int l, double* norm) {
  int s = fas_cuda(h, clear_norm(h), "clear norm");
  if (s == MGWR_OK)
    s = fas_cuda(h, launch_apply(h, l, h->u[l], h->f[l], h->rr[l], -1.0, true), "defect");
  return s == MGWR_OK ? read_norm(h, norm) : s;
}

// The launches of one cycle from the finest level and of its defect's norm.
cudaError_t enqueue_cycle(mgwr_fas* h, int nu1, int nu2, int gamma) {
  const int L = h->nlev - 1;
  cudaError_t e = fas_cycle(h, L, nu1, nu2, gamma);
  if (e == cudaSuccess) e = clear_norm(h);
  if (e == cudaSuccess) e = launch_apply(h, L, h->u[L], h->f[L], h->rr[L], -1.0, true);
  return e;
}

void drop_graph(mgwr_fas* h) {
  if (h->graph) cudaGraphExecDestroy(h->graph);
  h->graph = nullptr;
  h->graph_key = -1;
}

// enqueue_cycle as a graph replay, captured on first use; the launches themselves
// where the stream cannot be captured or the graph not be made.
cudaError_t replay_cycle(mgwr_fas* h, int nu1, int nu2, int gamma) {
  const long long key =
      (((long long)h->order * 4 + h->smoother) * 4 + gamma) * 1024 + nu1 * 32 + nu2;
  if (h->graph_key != key) {
    drop_graph(h);
    if (cudaStreamBeginCapture(h->stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
      cudaGetLastError();
      return enqueue_cycle(h, nu1, nu2, gamma);
    }
    const long long before = mgwr::launch_counter();
    cudaError_t e = enqueue_cycle(h, nu1, nu2, gamma);
    cudaGraph_t g = nullptr;
    const cudaError_t end = cudaStreamEndCapture(h->stream, &g);
    const long long kernels = mgwr::launch_counter() - before;
    mgwr::add_launches(-kernels);  // captured, not run
    if (e == cudaSuccess) e = end;
    if (e == cudaSuccess) e = cudaGraphInstantiate(&h->graph, g, 0);
    if (g) cudaGraphDestroy(g);
    if (e != cudaSuccess) {
      h->graph = nullptr;
      cudaGetLastError();
      return enqueue_cycle(h, nu1, nu2, gamma);
    }
    h->graph_key = key;
    h->graph_kernels = kernels;
  }
  const cudaError_t e = cudaGraphLaunch(h->graph, h->stream);
  if (e == cudaSuccess) mgwr::add_launches(h->graph_kernels);
  return e;
}

double* field_of(mgwr_fas* h, int l, int which) {
  switch (which) {
    case MGWR_U: return h->u[l];
    case MGWR_F: return h->f[l];
    case MGWR_R: return h->rr[l];
    default: return nullptr;
  }
}

void release(mgwr_fas* h) {
  drop_graph(h);
  auto fr = [](double* p) { if (p) cudaFree(p); };
  for (auto* v : {&h->u, &h->f, &h->rr, &h->ubar})
    for (double* p : *v) fr(p);
  fr(h->r);
  fr(h->dk);
  fr(h->params);
  fr(h->kcol);
  if (h->kspec) cudaFree(h->kspec);
  if (h->tw) cudaFree(h->tw);
  if (h->flags) cudaFree(h->flags);
  if (h->ev0) cudaEventDestroy(h->ev0);
  if (h->ev1) cudaEventDestroy(h->ev1);
  if (h->own) cudaStreamDestroy(h->own);
}

}  // namespace

extern "C" {

int mgwr_fas_create(int n, int M, double T, double alpha, double c, int coefficient,
                    mgwr_fas_t* out) {
  if (out == nullptr) return MGWR_E_INVAL;
  *out = nullptr;
  if (n < 1 || n > 4095 || ((n + 1) & n) != 0) return MGWR_E_INVAL;
  if (M < 1 || M > mgwr::kFasMaxM) return MGWR_E_INVAL;
  if (!(T > 0.0) || !std::isfinite(T) || !(alpha > 0.0) || !(alpha <= 1.0)) return MGWR_E_INVAL;
  if (!std::isfinite(c)) return MGWR_E_INVAL;
  if (coefficient != MGWR_FAS_D_POROUS && coefficient != MGWR_FAS_D_CONSTANT) return MGWR_E_INVAL;
  // the smoother starts each Newton solve in FP32: its coefficients, the L1 scale
  // tau^-alpha / Gamma(2 - alpha) and |c| / h, must stay far inside FP32's range
  const double l1_scale = std::pow(T / M, -alpha) / std::tgamma(2.0 - alpha);
  if (!(l1_scale <= 1e30) || !(std::fabs(c) <= 1e30)) return MGWR_E_INVAL;
  mgwr_fas* h = new (std::nothrow) mgwr_fas;
  if (h == nullptr) return MGWR_E_NOMEM;
  h->n = n;
  h->M = M;
  h->T = T;
  h->alpha = alpha;
  h->c = c;
  h->coef = coefficient;
  while (level_n(h->nlev) < n) ++h->nlev;
  ++h->nlev;  // levels 0..nlev-1 with level_n(nlev-1) = n
  h->line_smem = sizeof(double) * (size_t)(1 + mgwr::kLineWarps) * M;
  h->apply_smem = sizeof(double) * 3 * (size_t)M;
  auto bail = [&](int code) {
    release(h);
    delete h;
    return code;
  };
  if (cudaStreamCreateWithFlags(&h->own, cudaStreamNonBlocking) != cudaSuccess ||
      cudaEventCreate(&h->ev0) != cudaSuccess || cudaEventCreate(&h->ev1) != cudaSuccess) {
    cudaGetLastError();
    return bail(MGWR_E_CUDA);
  }
  h->stream = h->own;
  auto alloc = [&](double** p, size_t bytes) {
    if (cudaMalloc(p, bytes) != cudaSuccess) {
      cudaGetLastError();
      *p = nullptr;
      return false;
    }
    return true;
  };
  bool ok = alloc(&h->r, sizeof(double) * M) && alloc(&h->dk, sizeof(double) * (M + 1)) &&
            alloc(&h->params, sizeof(double) * 2);
  if (ok && cudaMalloc(&h->flags, 3 * sizeof(unsigned long long)) != cudaSuccess) {
    cudaGetLastError();
    h->flags = nullptr;
    ok = false;
  }
  for (int l = 0; ok && l < h->nlev; ++l) {
    double *u = nullptr, *f = nullptr, *r = nullptr, *ub = nullptr;
    ok = alloc(&u, field_bytes(h, l)) && alloc(&f, field_bytes(h, l)) &&
         alloc(&r, field_bytes(h, l)) && alloc(&ub, field_bytes(h, l));
    h->u.push_back(u);
    h->f.push_back(f);
    h->rr.push_back(r);
    h->ubar.push_back(ub);
  }
  if (!ok) return bail(MGWR_E_NOMEM);
  // (1 + kLineWarps) * 1024 and 3 * 1024 doubles: within the default 48 KB
  static_assert((1 + mgwr::kLineWarps) * mgwr::kFasMaxM * sizeof(double) <= 48 * 1024,
                "k_fas_line shared memory");
  cudaError_t e = cudaSuccess;
  const double params[2] = {alpha, l1_scale};
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(h->params, params, sizeof(params), cudaMemcpyHostToDevice, h->stream);
  if (e == cudaSuccess)
    e = mgwr::launch_coefficients(h->r, h->dk, M, h->params, h->params + 1, 1, h->stream);
  for (int l = 0; e == cudaSuccess && l < h->nlev; ++l) {
    e = cudaMemsetAsync(h->u[l], 0, field_bytes(h, l), h->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(h->f[l], 0, field_bytes(h, l), h->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(h->rr[l], 0, field_bytes(h, l), h->stream);
  }
  if (e == cudaSuccess)
    e = cudaMemsetAsync(h->flags, 0, 3 * sizeof(unsigned long long), h->stream);
  // the fixed-point smoother's setup (Sec. 5): per level sigma_l = 2/h_l^2 + |c|/h_l,
  // the first column of (T_M + sigma_l I)^{-1} by divide and conquer, its spectrum
  if (e == cudaSuccess && M >= 128 && (M & (M - 1)) == 0) {
    const int L = 2 * M;
    for (int l = 0; l < h->nlev; ++l) {
      const double hl = level_h(l);
      h->sigma.push_back(2.0 / (hl * hl) + std::fabs(c) / hl);
    }
    double* sig_dev = nullptr;
    Cx<double>* work = nullptr;
    ok = alloc(&h->kcol, sizeof(double) * (size_t)h->nlev * M) &&
         alloc(&sig_dev, sizeof(double) * (size_t)h->nlev) &&
         cudaMalloc(&h->kspec, sizeof(Cx<double>) * (size_t)h->nlev * L) == cudaSuccess &&
         cudaMalloc(&h->tw, sizeof(Cx<double>) * (size_t)L) == cudaSuccess &&
         cudaMalloc(&work, sizeof(Cx<double>) * (size_t)h->nlev * 3 * M) == cudaSuccess;
    if (ok) {
      e = cudaMemcpyAsync(sig_dev, h->sigma.data(), sizeof(double) * h->nlev,
                          cudaMemcpyHostToDevice, h->stream);
      if (e == cudaSuccess)
        e = mgwr::launch_inverse_columns(h->kcol, h->r, sig_dev, h->nlev, M, 1, work, h->stream);
      if (e == cudaSuccess) e = mgwr::launch_twiddles(h->tw, L, h->stream);
      if (e == cudaSuccess)
        e = mgwr::launch_spectra(h->kspec, h->kcol, h->nlev, M, h->tw, h->stream);
      if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    } else {
      cudaGetLastError();
    }
    if (sig_dev) cudaFree(sig_dev);
    if (work) cudaFree(work);
    if (!ok) return bail(MGWR_E_NOMEM);
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return bail(MGWR_E_CUDA);
  }
  *out = h;
  return MGWR_OK;
}

int mgwr_fas_destroy(mgwr_fas_t h) {
  if (h == nullptr) return MGWR_E_INVAL;
  if (h->stream) cudaStreamSynchronize(h->stream);
  release(h);
  delete h;
  return MGWR_OK;
}

const char* mgwr_fas_last_error(mgwr_fas_t h) { return h ? h->err.c_str() : "null handle"; }

int mgwr_fas_set_order(mgwr_fas_t h, int order) {
  if (h == nullptr) return MGWR_E_INVAL;
  if (order != MGWR_ORDER_TEXT && order != MGWR_ORDER_TABLE)
    return fas_fail(h, MGWR_E_INVAL, "order must be MGWR_ORDER_TEXT or MGWR_ORDER_TABLE");
  h->order = order;
  return MGWR_OK;
}

int mgwr_fas_set_stream(mgwr_fas_t h, void* stream) {
  if (h == nullptr) return MGWR_E_INVAL;
  int s = fas_cuda(h, cudaStreamSynchronize(h->stream), "synchronize");
  if (s == MGWR_OK) h->stream = stream ? static_cast<cudaStream_t>(stream) : h->own;
  return s;
}

int mgwr_fas_reset(mgwr_fas_t h) {
  if (h == nullptr) return MGWR_E_INVAL;
  const int L = h->nlev - 1;
  int s = fas_cuda(h, cudaMemsetAsync(h->u[L], 0, field_bytes(h, L), h->stream), "clear u");
  if (s == MGWR_OK)
    s = fas_cuda(h, cudaMemsetAsync(h->flags, 0, 2 * sizeof(unsigned long long), h->stream),
                 "clear flags");
  return s;
}

int mgwr_fas_levels(mgwr_fas_t h, int* levels) {
  if (h == nullptr || levels == nullptr) return MGWR_E_INVAL;
  *levels = h->nlev;
  return MGWR_OK;
}

int mgwr_fas_field_set(mgwr_fas_t h, int level, int which, const double* host) {
  if (h == nullptr) return MGWR_E_INVAL;
  if (level < 0 || level >= h->nlev || host == nullptr || field_of(h, level, which) == nullptr)
    return fas_fail(h, MGWR_E_INVAL, "bad level, field or pointer");
  int s = fas_cuda(h, cudaMemcpyAsync(field_of(h, level, which), host, field_bytes(h, level),
                                      cudaMemcpyHostToDevice, h->stream), "field_set");
  if (s == MGWR_OK) s = fas_cuda(h, cudaStreamSynchronize(h->stream), "synchronize");
  return s;
}

int mgwr_fas_field_get(mgwr_fas_t h, int level, int which, double* host) {
  if (h == nullptr) return MGWR_E_INVAL;
  if (level < 0 || level >= h->nlev || host == nullptr || field_of(h, level, which) == nullptr)
    return fas_fail(h, MGWR_E_INVAL, "bad level, field or pointer");
  int s = fas_cuda(h, cudaMemcpyAsync(host, field_of(h, level, which), field_bytes(h, level),
                                      cudaMemcpyDeviceToHost, h->stream), "field_get");
  if (s == MGWR_OK) s = fas_cuda(h, cudaStreamSynchronize(h->stream), "synchronize");
  return s;
}

int mgwr_fas_set_rhs(mgwr_fas_t h, const double* f) {
  if (h == nullptr) return MGWR_E_INVAL;
  if (f == nullptr) return fas_fail(h, MGWR_E_INVAL, "null right-hand side");
  const int L = h->nlev - 1;
  int s = fas_cuda(h, cudaMemsetAsync(h->u[L], 0, field_bytes(h, L), h->stream), "clear u");
  if (s == MGWR_OK)
    s = fas_cuda(h, cudaMemsetAsync(h->flags, 0, 2 * sizeof(unsigned long long), h->stream),
                 "clear flags");
  if (s == MGWR_OK) s = mgwr_fas_field_set(h, L, MGWR_F, f);
  return s;
}

int mgwr_fas_set_initial(mgwr_fas_t h, const double* u0) {
  if (h == nullptr) return MGWR_E_INVAL;
  if (u0 == nullptr) return fas_fail(h, MGWR_E_INVAL, "null initial iterate");
  const int s = fas_cuda(
      h, cudaMemsetAsync(h->flags, 0, 2 * sizeof(unsigned long long), h->stream), "clear flags");
  return s == MGWR_OK ? mgwr_fas_field_set(h, h->nlev - 1, MGWR_U, u0) : s;
}

int mgwr_fas_get_solution(mgwr_fas_t h, double* u_host) {
  if (h == nullptr) return MGWR_E_INVAL;
  return mgwr_fas_field_get(h, h->nlev - 1, MGWR_U, u_host);
}

int mgwr_fas_defect(mgwr_fas_t h, int level, double* norm_inf) {
  if (h == nullptr) return MGWR_E_INVAL;
  if (level < 0 || level >= h->nlev) return fas_fail(h, MGWR_E_INVAL, "bad level");
  double nrm = 0.0;
  const int s = defect_norm(h, level, &nrm);
  if (s == MGWR_OK && norm_inf) *norm_inf = nrm;
  return s;
}

int mgwr_fas_residual(mgwr_fas_t h, double* norm_inf, double* r_host) {
  if (h == nullptr) return MGWR_E_INVAL;
  const int L = h->nlev - 1;
  int s = mgwr_fas_defect(h, L, norm_inf);
  if (s == MGWR_OK && r_host) s = mgwr_fas_field_get(h, L, MGWR_R, r_host);
  return s;
}

int mgwr_fas_set_smoother(mgwr_fas_t h, int smoother) {
  if (h == nullptr) return MGWR_E_INVAL;
  if (smoother != MGWR_FAS_SMOOTHER_AUTO && smoother != MGWR_FAS_SMOOTHER_MARCH &&
      smoother != MGWR_FAS_SMOOTHER_FIXED)
    return fas_fail(h, MGWR_E_INVAL, "unknown smoother");
  if (smoother == MGWR_FAS_SMOOTHER_FIXED && h->kspec == nullptr)
    return fas_fail(h, MGWR_E_INVAL, "the fixed-point smoother needs M a power of two in 128..1024");
  h->smoother = smoother;
  return MGWR_OK;
}

int mgwr_fas_line_iterations(mgwr_fas_t h, long long* count) {
  if (h == nullptr || count == nullptr) return MGWR_E_INVAL;
  unsigned long long v = 0;
  int s = fas_cuda(h, cudaMemcpyAsync(&v, h->flags + 2, sizeof(v), cudaMemcpyDeviceToHost,
                                      h->stream), "read count");
  if (s == MGWR_OK) s = fas_cuda(h, cudaStreamSynchronize(h->stream), "synchronize");
  if (s == MGWR_OK) *count = (long long)v;
  return s;
}

int mgwr_fas_smooth(mgwr_fas_t h, int level, int colour) {
  if (h == nullptr) return MGWR_E_INVAL;
  if (level < 0 || level >= h->nlev || (colour != MGWR_RED && colour != MGWR_BLACK))
    return fas_fail(h, MGWR_E_INVAL, "bad level or colour");
  int s = fas_cuda(h, launch_line(h, level, colour_parity(h, colour), 0), "smooth");
  bool failed = false;
  if (s == MGWR_OK) s = read_flags(h, nullptr, &failed);
  if (s == MGWR_OK && failed)
    s = fas_fail(h, MGWR_E_NUMERIC, "a line solve did not settle (Newton's method or the whole-line fixed point)");
  return s;
}

int mgwr_fas_cycle(mgwr_fas_t h, int cycle, int nu1, int nu2) {
  if (h == nullptr) return MGWR_E_INVAL;
  if ((cycle != 1 && cycle != 2) || nu1 < 0 || nu2 < 0 || nu1 + nu2 < 1 || nu1 > 16 || nu2 > 16)
    return fas_fail(h, MGWR_E_INVAL, "bad cycle parameters");
  int s = fas_cuda(h, fas_cycle(h, h->nlev - 1, nu1, nu2, cycle), "cycle");
  bool failed = false;
  if (s == MGWR_OK) s = read_flags(h, nullptr, &failed);
  if (s == MGWR_OK && failed)
    s = fas_fail(h, MGWR_E_NUMERIC, "a line solve did not settle (Newton's method or the whole-line fixed point)");
  return s;
}

int mgwr_fas_solve(mgwr_fas_t h, int cycle, int nu1, int nu2, double tol, int max_cycles,
                   mgwr_stats* stats) {
  if (h == nullptr) return MGWR_E_INVAL;
  if ((cycle != 1 && cycle != 2) || nu1 < 0 || nu2 < 0 || nu1 + nu2 < 1 || nu1 > 16 ||
      nu2 > 16 || !(tol >= 0.0) || max_cycles < 0)
    return fas_fail(h, MGWR_E_INVAL, "bad solve parameters");
  const int L = h->nlev - 1;
  mgwr_stats st{};
  double r0 = 0.0;
  int s = defect_norm(h, L, &r0);
  if (s != MGWR_OK) return s;
  if (!std::isfinite(r0)) return fas_fail(h, MGWR_E_NUMERIC, "non-finite initial defect");
  if (r0 == 0.0) {
    if (stats) *stats = st;
    return MGWR_OK;
  }
  st.relres = 1.0;
  s = fas_cuda(h, cudaEventRecord(h->ev0, h->stream), "event");
  while (s == MGWR_OK && st.cycles < max_cycles && st.relres > tol) {
    s = fas_cuda(h, st.cycles == 0 ? enqueue_cycle(h, nu1, nu2, cycle)
                                   : replay_cycle(h, nu1, nu2, cycle), "cycle");
    double nrm = 0.0;
    if (s == MGWR_OK) s = read_norm(h, &nrm);
    if (s != MGWR_OK) break;
    ++st.cycles;
    st.relres = nrm / r0;
    if (!std::isfinite(st.relres)) s = fas_fail(h, MGWR_E_NUMERIC, "non-finite defect");
  }
  if (cudaEventRecord(h->ev1, h->stream) == cudaSuccess &&
      cudaEventSynchronize(h->ev1) == cudaSuccess) {
    float ms = 0.0f;
    if (cudaEventElapsedTime(&ms, h->ev0, h->ev1) == cudaSuccess) st.seconds = 1e-3 * ms;
  }
  cudaGetLastError();
  st.factor = st.cycles > 0 ? std::pow(st.relres, 1.0 / st.cycles) : 0.0;
  if (stats) *stats = st;
  if (s != MGWR_OK) return s;
  return st.relres <= tol ? MGWR_OK
                          : fas_fail(h, MGWR_E_NOCONV, "max_cycles reached before tol");
}

}  // extern "C"
