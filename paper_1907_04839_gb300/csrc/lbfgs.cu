// register_landmarks: minimise the loss of Eq. 3 over p0 by L-BFGS
// (Section 2.1; the outer optimisation of Algorithm 1).  The paper used
// VNL's L-BFGS without stating its settings; this one uses textbook choices:
//  * memory m, two-loop recursion with initial scaling gamma = s.y / y.y;
//  * first step -g scaled to 1/||g0||;
//  * strong-Wolfe line search (c1 = 1e-4, c2 = 0.9) by bracketing and zoom
//    with safeguarded cubic interpolation, at most 20 evaluations per search;
//  * a curvature pair is kept only if s.y > 1e-12 ||s|| ||y||;
//  * stop when ||g|| <= grad_tol ||g0||, or after max_iter iterations.
//
// The iterate, the gradient, the direction and the (s, y) history are FP64
// vectors on the device.  Dot products reduce deterministically, in a fixed
// order.  The host runs the scalar control flow of the line search.  An
// iteration is three launches around its evaluation and one readback: the
// direction with the step to the first trial point (one cluster), the sweeps,
// and every product the host may need of the result.  The first trial of
// an iteration is evaluated before the host has seen its slope; the rare
// direction that does not descend is thrown away with its evaluation.
//
// A registration at N = 256, T = 10, 8 iterations: 950 us; 2.70 ms with a launch
// and a copy per operation of the recursion, a synchronising copy per scalar
// and the gradient by launches per step.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

#include "engine.h"
#include "gs_device.cuh"

namespace gs {
namespace {

constexpr int kLT = 256;     // threads per CTA of the vector kernels
constexpr int kMaxM = 64;

int vec_grid(int n, int num_sms) { return std::max(1, std::min((n + kLT - 1) / kLT, 2 * num_sms)); }

// What the host reads back after an evaluation.
enum : int { kRbSlope, kRbSy, kRbYy, kRbSs, kRbGg, kRbLoss, kRbSlope0, kRbStatus, kRbWords };

struct EvalArgs {
  const double *x, *g, *d, *xt, *gt;
  int n;
  double* part;            // [kRbLoss][gridDim.x]
  unsigned* ticket;
  const double* loss;
  const unsigned* status;
  double* out;             // kRbWords (kRbSlope0 is k_direction's)
};

// The products of an evaluated trial point (xt, gt): its slope gt.d, and with
// s = xt - x, y = gt - g the numbers s.y, y.y, s.s and gt.gt that follow an
// accepted step.  One pass; the last CTA adds the partials in order.
__global__ void __launch_bounds__(kLT) k_eval_products(EvalArgs e) {
  constexpr int K = kRbLoss;
  __shared__ double sh[K][kLT / 32];
  __shared__ int am_last;
  double v[K] = {0.0, 0.0, 0.0, 0.0, 0.0};
  for (int i = blockIdx.x * kLT + threadIdx.x; i < e.n; i += gridDim.x * kLT) {
    const double gt = e.gt[i], s = e.xt[i] - e.x[i], y = gt - e.g[i];
    v[kRbSlope] = fma(gt, e.d[i], v[kRbSlope]);
    v[kRbSy] = fma(s, y, v[kRbSy]);
    v[kRbYy] = fma(y, y, v[kRbYy]);
    v[kRbSs] = fma(s, s, v[kRbSs]);
    v[kRbGg] = fma(gt, gt, v[kRbGg]);
  }
#pragma unroll
  for (int k = 0; k < K; ++k) v[k] = warp_sum_f64(v[k]);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0)
#pragma unroll
    for (int k = 0; k < K; ++k) sh[k][w] = v[k];
  __syncthreads();
  if (w == 0) {
    if (l < K) {
      double t = 0.0;
      for (int u = 0; u < kLT / 32; ++u) t += sh[l][u];
      e.part[l * gridDim.x + blockIdx.x] = t;
    }
    __threadfence();
    __syncwarp();
    if (l == 0) am_last = (atomicAdd(e.ticket, 1u) == gridDim.x - 1);
  }
  __syncthreads();
  if (!am_last || w >= K) return;
  __threadfence();
  double t = 0.0;
  for (unsigned b = l; b < gridDim.x; b += 32) t += *((volatile double*)&e.part[w * gridDim.x + b]);
  t = warp_sum_f64(t);
  if (l == 0) e.out[w] = t;
  if (threadIdx.x == 0) {
    e.out[kRbLoss] = *e.loss;
    e.out[kRbStatus] = static_cast<double>(*e.status);
    *e.ticket = 0u;
  }
}

constexpr int kDT = 512;  // threads per CTA of k_direction
constexpr int kDC = 16;   // CTAs of its cluster

enum : int { kAcceptNone = 0, kAcceptStep = 1, kAcceptGrad = 2 };

struct DirArgs {
  double *x, *g, *d, *xt;
  const double* gt;
  double *S, *Y;           // m x n history
  int n, m;
  int accept;              // kAcceptStep: x <- xt, g <- gt; kAcceptGrad: g <- gt
  int slot;                // with kAcceptStep: history slot of (xt - x, gt - g), -1: not kept
  int direction;           // 0: accept only
  int head, stored;        // the newest `stored` pairs end before slot `head`
  double gamma;
  double a1;               // xt <- x + a1 d
  double* slope;           // g.d
  double rho[kMaxM];
};

// Accept the last trial point, then d = -H g by the two-loop recursion, its
// slope and the first trial point.  One cluster: a recursion of `stored` pairs
// is 2 stored + 1 passes over d, each ended by a cluster-wide dot product, and
// every pass updates d with one pair and multiplies it with the next, so a
// pair costs two passes instead of four launches and a copy (N = 256, 7
// pairs: 28 launches and 8 copies before).  Each element is read and written
// by one thread throughout; only the dot products cross threads.
__global__ void __launch_bounds__(kDT) k_direction(DirArgs a) {
  __shared__ double sh[kDT / 32];
  __shared__ double peers[2][kDC];  // every CTA's partial, two passes in turn
  __shared__ double total;
  __shared__ double alpha[kMaxM];
  const int rank = static_cast<int>(cluster_rank());
  if (blockDim.x != kDT || cluster_size() != kDC) return;
  const int t0 = rank * kDT + threadIdx.x, step = kDC * kDT;
  int turn = 0;
  const auto cluster_total = [&](double v) -> double {
    v = block_sum_f64(v, sh);
    if (threadIdx.x < kDC) {
      // thread c of warp 0 sends to CTA c (block_sum leaves the sum in warp 0)
      v = __shfl_sync(0xffffu, v, 0);
      const uint32_t to = dsmem_addr(smem_u32(&peers[turn][rank]), threadIdx.x);
      asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(to), "d"(v) : "memory");
    }
    __syncwarp();
    cluster_sync();
    if (threadIdx.x < 32) {
      double p = threadIdx.x < kDC ? peers[turn][threadIdx.x] : 0.0;
      p = warp_sum_f64(p);
      if (threadIdx.x == 0) total = p;
    }
    __syncthreads();
    turn ^= 1;  // the next pass's stores may arrive while a slow CTA still reads this one's
    return total;
  };
  const auto pair = [&](int k) { return (a.head - 1 - k + a.m) % a.m; };
  cluster_sync();  // every CTA has started
  for (int i = t0; i < a.n; i += step) {
    double g = a.g[i];
    if (a.accept) {
      const double gt = a.gt[i];
      if (a.accept == kAcceptStep) {
        const double xt = a.xt[i];
        if (a.slot >= 0) {
          a.S[static_cast<size_t>(a.slot) * a.n + i] = xt - a.x[i];
          a.Y[static_cast<size_t>(a.slot) * a.n + i] = gt - g;
        }
        a.x[i] = xt;
      }
      a.g[i] = g = gt;
    }
    if (a.direction) a.d[i] = g;
  }
  if (!a.direction) return;  // no peer reads this CTA's shared memory
  const auto hist = [&](const double* h, int j) { return h + static_cast<size_t>(j) * a.n; };
  // d <- d - alpha_j Y_j, newest pair first
  double v = 0.0;
  if (a.stored > 0) {
    const double* S = hist(a.S, pair(0));
    for (int i = t0; i < a.n; i += step) v = fma(S[i], a.d[i], v);
  }
  for (int k = 0; k < a.stored; ++k) {
    const int j = pair(k);
    const double al = a.rho[j] * cluster_total(v);
    if (threadIdx.x == 0) alpha[j] = al;
    const double* Y = hist(a.Y, j);
    // next: the older pair's S, or (d scaled by gamma) the oldest pair's Y
    const bool lastp = k + 1 == a.stored;
    const double* N = lastp ? Y : hist(a.S, pair(k + 1));
    const double sc = lastp ? a.gamma : 1.0;
    v = 0.0;
    for (int i = t0; i < a.n; i += step) {
      const double d = sc * fma(-al, Y[i], a.d[i]);
      a.d[i] = d;
      v = fma(N[i], d, v);
    }
  }
  __syncthreads();
  for (int k = a.stored - 1; k >= 0; --k) {
    const int j = pair(k);
    const double c = alpha[j] - a.rho[j] * cluster_total(v);
    const double* S = hist(a.S, j);
    const double* N = k > 0 ? hist(a.Y, pair(k - 1)) : nullptr;
    v = 0.0;
    for (int i = t0; i < a.n; i += step) {
      const double d = fma(c, S[i], a.d[i]);
      a.d[i] = d;
      if (N) v = fma(N[i], d, v);
    }
  }
  v = 0.0;
  for (int i = t0; i < a.n; i += step) {
    const double d = -a.d[i];
    a.d[i] = d;
    a.xt[i] = fma(a.a1, d, a.x[i]);
    v = fma(a.g[i], d, v);
  }
  v = cluster_total(v);
  if (rank == 0 && threadIdx.x == 0) *a.slope = v;
  // The last remote store of the kernel came before the last cluster barrier.
}

// xt <- x + a d
__global__ void __launch_bounds__(kLT) k_step(double* xt, const double* x, const double* d, int n, double a) {
  for (int i = blockIdx.x * kLT + threadIdx.x; i < n; i += gridDim.x * kLT) xt[i] = fma(a, d[i], x[i]);
}

__global__ void __launch_bounds__(kLT) k_f32_to_f64(double* y, const float* x, int n) {
  for (int i = blockIdx.x * kLT + threadIdx.x; i < n; i += gridDim.x * kLT) y[i] = x ? (double)x[i] : 0.0;
}

__global__ void __launch_bounds__(kLT) k_f64_to_f32(float* y, const double* x, int n) {
  for (int i = blockIdx.x * kLT + threadIdx.x; i < n; i += gridDim.x * kLT) y[i] = (float)x[i];
}

// Landmark distances |q1_i - t_i| (Section 3.1): out[0] = sum, out[1] = max.
// Landmarks in dim = 2 or 3 dimensions.
__global__ void __launch_bounds__(kLT) k_dist(const double* q1, const double* t, int n, int dim, double* part,
                                             unsigned* ticket, double* out) {
  __shared__ double sh[kLT / 32];
  __shared__ double shm[kLT / 32];
  __shared__ int am_last;
  double sum = 0.0, mx = 0.0;
  for (int i = blockIdx.x * kLT + threadIdx.x; i < n; i += gridDim.x * kLT) {
    double r2 = 0.0;
    for (int k = 0; k < dim; ++k) {
      const double d = q1[dim * i + k] - t[dim * i + k];
      r2 += d * d;
    }
    const double r = sqrt(r2);
    sum += r;
    mx = fmax(mx, r);
  }
  const double bs = block_sum_f64(sum, sh);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0) shm[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    double m = 0.0;
    for (int w = 0; w < kLT / 32; ++w) m = fmax(m, shm[w]);
    part[blockIdx.x] = bs;
    part[gridDim.x + blockIdx.x] = m;
    __threadfence();
    am_last = (atomicAdd(ticket, 1u) == gridDim.x - 1);
  }
  __syncthreads();
  if (!am_last || threadIdx.x != 0) return;
  __threadfence();
  double s = 0.0, m = 0.0;
  for (unsigned b = 0; b < gridDim.x; ++b) {
    s += *((volatile double*)&part[b]);
    m = fmax(m, *((volatile double*)&part[gridDim.x + b]));
  }
  out[0] = s;
  out[1] = m;
  *ticket = 0u;
}

template <typename K, typename... Args>
cudaError_t vlaunch(int grid, cudaStream_t st, K kern, Args... args) {
  kern<<<grid, kLT, 0, st>>>(args...);
  return cudaGetLastError();
}

gs_status alloc_lbfgs(Workspace& w, int n3, int m) {
  LbfgsBufs& b = w.lb;
  if (b.n3 >= n3 && b.m >= m) return GS_OK;
  b.free_all();
  auto get = [&](double** p, size_t count) -> cudaError_t {
    void* v = nullptr;
    cudaError_t e = cudaMalloc(&v, count * sizeof(double) + 256);
    if (e == cudaSuccess) {
      b.allocs.push_back(v);
      *p = static_cast<double*>(v);
    }
    return e;
  };
  const size_t n = static_cast<size_t>(n3);
  GS_CUDA(get(&b.x, n));
  GS_CUDA(get(&b.g, n));
  GS_CUDA(get(&b.d, n));
  GS_CUDA(get(&b.xt, n));
  GS_CUDA(get(&b.gt, n));
  GS_CUDA(get(&b.S, n * m));
  GS_CUDA(get(&b.Y, n * m));
  GS_CUDA(get(&b.scal, 16));
  GS_CUDA(get(&b.part, 4 * 4 * 1024));
  double* t = nullptr;
  GS_CUDA(get(&t, 8));
  b.ticket = reinterpret_cast<unsigned*>(t);
  GS_CUDA(cudaMemset(b.ticket, 0, 8 * sizeof(double)));
  GS_CUDA(cudaMemset(b.S, 0, n * m * sizeof(double)));
  GS_CUDA(cudaMemset(b.Y, 0, n * m * sizeof(double)));
  // every vector starts finite: a product of an unused one is read back unused
  for (double* p : {b.x, b.g, b.d, b.xt, b.gt}) GS_CUDA(cudaMemset(p, 0, n * sizeof(double)));
  GS_CUDA(cudaDeviceSynchronize());  // the caller's stream need not wait for the default one
  if (!b.host) GS_CUDA(cudaMallocHost(&b.host, 16 * sizeof(double)));
  b.n3 = n3;
  b.m = m;
  return GS_OK;
}

// One register_landmarks run on the current device (caller holds the lock).
struct Lbfgs {
  Workspace& w;
  const gs_params& prm;
  cudaStream_t st;
  const float* dq;
  const float* dt;
  int n3, m, grid;
  int evals = 0;

  Lbfgs(Workspace& w_, const gs_params& p, cudaStream_t s, const float* q, const float* t)
      : w(w_), prm(p), st(s), dq(q), dt(t), n3(static_cast<int>(dim_of(p) * p.N)), m(p.lbfgs_m),
        grid(vec_grid(n3, w_.num_sms)) {}

  // Enqueue the evaluation of the momenta xv: gradient to gt, products to scal.
  gs_status enqueue_eval(const double* xv) {
    LbfgsBufs& b = w.lb;
    ShootOut out;
    out.gp64 = b.gt;
    gs_status s = enqueue_shoot(w, 1, prm, dq, nullptr, xv, dt, out, st);
    if (s != GS_OK) return s;
    const EvalArgs e{b.x, b.g, b.d, b.xt, b.gt, n3, b.part, b.ticket, w.scalars + 1, w.status, b.scal};
    GS_CUDA(vlaunch(grid, st, k_eval_products, e));
    return GS_OK;
  }

  // Wait for the evaluation; its products are in w.lb.host afterwards.
  gs_status readback() {
    GS_CUDA(cudaMemcpyAsync(w.lb.host, w.lb.scal, kRbWords * sizeof(double), cudaMemcpyDeviceToHost, st));
    GS_CUDA(cudaStreamSynchronize(st));
    return GS_OK;
  }

  // Count the evaluation read back last; its errors.
  gs_status count_eval() {
    ++evals;
    return w.lb.host[kRbStatus] != 0.0 ? finish_sync(w, st) : GS_OK;
  }

  // phi(a) = f(x + a d) and phi'(a) = g(x + a d).d; the point and its
  // gradient land in xt, gt.  first: the evaluation that followed the
  // direction, already read back.
  gs_status eval_step(double a, bool first, double* f, double* dphi) {
    gs_status s;
    if (!first) {
      GS_CUDA(vlaunch(grid, st, k_step, w.lb.xt, w.lb.x, w.lb.d, n3, a));
      if ((s = enqueue_eval(w.lb.xt)) != GS_OK) return s;
      if ((s = readback()) != GS_OK) return s;
    }
    if ((s = count_eval()) != GS_OK) return s;
    *f = w.lb.host[kRbLoss];
    *dphi = w.lb.host[kRbSlope];
    return GS_OK;
  }

  static double cubic_min(double a, double fa, double da, double b, double fb, double db) {
    const double d1 = da + db - 3.0 * (fa - fb) / (a - b);
    const double disc = d1 * d1 - da * db;
    if (!(disc >= 0.0)) return NAN;
    const double d2 = (b > a ? 1.0 : -1.0) * std::sqrt(disc);
    const double den = db - da + 2.0 * d2;
    if (den == 0.0) return NAN;
    return b - (b - a) * (db + d2 - d1) / den;
  }

  // Strong-Wolfe line search from f0 with slope dphi0 < 0 and first trial a1.
  // On success *step > 0 and xt, gt, *fnew hold the accepted point.
  gs_status line_search(double f0, double dphi0, double a1, double* step, double* fnew) {
    const double c1 = 1e-4, c2 = 0.9;
    const int max_evals = 20;
    *step = 0.0;
    int used = 0;
    double a_prev = 0.0, f_prev = f0, d_prev = dphi0, a = a1;
    for (int it = 0; used < max_evals; ++it) {
      double fa, da;
      gs_status s = eval_step(a, used == 0, &fa, &da);
      if (s != GS_OK) return s;
      ++used;
      bool zoom = false;
      double lo = 0, flo = 0, dlo = 0, hi = 0, fhi = 0, dhi = 0;
      if (!(fa <= f0 + c1 * a * dphi0) || (it > 0 && fa >= f_prev)) {
        zoom = true;
        lo = a_prev; flo = f_prev; dlo = d_prev; hi = a; fhi = fa; dhi = da;
      } else if (std::fabs(da) <= -c2 * dphi0) {
        *step = a;
        *fnew = fa;
        return GS_OK;
      } else if (da >= 0.0) {
        zoom = true;
        lo = a; flo = fa; dlo = da; hi = a_prev; fhi = f_prev; dhi = d_prev;
      }
      if (zoom) {
        while (used < max_evals) {
          double aj = cubic_min(lo, flo, dlo, hi, fhi, dhi);
          const double wdt = hi - lo;
          const double b0 = wdt > 0 ? lo + 0.1 * wdt : hi - 0.1 * wdt;
          const double b1 = wdt > 0 ? hi - 0.1 * wdt : lo + 0.1 * wdt;
          if (!(aj >= std::min(b0, b1) && aj <= std::max(b0, b1))) aj = 0.5 * (lo + hi);
          double fj, dj;
          s = eval_step(aj, false, &fj, &dj);
          if (s != GS_OK) return s;
          ++used;
          if (!(fj <= f0 + c1 * aj * dphi0) || fj >= flo) {
            hi = aj; fhi = fj; dhi = dj;
          } else {
            if (std::fabs(dj) <= -c2 * dphi0) {
              *step = aj;
              *fnew = fj;
              return GS_OK;
            }
            if (dj * (hi - lo) >= 0.0) {
              hi = lo; fhi = flo; dhi = dlo;
            }
            lo = aj; flo = fj; dlo = dj;
          }
        }
        return GS_OK;  // no acceptable step: *step == 0
      }
      a_prev = a; f_prev = fa; d_prev = da;
      a = 2.0 * a;
    }
    return GS_OK;
  }

  gs_status launch_direction(const DirArgs& a) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kDC);
    cfg.blockDim = dim3(kDT);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kDC;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    GS_CUDA(cudaFuncSetAttribute(k_direction, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    GS_CUDA(cudaLaunchKernelEx(&cfg, k_direction, a));
    return GS_OK;
  }

  gs_status run(gs_register_info* info) {
    LbfgsBufs& b = w.lb;
    int head = 0, stored = 0, status = 1, it = 0;
    DirArgs da;
    std::memset(&da, 0, sizeof(da));
    da.x = b.x;
    da.g = b.g;
    da.d = b.d;
    da.xt = b.xt;
    da.gt = b.gt;
    da.S = b.S;
    da.Y = b.Y;
    da.n = n3;
    da.m = m;
    da.gamma = 1.0;
    da.slope = b.scal + kRbSlope0;
    da.accept = kAcceptGrad;
    da.slot = -1;
    gs_status s = enqueue_eval(b.x);
    if (s != GS_OK) return s;
    if ((s = readback()) != GS_OK) return s;
    if ((s = count_eval()) != GS_OK) return s;
    double f = b.host[kRbLoss];
    const double g0 = std::sqrt(b.host[kRbGg]);
    double gnorm = g0;
    if (g0 == 0.0) status = 0;
    for (it = 0; status == 1 && it < prm.max_iter; ++it) {
      da.direction = 1;
      da.head = head;
      da.stored = stored;
      da.a1 = (it == 0) ? 1.0 / g0 : 1.0;
      if ((s = launch_direction(da)) != GS_OK) return s;
      if ((s = enqueue_eval(b.xt)) != GS_OK) return s;
      if ((s = readback()) != GS_OK) return s;
      da.accept = kAcceptNone;
      double dphi0 = b.host[kRbSlope0];
      if (!(dphi0 < 0.0)) {  // not a descent direction: restart from -g
        if (!goes_with_its_point(static_cast<unsigned>(b.host[kRbStatus]))) return finish_sync(w, st);
        if (b.host[kRbStatus] != 0.0) GS_CUDA(cudaMemsetAsync(w.status, 0, sizeof(unsigned), st));
        dphi0 = -gnorm * gnorm;
        da.stored = stored = 0;
        if ((s = launch_direction(da)) != GS_OK) return s;
        if ((s = enqueue_eval(b.xt)) != GS_OK) return s;
        if ((s = readback()) != GS_OK) return s;
      }
      double a = 0.0, fn = 0.0;
      if ((s = line_search(f, dphi0, da.a1, &a, &fn)) != GS_OK) return s;
      if (a == 0.0) {
        status = 2;  // no step met the Wolfe conditions: noise floor reached
        break;
      }
      // The accepted point is the one evaluated last.
      const double sy = b.host[kRbSy], yy = b.host[kRbYy], ss = b.host[kRbSs];
      da.accept = kAcceptStep;
      da.slot = -1;
      if (sy > 1e-12 * std::sqrt(ss * yy)) {
        da.slot = head;
        da.rho[head] = 1.0 / sy;
        da.gamma = sy / yy;
        head = (head + 1) % m;
        if (stored < m) ++stored;
      }
      f = fn;
      gnorm = std::sqrt(b.host[kRbGg]);
      if (gnorm <= prm.grad_tol * g0) {
        status = 0;
        ++it;
        break;
      }
    }
    if (da.accept == kAcceptStep) {  // the last step's x
      da.direction = 0;
      if ((s = launch_direction(da)) != GS_OK) return s;
    }
    if (info) {
      info->loss = f;
      info->grad_norm0 = g0;
      info->grad_norm = gnorm;
      info->iters = it;
      info->evals = evals;
      info->status = status;
    }
    return GS_OK;
  }
};

gs_status run_register(const gs_params* prm, const float* q0, const float* target, float* p0_inout,
                       gs_register_info* info, void* stream) {
  gs_status s = check_params(prm);
  if (s != GS_OK) return s;
  if (!q0 || !target || !p0_inout) return fail(GS_EINVAL, "q0, target and p0_inout must not be NULL");
  if (prm->lbfgs_m < 1 || prm->lbfgs_m > kMaxM) return fail(GS_EINVAL, "lbfgs_m must be in [1, 64]");
  if (prm->max_iter < 0) return fail(GS_EINVAL, "max_iter must be >= 0");
  if (!(prm->grad_tol >= 0.0)) return fail(GS_EINVAL, "grad_tol must be >= 0");
  std::lock_guard<std::mutex> lk(engine_mutex());
  Workspace* w = nullptr;
  if ((s = get_workspace(&w)) != GS_OK) return s;
  const int n = static_cast<int>(prm->N), n3 = dim_of(*prm) * n;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // (the flow at the end keeps every state)
  if ((s = reserve_sweep(*w, 1, *prm, stages_of(prm->integrator) * prm->T, st)) != GS_OK) return s;
  if ((s = alloc_lbfgs(*w, n3, prm->lbfgs_m)) != GS_OK) return s;
  bool host = false;
  const float *dq = nullptr, *dt = nullptr, *dp = nullptr;
  if ((s = stage_in(q0, w->in_q, n3, st, &dq, &host)) != GS_OK) return s;
  if ((s = stage_in(target, w->in_t, n3, st, &dt, &host)) != GS_OK) return s;
  if ((s = stage_in(p0_inout, w->in_p, n3, st, &dp, &host)) != GS_OK) return s;
  const int grid = vec_grid(n3, w->num_sms);
  GS_CUDA(vlaunch(grid, st, k_f32_to_f64, w->lb.x, dp, n3));
  Lbfgs opt(*w, *prm, st, dq, dt);
  if ((s = opt.run(info)) != GS_OK) return s;
  // result: p0 back to float32, and the landmark distances at q(1)
  GS_CUDA(vlaunch(grid, st, k_f64_to_f32, w->out_a, (const double*)w->lb.x, n3));
  bool dummy = false;
  if ((s = copy_out(p0_inout, w->out_a, n3, st, &dummy)) != GS_OK) return s;
  if (info) {
    ShootOut flow;
    flow.order_flow = w->ordered;  // q(1) in the order of the last gradient's targets
    if ((s = enqueue_shoot(*w, 0, *prm, dq, nullptr, w->lb.x, nullptr, flow, st)) != GS_OK) return s;
    GS_CUDA(vlaunch(grid, st, k_dist, (const double*)w->q64, (const double*)w->t64, n, dim_of(*prm), w->lb.part,
                    w->lb.ticket, w->lb.scal));
    double* const dist = w->lb.host;
    GS_CUDA(cudaMemcpyAsync(dist, w->lb.scal, 2 * sizeof(double), cudaMemcpyDeviceToHost, st));
    if ((s = finish_sync(*w, st)) != GS_OK) return s;
    info->avg_dist = dist[0] / n;
    info->max_dist = dist[1];
    return info->status == 0 ? GS_OK : GS_NOT_CONVERGED;
  }
  if ((s = finish_sync(*w, st)) != GS_OK) return s;
  return GS_OK;
}

}  // namespace
}  // namespace gs

extern "C" gs_status register_landmarks(const gs_params* prm, const float* q0, const float* target, float* p0_inout,
                                        gs_register_info* info, void* stream) {
  gs::set_last_error("");
  return gs::run_register(prm, q0, target, p0_inout, info, stream);
}
