// Whole sweeps of small problems in one launch.
//
// Up to kSmallNpad landmarks a time step holds too little work for the
// chip: a launch per step spends about 4.2 us whatever the size, on launch
// hand-over, fill, cluster reduction and drain.  Here one cluster of 16 CTAs
// runs the whole flow, the loss and the whole reverse sweep.
//
// Work split.  CTA r owns landmarks [r*Mc, (r+1)*Mc), Mc = Npad / 16, and
// keeps their FP64 state and adjoint in registers from the first step to the
// last.  Every CTA holds the records of all landmarks in shared memory.  Per
// step, thread (lt, g) sums target lt over every G-th source record in plain
// FP32 (at most 32 records); the G group sums of a target meet in shared
// memory and are added error-free (TwoSum).  So a target's sum never leaves
// its CTA, and the step ends by sending the Mc new records to the next buffer
// of all 16 CTAs: asynchronous remote stores that count down the receiver's
// mbarrier, so one trip carries data and signal (a cluster barrier after plain
// remote stores took 1800 cycles a step, these 900).  Two buffers suffice: a
// CTA sends into a buffer only after it has every record of the step before,
// whose senders had finished reading that buffer.
//
// The FP64 unit issues one warp's instruction in 19 cycles, so the state is
// kept in record units (kq q, kappa beta): a step's update is one FMA a
// coordinate and its record a conversion.
//
// The forward sweep also writes each state to its trajectory slot; the
// reverse sweep reads the state of the step before from there (L2) while the
// current step's pair sums run.
//
// A gradient at N = 256, T = 10 as a call from Python: 98 us, 165 by launches
// per step.  What bounds it: the chain of one exchange, one shared-memory reduction and
// the dependent FP64 update a step up to about 200 landmarks, then the FP32
// pipe of its 16 SMs, which is where the launch-per-step path takes over.
#include <algorithm>
#include <map>
#include <mutex>

#include "pair_tile.cuh"

namespace gs {
namespace {

constexpr int kSmallT = 256;  // threads per CTA: two warps a scheduler fill the reverse loop
constexpr int kSmallC = 16;   // CTAs of the cluster

__device__ __forceinline__ void st_dsmem_f64(uint32_t addr, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}

// Remote store that completes 16 bytes of transaction count on the remote
// mbarrier (addresses from dsmem_addr, same CTA).
__device__ __forceinline__ void st_async_f4(uint32_t addr, float4 v, uint32_t bar) {
  asm volatile(
      "st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr),
      "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(bar)
      : "memory");
}

// mbar_wait for data that other CTAs of the cluster sent.
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t* bar, unsigned parity) {
  const uint32_t addr = smem_u32(bar);
  for (long it = 0; it < kSpinLimit; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(addr), "r"(parity) : "memory");
    if (ok) return true;
  }
  return false;
}

// K sums r[k][0] + r[k][stride] + ... (count terms), the rounding errors
// carried along; loads in batches ahead of the chains.
template <int K>
__device__ __forceinline__ void sum_groups(const float* const (&r)[K], int count, int stride, double (&out)[K]) {
  constexpr int B = 8;
  float s[K], e[K];
#pragma unroll
  for (int k = 0; k < K; ++k) s[k] = e[k] = 0.f;
  for (int g = 0; g < count; g += B) {
    float x[K][B];
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
      for (int u = 0; u < B; ++u) x[k][u] = g + u < count ? r[k][(g + u) * stride] : 0.f;
#pragma unroll
    for (int u = 0; u < B; ++u)
#pragma unroll
      for (int k = 0; k < K; ++k) {
        float er;
        two_sum(s[k], x[k][u], s[k], er);
        e[k] = __fadd_rn(e[k], er);
      }
  }
#pragma unroll
  for (int k = 0; k < K; ++k) out[k] = static_cast<double>(s[k]) + static_cast<double>(e[k]);
}

template <int D>
__global__ void __launch_bounds__(kSmallT) k_small_sweep(SmallArgs a) {
  extern __shared__ __align__(16) float4 dyn[];
  __shared__ double sh[kSmallT / 32];
  __shared__ double clsum[2][kSmallC];  // rank 0: every CTA's H and mismatch sums
  __shared__ __align__(8) uint64_t full[4];  // record buffers: state 0, 1, adjoint 0, 1
  const int tid = threadIdx.x;
  const int rank = static_cast<int>(cluster_rank());
  const int recs = a.npad / 2, RF = recs * D;
  const int Mc = a.npad / kSmallC;  // a multiple of 4: whole records
  const int nf = Mc / 2 * D;        // float4 of this CTA's records
  const int G = a.groups;
  // Record buffers: 0 and 1 the state, 2 and 3 the adjoint.
  const auto buf = [&](int b) { return dyn + b * RF; };
  float4* stage = dyn + 4 * RF;
  float* red = reinterpret_cast<float*>(stage + nf);
  // The launch must match the kernel (the same outcome in every CTA).
  if (blockDim.x != kSmallT || cluster_size() != kSmallC || (a.npad & 63) != 0 || G * Mc > kSmallT) {
    if (tid == 0) atomicOr(a.status, kErrBadLaunch);
    return;
  }
  if (tid == 0) {
    for (int b = 0; b < 4; ++b) mbar_init(&full[b], 1);
    fence_mbar_init();
    for (int b = 0; b < 4; ++b) mbar_arrive_expect_tx(&full[b], RF * 16);
  }
  const int S = a.rk ? 4 : 1, J = S * a.T;

  // Summing role: target slt, source records sg, sg + G, ...
  const int slt = tid % Mc, sg = tid / Mc;
  const bool sums = sg < G;
  const int si = rank * Mc + slt;
  // Updating role: coordinate k of target lt; part 0 holds q and alpha, part
  // 1 holds p and beta (neighbouring lanes, so the two exchange by shuffle).
  // FP64 in record units: kq q, p, alpha, kappa beta.
  const int part = tid & 1, k = (tid >> 1) % D, lt = (tid >> 1) / D;
  const bool own = lt < Mc;
  const int i = rank * Mc + lt;
  const bool live = own && i < a.n;
  const int tt = D * i + k;
  float* const rec = reinterpret_cast<float*>(stage + (lt >> 1) * D) + 2 * D * part + 2 * k + (lt & 1);
  // Sending role: float4 f of the staged records to CTAs peer, peer + dp, ...
  const int sf = tid % nf, speer = tid / nf, dp = kSmallT / nf;

  // The new records of this CTA's landmarks to buffer b of every CTA, and to
  // a trajectory slot.
  const auto publish = [&](int b, float4* slot) {
    __syncthreads();  // stage is complete
    const float4 v = stage[sf];
    const uint32_t to = smem_u32(buf(b) + rank * nf + sf), bar = smem_u32(&full[b]);
    if (speer < dp)
      for (int peer = speer; peer < kSmallC; peer += dp) st_async_f4(dsmem_addr(to, peer), v, dsmem_addr(bar, peer));
    if (slot && speer == 0) slot[rank * nf + sf] = v;
  };
  // Wait until buffer b holds every CTA's records.  An expired wait is
  // reported and ends the waiting, not the sequence of cluster barriers.
  bool ok = true;
  unsigned phase = 0;  // bit b: the phase of full[b]
  const auto receive = [&](int b) {
    if (ok && !mbar_wait_cluster(&full[b], (phase >> b) & 1u)) {
      ok = false;
      atomicOr(a.status, kErrTimeout);
    }
    phase ^= 1u << b;
    // Armed again before this CTA's next records leave, which every sender
    // into this buffer waits for.
    if (ok && tid == 0) mbar_arrive_expect_tx(&full[b], RF * 16);
  };
  // Pair sums of the forward step at the state in Q; then this thread's sum:
  // sum g p (part 0) or sum c g d~ (part 1) of its coordinate.
  const auto ham = [&](const float4* Q) -> double {
    if (sums) {
      const float* r = reinterpret_cast<const float*>(Q + (si >> 1) * D) + (si & 1);
      float2 q[D], p[D], aF[D], aG[D];
#pragma unroll
      for (int c = 0; c < D; ++c) {
        q[c] = dup(-r[2 * c]);
        p[c] = dup(r[2 * D + 2 * c]);
        aF[c] = aG[c] = make_float2(0.f, 0.f);
      }
#pragma unroll 4
      for (int x = sg; x < recs; x += G) {
        float2 v[2 * D];
        rec_split<D>(Q + x * D, v);
        fwd_record<D>(q, p, v, aF, aG);
      }
#pragma unroll
      for (int c = 0; c < D; ++c) {
        red[(c * G + sg) * Mc + slt] = __fadd_rn(aF[c].x, aF[c].y);
        red[((D + c) * G + sg) * Mc + slt] = __fadd_rn(aG[c].x, aG[c].y);
      }
    }
    __syncthreads();
    double v[1] = {0.0};
    const float* const r[1] = {red + (part * D + k) * G * Mc + lt};
    if (own) sum_groups<1>(r, G, Mc, v);
    return v[0];
  };

  // The caller's arrays: FP64 state of the owned coordinate, record slot 0.
  double s = 0.0, tgt = 0.0;
  if (live) {
    s = part ? (a.p64_in ? a.p64_in[tt] : (a.p ? static_cast<double>(a.p[tt]) : 0.0))
             : a.kq * static_cast<double>(a.q[tt]);
    if (a.tgt) tgt = a.tgt[tt];
    if (!isfinite(s) || !isfinite(tgt)) atomicOr(a.status, kErrNonFinite);
    if (a.t64 && !part) a.t64[tt] = tgt;
  }
  const auto state_rec = [&](double x) { return part ? static_cast<float>(x) : -static_cast<float>(x); };
  const auto adj_rec = [&](double x) { return part ? -static_cast<float>(x) : static_cast<float>(x); };
  if (own) *rec = state_rec(s);
  __syncwarp();
  cluster_sync();  // every CTA has started, its barriers are armed
  publish(0, a.traj);

  // ---- forward sweep
  // (d/dt) of the state in record units = cf times the part's sum.
  const double cf = part ? a.kappa : a.kq, cdt = cf * a.dt;
  double adj = 0.0, acc = 0.0, h0 = 0.0, hc = 0.0, mc = 0.0;
  for (int j = 0; j < J; ++j) {
    const int st = a.rk ? (j & 3) : 0;
    receive(j & 1);
    const double mine = ham(buf(j & 1));
    const bool last = j == J - 1;
    if (j == 0) {
      // Hq = -kappa sum for the owner of q, Hp for the owner of p;
      // H0 = 1/2 sum p . Hp
      h0 = __shfl_xor_sync(0xffffffffu, mine, 1);
      if (!part) h0 *= -a.kappa;
      if (live && part) hc = 0.5 * s * h0;
    }
    if (live) {
      double x;  // the next state's coordinate
      if (a.rk) {
        const double f = cf * mine;
        if (st == 0) acc = f;
        else if (st < 3) acc += 2.0 * f;
        if (st < 3) {
          x = s + (st == 2 ? 1.0 : 0.5) * a.dt * f;
        } else {
          x = s = s + a.dt / 6.0 * (acc + f);
        }
      } else {
        x = s = fma(cdt, mine, s);
      }
      if (!isfinite(x)) atomicOr(a.status, kErrNonFinite);
      *rec = state_rec(x);
      if (last && a.kind == 1 && !a.h_end) {  // loss and adjoint of the end state
        if (part == 0) {
          const double r = s / a.kq - tgt;
          mc = r * r;
          adj = 2.0 * a.lambda * r;
        }
        *rec = adj_rec(a.adj_scale * adj);
      }
    }
    if (!last || (a.kind == 1 && a.h_end))
      publish((j + 1) & 1, a.traj + static_cast<size_t>(j + 1) * a.slot);
  }
  if (a.kind == 1 && a.h_end) {
    // The end state's kinetic term and the adjoint that starts from it:
    // alpha = 2 lambda (q(1) - target) + Hq, beta = Hp.
    receive(J & 1);
    const double mine = ham(buf(J & 1));
    const double other = __shfl_xor_sync(0xffffffffu, mine, 1);
    hc = 0.0;
    if (live) {
      if (part) {
        adj = a.kappa * other;
        hc = 0.5 * s * other;
      } else {
        const double r = s / a.kq - tgt;
        mc = r * r;
        adj = 2.0 * a.lambda * r - a.kappa * other;
      }
      if (!isfinite(adj)) atomicOr(a.status, kErrNonFinite);
      *rec = adj_rec(a.adj_scale * adj);
    }
  }
  const double bh = block_sum_f64(hc, sh);
  const double bm = block_sum_f64(mc, sh);
  if (tid == 0) {
    st_dsmem_f64(dsmem_addr(smem_u32(&clsum[0][rank]), 0), bh);
    st_dsmem_f64(dsmem_addr(smem_u32(&clsum[1][rank]), 0), bm);
  }
  __syncwarp();
  cluster_sync();  // the sums have reached rank 0, the trajectory is visible to the cluster
  if (a.kind == 1) publish(2, nullptr);
  if (rank == 0 && tid == 0) {
    double h = 0.0, m = 0.0;
    for (int c = 0; c < kSmallC; ++c) {
      h += clsum[0][c];
      m += clsum[1][c];
    }
    a.scalars[a.h_end && a.kind == 1 ? 2 : 0] = h;
    if (a.kind == 1) a.scalars[1] = h + a.lambda * m;
  }
  if (a.kind == 0) {
    if (live) {
      const double v = part ? s : s / a.kq;
      (part ? a.p64 : a.q64)[tt] = v;
      float* o = part ? a.out_b : a.out_a;
      if (o) o[tt] = static_cast<float>(v);
    }
    __syncwarp();
    cluster_sync();  // after an expired wait records may still be on their way here
    return;
  }

  // ---- reverse sweep: launch r uses the state of record slot J-1-r
  double y = 0.0;
  for (int r = 0; r < J; ++r) {
    const int j = J - 1 - r, st = a.rk ? (j & 3) : 0;
    // The state of the next launch, from its slot into the idle buffer,
    // in flight during the sums.  All threads left that buffer before the
    // last CTA barrier, and no more records are sent to it.
    constexpr int kNx = (kSmallNpad / 2 * D + kSmallT - 1) / kSmallT;
    float4 nx[kNx];
    const float4* nsl = a.traj + static_cast<size_t>(j - 1) * a.slot;
    if (j > 0) {
#pragma unroll
      for (int u = 0; u < kNx; ++u)
        if (tid + u * kSmallT < RF) nx[u] = __ldcg(nsl + tid + u * kSmallT);
    }
    receive(2 + (r & 1));
    const float4* Q = buf(j & 1);
    const float4* A = buf(2 + (r & 1));
    if (sums) {
      const float* rq = reinterpret_cast<const float*>(Q + (si >> 1) * D) + (si & 1);
      const float* ra = reinterpret_cast<const float*>(A + (si >> 1) * D) + (si & 1);
      float2 q[D], p[D], al[D], be[D], a1[D], a2[D], bb[D];
#pragma unroll
      for (int c = 0; c < D; ++c) {
        q[c] = dup(-rq[2 * c]);
        p[c] = dup(rq[2 * D + 2 * c]);
        al[c] = dup(ra[2 * c]);
        be[c] = dup(-ra[2 * D + 2 * c]);
        a1[c] = a2[c] = bb[c] = make_float2(0.f, 0.f);
      }
#pragma unroll 2
      for (int x = sg; x < recs; x += G) {
        float2 v[2 * D], w[2 * D];
        rec_split<D>(Q + x * D, v);
        rec_split<D>(A + x * D, w);
        bwd_record<D>(q, p, al, be, v, w, a1, a2, bb);
      }
#pragma unroll
      for (int c = 0; c < D; ++c) {
        red[(c * G + sg) * Mc + slt] = __fadd_rn(a1[c].x, a1[c].y);
        red[((D + c) * G + sg) * Mc + slt] = __fadd_rn(a2[c].x, a2[c].y);
        red[((2 * D + c) * G + sg) * Mc + slt] = __fadd_rn(bb[c].x, bb[c].y);
      }
    }
    if (j > 0) {
      float4* nb = buf((j - 1) & 1);
#pragma unroll
      for (int u = 0; u < kNx; ++u)
        if (tid + u * kSmallT < RF) nb[tid + u * kSmallT] = nx[u];
    }
    __syncthreads();
    if (live) {
      // dalpha = kq A1 - kappa A2 (part 0), kappa dbeta = kappa B (part 1):
      // two sums for part 0, B and A2 (unused) for part 1.
      double t[2];
      const float* const rr[2] = {red + (part * 2 * D + k) * G * Mc + lt, red + (D + k) * G * Mc + lt};
      sum_groups<2>(rr, G, Mc, t);
      const double v = part ? a.kappa * t[0] : a.kq * t[0] - a.kappa * t[1];
      double x;  // the adjoint record's value
      if (a.rk) {
        // J(Y_s)^T kbar_s summed over the stages; the next stage adjoint
        // kbar_{s-1} = dt b_{s-1} w + c_s dt v (as in the step kernels).
        y = (st == 3 ? adj : y) + v;
        if (!isfinite(y)) atomicOr(a.status, kErrNonFinite);
        if (st > 0) {
          x = (st == 1 ? 1.0 / 6.0 : 1.0 / 3.0) * a.dt * adj + (st == 3 ? 1.0 : 0.5) * a.dt * v;
        } else {
          adj = y;
          x = a.dt / 6.0 * adj;
        }
      } else {
        x = adj = fma(a.dt, v, adj);
        if (!isfinite(x)) atomicOr(a.status, kErrNonFinite);
      }
      *rec = adj_rec(x);
    }
    if (j > 0) publish(2 + ((r + 1) & 1), nullptr);
  }
  if (live) {
    const double gr = (part ? adj / a.kappa : adj) + (a.h_end ? 0.0 : h0);
    float* o = part ? a.out_a : a.out_b;  // dL/dp0, dL/dq0
    if (o) o[tt] = static_cast<float>(gr);
    if (part && a.gp64) a.gp64[tt] = gr;
  }
  __syncwarp();
  cluster_sync();  // after an expired wait records may still be on their way here
}

size_t small_smem(int npad, int D, int groups) {
  const int RF = npad / 2 * D, Mc = npad / kSmallC, nf = Mc / 2 * D;
  return sizeof(float4) * (4 * static_cast<size_t>(RF) + nf) + sizeof(float) * 3 * D * groups * Mc;
}

std::mutex g_small_mu;
std::map<int, bool> g_small_ok;  // device -> one such cluster fits the device

cudaError_t prepare_small(void (*kern)(SmallArgs), int D) {
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(small_smem(kSmallNpad, D, kSmallT / (kSmallNpad / kSmallC))) + 4096);
  return e;
}

void small_launch_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* at, size_t smem, cudaStream_t st) {
  cfg = {};
  cfg.gridDim = dim3(kSmallC);
  cfg.blockDim = dim3(kSmallT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kSmallC;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
}

}  // namespace

bool small_supported() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  std::lock_guard<std::mutex> lk(g_small_mu);
  const auto it = g_small_ok.find(dev);
  if (it != g_small_ok.end()) return it->second;
  bool ok = prepare_small(k_small_sweep<3>, 3) == cudaSuccess && prepare_small(k_small_sweep<2>, 2) == cudaSuccess;
  if (ok) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[1];
    small_launch_config(cfg, at, small_smem(kSmallNpad, 3, kSmallT / (kSmallNpad / kSmallC)), nullptr);
    int clusters = 0;
    ok = cudaOccupancyMaxActiveClusters(&clusters, k_small_sweep<3>, &cfg) == cudaSuccess && clusters > 0;
  }
  if (!ok) cudaGetLastError();
  g_small_ok[dev] = ok;
  return ok;
}

cudaError_t launch_small_sweep(const SmallArgs& args, int dim, cudaStream_t st) {
  SmallArgs a = args;
  const int Mc = a.npad / kSmallC;
  // At least four records a thread: fewer would only lengthen the reduction.
  a.groups = std::max(1, std::min(kSmallT / Mc, a.npad / 2 / 4));
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[1];
  small_launch_config(cfg, at, small_smem(a.npad, dim, a.groups), st);
  return dim == 2 ? cudaLaunchKernelEx(&cfg, k_small_sweep<2>, a) : cudaLaunchKernelEx(&cfg, k_small_sweep<3>, a);
}

}  // namespace gs
