// Spatial order of a problem's landmarks, and packing in that order.
//
// g = 2^-r2 is exactly zero in the kernels' arithmetic once r2 > 126 (ex2
// flushes results below 2^-126), so every term of such a pair is exactly
// zero.  With landmarks stored along a space-filling curve, a run of kGran
// consecutive ones is compact, and the step kernels leave out the runs whose
// box lies that far from their targets' box (step_kernels.cu): the sums keep
// every non-zero term.
//
// k_codes: the place of each landmark on a Hilbert curve (J. Skilling,
// "Programming the Hilbert curve", 2004), in cells of a quarter of the
// prescaled unit around landmark 0.  k_rank_pack: each landmark's rank in
// (code, index) order by counting, then the pack of the caller's arrays at
// that rank.  Counting reads N codes per landmark, about three integer instructions
// a pair against 51 for one time step's sums, needs no scratch and
// no further launch, and gives the same order on every run.
#include <algorithm>

#include "gs_device.cuh"
#include "gs_internal.h"

namespace gs {
namespace {

constexpr int kOT = 256;
constexpr int kLanes = 8;  // lanes that count for two landmarks
constexpr int kTile4 = 8 * kOT;  // uint4 of codes staged at a time (32 KB)

template <int D>
__device__ __forceinline__ unsigned hilbert_code(unsigned (&x)[D]) {
  constexpr int B = 30 / D;
  for (unsigned q = 1u << (B - 1); q > 1; q >>= 1) {
    const unsigned m = q - 1;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      if (x[k] & q) {
        x[0] ^= m;
      } else {
        const unsigned t = (x[0] ^ x[k]) & m;
        x[0] ^= t;
        x[k] ^= t;
      }
    }
  }
#pragma unroll
  for (int k = 1; k < D; ++k) x[k] ^= x[k - 1];
  unsigned t = 0;
  for (unsigned q = 1u << (B - 1); q > 1; q >>= 1)
    if (x[D - 1] & q) t ^= q - 1;
  unsigned code = 0;
#pragma unroll
  for (int b = B - 1; b >= 0; --b)
#pragma unroll
    for (int k = 0; k < D; ++k) code = (code << 1) | (((x[k] ^ t) >> b) & 1u);
  return code;
}

// codes[0, round_up(n, 32)) (the padding sorts last); boxes[0, nbox4) <- 0.
template <int D>
__global__ void __launch_bounds__(kOT) k_codes(const float* q, int n, float kq, unsigned* codes, uint4* boxes,
                                              size_t nbox4) {
  const size_t t0 = blockIdx.x * static_cast<size_t>(kOT) + threadIdx.x;
  for (size_t b = t0; b < nbox4; b += static_cast<size_t>(gridDim.x) * kOT) boxes[b] = make_uint4(0u, 0u, 0u, 0u);
  const int np = (n + 31) & ~31;
  for (size_t i = t0; i < static_cast<size_t>(np); i += static_cast<size_t>(gridDim.x) * kOT) {
    if (i >= static_cast<size_t>(n)) {
      codes[i] = 0x7fffffffu;
      continue;
    }
    constexpr int B = 30 / D;
    unsigned x[D];
#pragma unroll
    for (int k = 0; k < D; ++k) {
      const float c = 4.f * kq * (q[D * i + k] - q[k]) + static_cast<float>(1 << (B - 1));
      x[k] = static_cast<unsigned>(fminf(fmaxf(c, 0.f), static_cast<float>((1 << B) - 1)));  // NaN: 0
    }
    codes[i] = hilbert_code<D>(x);
  }
}

// Whether nearly all of the packed state's pairs are in reach, from 16 tiles of
// 64 landmarks against 256 runs, spread evenly.  Then testing runs and
// copying them piecemeal costs more than it saves, and the step kernels stream
// every source.  The lines: at 16384 landmarks and more the test is a small part
// of a CTA's time and pays from 5 % of the pairs on (sigma = 0.1 at 38785:
// 60.3 against 66.2 ms); at 5000 to 10000 it costs 4-13 % of a step, saved from 15 %
// on.
template <int D>
__device__ __forceinline__ bool mostly_in_reach(const unsigned* boxes, int npad) {
  const int nrun = npad / kGran, ntile = npad / 64;
  const int tiles = min(ntile, 16), runs = min(nrun, 256);
  int in = 0;
  for (int x = threadIdx.x; x < tiles * runs; x += kOT) {
    const int t = static_cast<int>(static_cast<long long>(x / runs) * ntile / tiles);
    const int r = static_cast<int>(static_cast<long long>(x % runs) * nrun / runs);
    RunBox<D> b = run_box<D>(load_box(boxes, 2 * t));
    const RunBox<D> b1 = run_box<D>(load_box(boxes, 2 * t + 1));
#pragma unroll
    for (int k = 0; k < D; ++k) {
      b.hi[k] = fmaxf(b.hi[k], b1.hi[k]);
      b.lo[k] = fmaxf(b.lo[k], b1.lo[k]);
    }
    in += in_reach(b, run_box<D>(load_box(boxes, r)));
  }
  __shared__ int total;
  if (threadIdx.x == 0) total = 0;
  __syncthreads();
  atomicAdd(&total, in);
  __syncthreads();
  return total > (npad >= 16384 ? 0.95f : 0.85f) * static_cast<float>(tiles * runs);
}

template <int D>
__device__ __forceinline__ void rank_pack(const PackArgs& a, const unsigned* codes, int* perm, unsigned* boxes) {
  // Eight lanes count for landmarks 2 g and 2 g + 1, each over every eighth
  // group of four codes.
  const int gt = blockIdx.x * kOT + threadIdx.x;
  const int i0 = 2 * (gt / kLanes), lane = gt % kLanes;
  // Codes pass through shared memory, a tile at a time: from L2 directly, few
  // loads in flight made this 15 us at N = 4096.
  __shared__ int4 tile[kTile4];
  const int c0 = i0 < a.n ? static_cast<int>(codes[i0]) : 0, c1 = i0 + 1 < a.n ? static_cast<int>(codes[i0 + 1]) : 0;
  int n0 = 0, n1 = 0;
  const int4* c4 = reinterpret_cast<const int4*>(codes);
  const int n4 = ((a.n + 31) & ~31) / 4;
  for (int t0 = 0; t0 < n4; t0 += kTile4) {
    const int len = min(kTile4, n4 - t0);
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kTile4 / kOT; ++u)
      if (threadIdx.x + u * kOT < len) tile[threadIdx.x + u * kOT] = c4[t0 + threadIdx.x + u * kOT];
    __syncthreads();
    // Codes before a landmark's own count, equal ones only at a smaller index
    // (i0 is even, so both landmarks lie in one group of four); codes have 30
    // bits, so the sign of a difference tells.
#pragma unroll 4
    for (int j = lane; j < len; j += kLanes) {
      const int4 c = tile[j];
      const int lt = 4 * (t0 + j) + 3 < i0 ? 1 : 0;
      const int h0 = c0 + lt, h1 = c1 + lt;
      n0 += ((c.x - h0) >> 31) + ((c.y - h0) >> 31) + ((c.z - h0) >> 31) + ((c.w - h0) >> 31);
      n1 += ((c.x - h1) >> 31) + ((c.y - h1) >> 31) + ((c.z - h1) >> 31) + ((c.w - h1) >> 31);
    }
  }
  n0 = -n0;
  n1 = -n1;
  if ((i0 >> 2) % kLanes == lane && i0 < a.n) {
    for (int j = i0 & ~3; j < i0; ++j) n0 += static_cast<int>(codes[j]) == c0;
    for (int j = i0 & ~3; j <= i0; ++j) n1 += static_cast<int>(codes[j]) == c1;
  }
#pragma unroll
  for (int o = 1; o < kLanes; o <<= 1) {
    n0 += __shfl_xor_sync(0xffffffffu, n0, o);
    n1 += __shfl_xor_sync(0xffffffffu, n1, o);
  }
  // Lanes 0..D-1 pack the first landmark's coordinates, lanes 4.. the second's.
  const int i = i0 + lane / 4, k = lane % 4;
  if (k >= D) return;
  if (i >= a.n) {
    if (i < a.npad) {  // the padding of the record slot
      float* rec = reinterpret_cast<float*>(a.qp + (i >> 1) * D) + 2 * k + (i & 1);
      rec[0] = rec[2 * D] = 0.f;
    }
    return;
  }
  const int r = lane / 4 ? n1 : n0;
  if (k == 0) perm[r] = i;
  const int src = D * i + k, dst = D * r + k;
  const float q = a.q[src];
  const double p = a.p64_in ? a.p64_in[src] : (a.p ? (double)a.p[src] : 0.0);
  const float tg = a.tgt ? a.tgt[src] : 0.f;
  if (!isfinite(q) || !isfinite(p) || !isfinite(tg)) atomicOr(a.status, kErrNonFinite);
  a.q64[dst] = q;
  a.p64[dst] = p;
  if (a.t64) a.t64[dst] = tg;
  float* rec = reinterpret_cast<float*>(a.qp + (r >> 1) * D) + 2 * k + (r & 1);
  const float v = -(float)(a.kq * (double)q);
  rec[0] = v;
  rec[2 * D] = (float)p;
  box_add(boxes, r, k, v);
}

template <int D>
__global__ void __launch_bounds__(kOT) k_rank_pack(PackArgs a, const unsigned* codes, int* perm, unsigned* boxes,
                                                  int* dense) {
  __shared__ int am_last;
  pdl_wait();  // the codes
  rank_pack<D>(a, codes, perm, boxes);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) am_last = atomicAdd(dense, 1) == static_cast<int>(gridDim.x) - 1;
  __syncthreads();
  if (!am_last) return;
  __threadfence();
  const bool d = mostly_in_reach<D>(boxes, a.npad);
  if (threadIdx.x == 0) {
    dense[1] = d;
    dense[0] = 0;
  }
}

}  // namespace

cudaError_t launch_order_pack(const PackArgs& a, unsigned* codes, int* perm, unsigned* boxes, size_t nbox, int* dense,
                              cudaStream_t st) {
  const size_t nbox4 = nbox / 4;
  const int grid = static_cast<int>(std::min<size_t>(std::max<size_t>((a.n + 31 + kOT) / kOT, nbox4 / (4 * kOT)), 1216));
  const long long threads = static_cast<long long>(a.npad) / 2 * kLanes;
  const int rgrid = static_cast<int>((threads + kOT - 1) / kOT);
  uint4* b4 = reinterpret_cast<uint4*>(boxes);
  const float kq = static_cast<float>(a.kq);
  if (a.dim == 2)
    k_codes<2><<<grid, kOT, 0, st>>>(a.q, a.n, kq, codes, b4, nbox4);
  else
    k_codes<3><<<grid, kOT, 0, st>>>(a.q, a.n, kq, codes, b4, nbox4);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(rgrid);
  cfg.blockDim = dim3(kOT);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const unsigned* const cc = codes;
  return a.dim == 2 ? cudaLaunchKernelEx(&cfg, k_rank_pack<2>, a, cc, perm, boxes, dense)
                    : cudaLaunchKernelEx(&cfg, k_rank_pack<3>, a, cc, perm, boxes, dense);
}

}  // namespace gs
