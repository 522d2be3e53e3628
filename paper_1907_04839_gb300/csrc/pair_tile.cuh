// Per-thread target tiles of the StepForward / StepBackward pair sums, and
// the TMA pipeline that streams a range of sources through shared memory.
// Both the split-partial kernels (pair_kernels.cu) and the fused step kernels
// (step_kernels.cu) are built from these pieces.
//
// Packed arithmetic.  Sources sit in memory as pair records: two landmarks
// interleaved per coordinate (layout in gs_internal.h; D float4 per record
// for landmarks in D = 3 or 2 dimensions).  The inner loop uses
// the sm_100+ paired FP32 instructions (__fadd2_rn, __fmul2_rn, __ffma2_rn).
// Each instruction applies one target to two sources, which halves the issue
// slots spent on FP32 work.  Positions are stored negated, so q_i - q_j is a
// single paired add.  The Gaussian is one MUFU ex2 per pair, on prescaled
// coordinates.
//
// A thread holds R targets in registers.  The threads of a CTA form one or
// more warp groups; each group holds the same targets (base + r*TG, r < R,
// TG threads per group) and takes its own share of every staged chunk of
// sources, so a CTA with W groups splits its sources W ways.  The whole warp
// reads the same source record, so the shared-memory load is a broadcast.
// Sums are plain FP32 over a sub-block of at most kSub sources, then the two
// halves of each paired accumulator are added and folded into a Kahan (sum,
// compensation) pair.
#pragma once

#include "gs_device.cuh"
#include "gs_internal.h"

namespace gs {

// Sources per plain-FP32 sub-block before a Kahan fold: one staged chunk.
// Measured on GB300 in whole gradients (T = 20), 128 against 64: -1.7 % at
// N = 4096 and 16384, both kernels.
constexpr int kSub = 128;
constexpr int kUnroll = 8;  // split lengths are multiples of this

// kStages chunk buffers for NA record arrays (kChunk sources = kChunk/2
// records of D float4 each, D the dimension of the landmarks).  The
// mbarriers live outside (struct Pipe), so this memory can be reused once
// the last chunk has been consumed.
template <int NA, int D = 3>
struct StageBuf {
  float4 buf[kStages][NA][D * kChunk / 2];
  float4 ahead[4 * D];  // a loop that loads ahead may read (not use) this far past the last stage
};

// full[s]: the bulk copies of the chunk in stage s have landed (transaction
// count).  empty[s]: every warp has finished reading stage s (one arrival per
// warp).  abort: set by a thread whose wait expired.
struct Pipe {
  uint64_t full[kStages];
  uint64_t empty[kStages];
  int abort;
};

__device__ __forceinline__ void pipe_init(Pipe& p, int warps) {
#pragma unroll
  for (int s = 0; s < kStages; ++s) {
    mbar_init(&p.full[s], 1);
    mbar_init(&p.empty[s], warps);
  }
  p.abort = 0;
  fence_mbar_init();
}

// Issue the bulk copies of chunk c (NA record arrays) into stage c % kStages (of
// the absolute chunk number, where it differs).
// Source offsets and lengths are even, so records are copied whole.
template <int NA, int D>
__device__ __forceinline__ void issue_chunk(StageBuf<NA, D>& st, Pipe& pp, const float4* const* src, int j0, int j1,
                                            int c, int abs = -1) {
  const int off = j0 + c * kChunk;
  const int len = min(kChunk, j1 - off);
  const unsigned bytes = static_cast<unsigned>(len) * (16 * D / 2);
  const int s = (abs < 0 ? c : abs) % kStages;
  uint64_t* bar = &pp.full[s];
  mbar_arrive_expect_tx(bar, NA * bytes);
#pragma unroll
  for (int a = 0; a < NA; ++a) bulk_g2s(&st.buf[s][a][0], src[a] + (off / 2) * D, bytes, bar);
}

// Stream sources [j0, j1) through the stage ring.  Warp group `group` of
// `groups` consumes its share of each chunk: tile.consume(buffers, lo, hi)
// with [lo, hi) a contiguous piece, in multiples of 8 sources, of the chunk's
// sources.  The whole CTA calls this; thread 0 issues the copies.  Warps move on to the next chunk as soon as it has landed: a warp
// releases a stage through empty[s], and thread 0 refills a stage only after
// every warp has released it.  Returns false in every thread if a wait
// expired; the expiry is recorded in *status, and every copy still in flight
// has been waited for (bounded) before return.  Ends with a CTA barrier.
template <int NA, int Groups = 1, int D = 3, class Tile>
__device__ bool stream_sources(StageBuf<NA, D>& st, Pipe& pp, const float4* const* src, int j0, int j1, Tile& tile,
                               unsigned* status, int group = 0) {
  const int tid = threadIdx.x;
  const int nch = j1 > j0 ? (j1 - j0 + kChunk - 1) / kChunk : 0;
  int issued = 0;
  if (tid == 0) {
    for (; issued < nch && issued < kStages; ++issued) issue_chunk<NA, D>(st, pp, src, j0, j1, issued);
  }
  volatile int* abort = &pp.abort;
  for (int c = 0; c < nch; ++c) {
    const int s = c % kStages;
    if (*abort) break;
    if (!mbar_wait(&pp.full[s], (c / kStages) & 1)) {
      *abort = 1;
      break;
    }
    const float4* bufs[NA];
#pragma unroll
    for (int a = 0; a < NA; ++a) bufs[a] = st.buf[s][a];
    const int len = min(kChunk, j1 - (j0 + c * kChunk));
    if constexpr (Groups == 1) {
      tile.consume(bufs, 0, len);
    } else {
      const int piece = (len + kUnroll * Groups - 1) / (kUnroll * Groups) * kUnroll;
      const int lo = min(group * piece, len);
      tile.consume(bufs, lo, min(lo + piece, len));
    }
    __syncwarp();
    if ((tid & 31) == 0) mbar_arrive(&pp.empty[s]);
    if (tid == 0 && c + kStages < nch) {
      // Refill stage s with chunk c + kStages once every warp has released it.
      if (mbar_wait(&pp.empty[s], (c / kStages) & 1)) {
        fence_proxy_async_smem();
        issue_chunk<NA, D>(st, pp, src, j0, j1, c + kStages);
        issued = c + kStages + 1;
      } else {
        *abort = 1;
      }
    }
  }
  __syncthreads();
  if (*abort) {
    if (tid == 0) {
      atomicOr(status, kErrTimeout);
      // Let every copy that was issued land before the CTA reuses or leaves
      // this memory: the last kStages chunks issued are the only ones that
      // can still be in flight.
      for (int d = max(0, issued - kStages); d < issued; ++d)
        (void)mbar_wait(&pp.full[d % kStages], (d / kStages) & 1);
    }
    __syncthreads();
    return false;
  }
  return true;
}

// Runs of a culling kernel's list per window: half a KB, so that the one-warp
// reverse CTAs still fit eight to an SM (seven were 20 % slower at N = 8192).
constexpr int kListCap = 128;
constexpr int kGranPerChunk = kChunk / kGran;
// Copy runs list[4c .. 4c+3] (fewer at the end of the list) of every record
// array into the stage of absolute chunk `abs`.
template <int NA, int D>
__device__ __forceinline__ void issue_runs(StageBuf<NA, D>& st, Pipe& pp, const float4* const* src, const unsigned* list,
                                           int cnt, int c, int abs) {
  constexpr int kRunF4 = kGran / 2 * D;  // float4 per run and array
  const int m = min(kGranPerChunk, cnt - c * kGranPerChunk);
  const int s = abs % kStages;
  uint64_t* bar = &pp.full[s];
  mbar_arrive_expect_tx(bar, NA * m * kRunF4 * 16);
  for (int g = 0; g < m; ++g) {
    const size_t off = static_cast<size_t>(list[c * kGranPerChunk + g]) * kRunF4;
#pragma unroll
    for (int a = 0; a < NA; ++a) bulk_g2s(&st.buf[s][a][g * kRunF4], src[a] + off, kRunF4 * 16, bar);
  }
}

// stream_sources over nsrc sources: those from first on, or (first < 0) the
// runs of list.  base: chunks the CTA has streamed before (the stage ring and
// its barrier phases run on); the caller adds the chunks of this call.  One
// warp group.  One loop for both: two copies of it cost 17 registers and 8 % of
// the forward step.
template <int NA, int D, class Tile>
__device__ bool stream_runs(StageBuf<NA, D>& st, Pipe& pp, const float4* const* src, const unsigned* list, int first,
                            int nsrc, int base, Tile& tile, unsigned* status) {
  const int tid = threadIdx.x;
  const int nch = (nsrc + kChunk - 1) / kChunk;
  const auto issue = [&](int c) {
    if (first >= 0)
      issue_chunk<NA, D>(st, pp, src, first, first + nsrc, c, base + c);
    else
      issue_runs<NA, D>(st, pp, src, list, nsrc / kGran, c, base + c);
  };
  int issued = 0;
  if (tid == 0) {
    for (; issued < nch && issued < kStages; ++issued) issue(issued);
  }
  volatile int* abort = &pp.abort;
  for (int c = 0; c < nch; ++c) {
    const int s = (base + c) % kStages;
    const unsigned ph = ((base + c) / kStages) & 1;
    if (*abort) break;
    if (!mbar_wait(&pp.full[s], ph)) {
      *abort = 1;
      break;
    }
    const float4* bufs[NA];
#pragma unroll
    for (int a = 0; a < NA; ++a) bufs[a] = st.buf[s][a];
    tile.consume(bufs, 0, min(kChunk, nsrc - c * kChunk));
    __syncwarp();
    if ((tid & 31) == 0) mbar_arrive(&pp.empty[s]);
    if (tid == 0 && c + kStages < nch) {
      if (mbar_wait(&pp.empty[s], ph)) {
        fence_proxy_async_smem();
        issue(c + kStages);
        issued = c + kStages + 1;
      } else {
        *abort = 1;
      }
    }
  }
  __syncthreads();
  if (*abort) {
    if (tid == 0) {
      atomicOr(status, kErrTimeout);
      for (int d = max(0, issued - kStages); d < issued; ++d)
        (void)mbar_wait(&pp.full[(base + d) % kStages], ((base + d) / kStages) & 1);
    }
    __syncthreads();
    return false;
  }
  return true;
}

// Box of the M targets from tile0 on (whole runs; npad a multiple of a run).
template <int D, int M>
__device__ __forceinline__ RunBox<D> tile_box(const unsigned* boxes, int tile0, int nrun) {
  static_assert(M % kGran == 0, "tiles are whole runs");
  BoxWords w[M / kGran];
#pragma unroll
  for (int g = 0; g < M / kGran; ++g) w[g] = load_box(boxes, min(tile0 / kGran + g, nrun - 1));
  RunBox<D> t = run_box<D>(w[0]);
#pragma unroll
  for (int g = 1; g < M / kGran; ++g) {
    const RunBox<D> b = run_box<D>(w[g]);
#pragma unroll
    for (int k = 0; k < D; ++k) {
      t.hi[k] = fmaxf(t.hi[k], b.hi[k]);
      t.lo[k] = fmaxf(t.lo[k], b.lo[k]);
    }
  }
  return t;
}

// Runs [w0, w1) of CTA `rank` of C (its run m is run rank + m C): those in reach
// of box tbox() go to list.  One warp, 32 runs at a time, in bit-reversed
// order: neighbours on the curve land in different chunks, so that a target's
// near sources, which carry its sum, do not all add up in one plain-FP32
// sub-block.  Returns their count.
template <int D, class Box>
__device__ __forceinline__ int list_in_reach(const unsigned* boxes, Box tbox, int rank, int C, int w0, int w1,
                                             unsigned* list) {
  const unsigned lane = threadIdx.x & 31;
  const int mine = static_cast<int>(__brev(lane) >> 27);
  // the first boxes are on their way before the tile's are waited for
  const auto at = [&](int m) { return rank + min(m + mine, w1 - 1) * C; };
  BoxWords next = load_box(boxes, at(w0));
  const RunBox<D> t = tbox();
  int cnt = 0;
  for (int m = w0; m < w1; m += 32) {
    const RunBox<D> b = run_box<D>(next);
    if (m + 32 < w1) next = load_box(boxes, at(m + 32));
    const bool in = m + mine < w1 && in_reach(t, b);
    const unsigned v = __ballot_sync(0xffffffffu, in);
    if (in) list[cnt + __popc(v & ((1u << lane) - 1u))] = at(m);
    cnt += __popc(v);
  }
  return cnt;
}

// The two uses, compiled apart from the pair loops: inlined, they cost the
// loops up to 28 registers and, on a dense problem, 8 % of the forward step.
template <int D, int M>
__device__ __noinline__ int list_for_tile(const unsigned* boxes, int tile0, int nrun, int rank, int C, int w0, int w1,
                                          unsigned* list) {
  return list_in_reach<D>(boxes, [&] { return tile_box<D, M>(boxes, tile0, nrun); }, rank, C, w0, w1, list);
}

template <int D>
__device__ __noinline__ int list_for_box(const unsigned* boxes, RunBox<D> t, int rank, int C, int w0, int w1,
                                         unsigned* list) {
  return list_in_reach<D>(boxes, [&] { return t; }, rank, C, w0, w1, list);
}

// The pair sums of a tile over every C-th run of the sources, from run `rank`
// on, runs out of the tile's reach left out.  Interleaving gives the CTAs of
// the cluster nearly equal lists, as neighbours on the curve are in or out of
// reach together.  make(w0, w1, list) is
// list_for_tile or list_for_box, called by warp 0.  list: kListCap + 1 words of
// shared memory (the last holds the count).  dense: every source of [j0, j1)
// instead.  Ends with a CTA barrier.
template <int NA, int D, class Tile, class Make>
__device__ __forceinline__ void sum_in_reach(StageBuf<NA, D>& st, Pipe& pp, const float4* const* src, Make make,
                                             int nrun, int rank, int C, bool dense, int j0, int j1, Tile& tile,
                                             unsigned* list, unsigned* status) {
  const int mine = (nrun - rank + C - 1) / C;  // runs of this CTA
  int base = 0, w0 = 0;
  do {
    int nsrc = j1 - j0;
    if (!dense) {
      if (threadIdx.x < 32) {
        const int cnt = w0 < mine ? make(w0, min(w0 + kListCap, mine), list) : 0;
        if (threadIdx.x == 0) list[kListCap] = cnt;
      }
      __syncthreads();
      nsrc = static_cast<int>(list[kListCap]) * kGran;
    }
    if (!stream_runs<NA, D>(st, pp, src, list, dense ? j0 : -1, nsrc, base, tile, status)) return;
    base += (nsrc + kChunk - 1) / kChunk;
    w0 += kListCap;
  } while (!dense && w0 < mine);
}

__device__ __forceinline__ float2 dup(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 lo2(float4 v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(float4 v) { return make_float2(v.z, v.w); }

// Gaussian of two pairs at once from their squared prescaled distances.
__device__ __forceinline__ float2 gauss2(float2 r2) {
  return make_float2(ex2_approx(-r2.x), ex2_approx(-r2.y));
}

// Coordinate k (0..D-1) of landmark i from a pair-record array; field f
// selects the first (0) or second (1) quantity of the record.
template <int D = 3>
__device__ __forceinline__ float rec_get(const float4* rec, int i, int f, int k) {
  const float* r = reinterpret_cast<const float*>(rec + (i >> 1) * D);
  return __ldcg(r + 2 * D * f + 2 * k + (i & 1));
}

// The 2D float2 values of one pair record (D float4): value c < D is
// coordinate c of the first quantity, value D + c of the second, each for
// the record's two landmarks.
template <int D>
__device__ __forceinline__ void rec_split(const float4* rec, float2 (&v)[2 * D]) {
#pragma unroll
  for (int f = 0; f < D; ++f) {
    const float4 x = rec[f];
    v[2 * f] = lo2(x);
    v[2 * f + 1] = hi2(x);
  }
}

// U records at p.
template <int U, int D>
__device__ __forceinline__ void load_records(const float4* p, float4 (&x)[U][D]) {
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int f = 0; f < D; ++f) x[u][f] = p[u * D + f];
}

// Records that the 64-thread reverse CTAs' loop loads ahead of the ones in use
// where the grid has several waves (ordered sweeps, packed batches).  One warp's
// loop alone on a scheduler takes 102.8 instead of 109.0 cycles a record; the
// registers (96 to 119) decide what whole steps gain: 302 against 313 us at
// N = 16384, 1533 against 1593 at 38785; 32-thread CTAs lose (94.2 against 90.2
// at 8192), and so do one-wave grids (11.7 against 9.6 us at 1847, 29.5 against
// 28.5 at 4096).  The forward loop gained nothing in whole gradients (four
// ahead: 57.7 against 83.7 cycles alone, but 92 registers).
constexpr int kAhead = 2;

// One target against one source record (two sources) of StepForward.
// q, p: the target, duplicated; v[k] = -q~_j, v[D + k] = p_j; aF += g p_j,
// aG += c g d~.
template <int D>
__device__ __forceinline__ void fwd_record(const float2 (&q)[D], const float2 (&p)[D], const float2 (&v)[2 * D],
                                           float2 (&aF)[D], float2 (&aG)[D]) {
  float2 d[D];
#pragma unroll
  for (int k = 0; k < D; ++k) d[k] = __fadd2_rn(q[k], v[k]);
  float2 r2 = __fmul2_rn(d[0], d[0]);
#pragma unroll
  for (int k = 1; k < D; ++k) r2 = __ffma2_rn(d[k], d[k], r2);
  const float2 g = gauss2(r2);
  float2 cc = __fmul2_rn(p[0], v[D]);
#pragma unroll
  for (int k = 1; k < D; ++k) cc = __ffma2_rn(p[k], v[D + k], cc);
  const float2 w = __fmul2_rn(g, cc);
#pragma unroll
  for (int k = 0; k < D; ++k) aF[k] = __ffma2_rn(g, v[D + k], aF[k]);
#pragma unroll
  for (int k = 0; k < D; ++k) aG[k] = __ffma2_rn(w, d[k], aG[k]);
}

// One target against one source record of StepBackward.  v as above; w[k] =
// alpha_j, w[D + k] = -b~_j.  With m_j = alpha_j + t p_j (which B needs
// anyway), h = u + c t = alpha_i.p_j + p_i.m_j: 35 paired instructions instead
// of the 36 that forming u and c t apart takes (the loop is bound by the FP32
// pipe and its operand reads).  Whole gradients: 19.64 against 19.89 ms at
// N = 16384 (T = 40), 998 against 1006 us at 4096 (T = 20).
template <int D>
__device__ __forceinline__ void bwd_record(const float2 (&q)[D], const float2 (&p)[D], const float2 (&a)[D],
                                           const float2 (&b)[D], const float2 (&v)[2 * D], const float2 (&w)[2 * D],
                                           float2 (&a1)[D], float2 (&a2)[D], float2 (&bb)[D]) {
  float2 d[D], e[D], m[D];
#pragma unroll
  for (int k = 0; k < D; ++k) d[k] = __fadd2_rn(q[k], v[k]);
  float2 r2 = __fmul2_rn(d[0], d[0]);
#pragma unroll
  for (int k = 1; k < D; ++k) r2 = __ffma2_rn(d[k], d[k], r2);
  const float2 g = gauss2(r2);
  float2 cc = __fmul2_rn(p[0], v[D]);
#pragma unroll
  for (int k = 1; k < D; ++k) cc = __ffma2_rn(p[k], v[D + k], cc);
#pragma unroll
  for (int k = 0; k < D; ++k) e[k] = __fadd2_rn(b[k], w[D + k]);
  float2 t = __fmul2_rn(e[0], d[0]);
#pragma unroll
  for (int k = 1; k < D; ++k) t = __ffma2_rn(e[k], d[k], t);
#pragma unroll
  for (int k = 0; k < D; ++k) m[k] = __ffma2_rn(t, v[D + k], w[k]);
  float2 h = __fmul2_rn(a[0], v[D]);
#pragma unroll
  for (int k = 1; k < D; ++k) h = __ffma2_rn(a[k], v[D + k], h);
#pragma unroll
  for (int k = 0; k < D; ++k) h = __ffma2_rn(p[k], m[k], h);
  const float2 gc = __fmul2_rn(g, cc);
  const float2 gh = __fmul2_rn(g, h);
#pragma unroll
  for (int k = 0; k < D; ++k) a1[k] = __ffma2_rn(gc, e[k], a1[k]);
#pragma unroll
  for (int k = 0; k < D; ++k) a2[k] = __ffma2_rn(gh, d[k], a2[k]);
#pragma unroll
  for (int k = 0; k < D; ++k) bb[k] = __ffma2_rn(g, m[k], bb[k]);
}

// ---------------------------------------------------------------- StepForward tile
// Per target i:  Hp_i = sum_j g_ij p_j  and  G~_i = sum_j c_ij g_ij (q~_i - q~_j),
// with Hq_i = -kappa G~_i.  D = 3 (or 2 for planar landmarks) coordinates.
template <int R, int D = 3>
struct FwdTile {
  float2 q[R][D], p[R][D];  // target, duplicated
  float sF[R][D], cF[R][D], sG[R][D], cG[R][D];

  __device__ __forceinline__ void load(const float4* qp, int base, int stride, int npad) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int i = base + r * stride;
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const float qk = i < npad ? -rec_get<D>(qp, i, 0, k) : 0.f;
        const float pk = i < npad ? rec_get<D>(qp, i, 1, k) : 0.f;
        q[r][k] = dup(qk);
        p[r][k] = dup(pk);
        sF[r][k] = cF[r][k] = sG[r][k] = cG[r][k] = 0.f;
      }
    }
  }

  // Sources [lo, hi) of the staged chunk; lo is a multiple of 8.
  __device__ __forceinline__ void consume(const float4* const* bufs, int lo, int hi) {
    const float4* Q = bufs[0];
    for (int sb = lo; sb < hi; sb += kSub) {
      const int sl = min(kSub, hi - sb);
      float2 aF[R][D], aG[R][D];
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int k = 0; k < D; ++k) aF[r][k] = aG[r][k] = make_float2(0.f, 0.f);
      for (int jj = 0; jj < sl; jj += kUnroll) {
#pragma unroll
        for (int u = 0; u < kUnroll / 2; ++u) {
          float2 v[2 * D];  // v[k] = -q~_j, v[D + k] = p_j
          rec_split<D>(Q + ((sb + jj) / 2 + u) * D, v);
#pragma unroll
          for (int r = 0; r < R; ++r) fwd_record<D>(q[r], p[r], v, aF[r], aG[r]);
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int k = 0; k < D; ++k) {
          kahan_add(sF[r][k], cF[r][k], __fadd_rn(aF[r][k].x, aF[r][k].y));
          kahan_add(sG[r][k], cG[r][k], __fadd_rn(aG[r][k].x, aG[r][k].y));
        }
    }
  }

  // out[0..D) = Hp, out[D..2D) = Hq of target r, as double-single values.
  __device__ __forceinline__ void result(int r, float kappa, ds out[2 * D]) const {
#pragma unroll
    for (int k = 0; k < D; ++k) {
      out[k] = ds_from_kahan(sF[r][k], cF[r][k]);
      out[D + k] = ds_mul_f(ds_from_kahan(sG[r][k], cG[r][k]), -kappa);
    }
  }
};

// ---------------------------------------------------------------- StepBackward tile
// Sources carry q~ = kq q, p (QP records) and alpha, b~ = kappa beta (AB
// records).  Per pair:
//   d~ = q~_i - q~_j, g = 2^-|d~|^2, c = p_i.p_j, e~ = b~_i - b~_j,
//   t = e~.d~ (= s e.d), m_j = alpha_j + t p_j, h = u + c t = alpha_i.p_j + p_i.m_j,
//   A1 += g c e~,  A2 += g h d~,  B += g m_j;
// dalpha = kq A1 - kappa A2 and dbeta = B.
// U: records loaded ahead of the ones in use (0: none).
template <int R, int D = 3, int U = 0>
struct BwdTile {
  float2 q[R][D], p[R][D], a[R][D], b[R][D];
  float s1[R][D], c1[R][D], s2[R][D], c2[R][D], sB[R][D], cB[R][D];

  __device__ __forceinline__ void load(const float4* qp, const float4* ab, int base, int stride, int npad) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int i = base + r * stride;
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const bool in = i < npad;
        q[r][k] = dup(in ? -rec_get<D>(qp, i, 0, k) : 0.f);
        p[r][k] = dup(in ? rec_get<D>(qp, i, 1, k) : 0.f);
        a[r][k] = dup(in ? rec_get<D>(ab, i, 0, k) : 0.f);
        b[r][k] = dup(in ? -rec_get<D>(ab, i, 1, k) : 0.f);
        s1[r][k] = c1[r][k] = s2[r][k] = c2[r][k] = sB[r][k] = cB[r][k] = 0.f;
      }
    }
  }

  // Sources [lo, hi) of the staged chunk; lo is a multiple of 8.
  __device__ __forceinline__ void consume(const float4* const* bufs, int lo, int hi) {
    if constexpr (U > 0)
      consume_ahead(bufs, lo, hi);
    else
      consume_plain(bufs, lo, hi);
  }

  __device__ __forceinline__ void consume_plain(const float4* const* bufs, int lo, int hi) {
    const float4* Q = bufs[0];
    const float4* Ab = bufs[1];
    for (int sb = lo; sb < hi; sb += kSub) {
      const int sl = min(kSub, hi - sb);
      float2 a1[R][D], a2[R][D], bb[R][D];
      zero(a1, a2, bb);
      for (int jj = 0; jj < sl; jj += kUnroll) {
#pragma unroll
        for (int u = 0; u < kUnroll / 2; ++u) {
          const int ri = ((sb + jj) / 2 + u) * D;
          float2 v[2 * D], w[2 * D];  // v: -q~_j, p_j;  w: alpha_j, -b~_j
          rec_split<D>(Q + ri, v);
          rec_split<D>(Ab + ri, w);
#pragma unroll
          for (int r = 0; r < R; ++r) bwd_record<D>(q[r], p[r], a[r], b[r], v, w, a1[r], a2[r], bb[r]);
        }
      }
      fold(a1, a2, bb);
    }
  }

  // The same with the next U records on their way, across the sub-blocks.
  __device__ __forceinline__ void consume_ahead(const float4* const* bufs, int lo, int hi) {
    constexpr int V = U > 0 ? U : 1;
    static_assert(kUnroll % (2 * V) == 0, "groups must divide the split granule");
    const float4 *P = bufs[0] + lo / 2 * D, *PA = bufs[1] + lo / 2 * D;
    float4 nx[V][D], ny[V][D];
    load_records<V, D>(P, nx);
    load_records<V, D>(PA, ny);
    for (int sb = lo; sb < hi; sb += kSub) {
      const int sl = min(kSub, hi - sb);
      float2 a1[R][D], a2[R][D], bb[R][D];
      zero(a1, a2, bb);
      for (int jj = 0; jj < sl; jj += 2 * V) {
        float4 cu[V][D], cy[V][D];
#pragma unroll
        for (int u = 0; u < V; ++u)
#pragma unroll
          for (int f = 0; f < D; ++f) {
            cu[u][f] = nx[u][f];
            cy[u][f] = ny[u][f];
          }
        P += V * D;
        PA += V * D;
        load_records<V, D>(P, nx);
        load_records<V, D>(PA, ny);
#pragma unroll
        for (int u = 0; u < V; ++u) {
          float2 v[2 * D], w[2 * D];
          rec_split<D>(cu[u], v);
          rec_split<D>(cy[u], w);
#pragma unroll
          for (int r = 0; r < R; ++r) bwd_record<D>(q[r], p[r], a[r], b[r], v, w, a1[r], a2[r], bb[r]);
        }
      }
      fold(a1, a2, bb);
    }
  }

  __device__ __forceinline__ static void zero(float2 (&a1)[R][D], float2 (&a2)[R][D], float2 (&bb)[R][D]) {
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int k = 0; k < D; ++k) a1[r][k] = a2[r][k] = bb[r][k] = make_float2(0.f, 0.f);
  }

  // Both halves of the plain sums into the Kahan pairs.
  __device__ __forceinline__ void fold(const float2 (&a1)[R][D], const float2 (&a2)[R][D], const float2 (&bb)[R][D]) {
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int k = 0; k < D; ++k) {
        kahan_add(s1[r][k], c1[r][k], __fadd_rn(a1[r][k].x, a1[r][k].y));
        kahan_add(s2[r][k], c2[r][k], __fadd_rn(a2[r][k].x, a2[r][k].y));
        kahan_add(sB[r][k], cB[r][k], __fadd_rn(bb[r][k].x, bb[r][k].y));
      }
  }

  // out[0..D) = dalpha, out[D..2D) = dbeta of target r.
  __device__ __forceinline__ void result(int r, float kq, float kappa, ds out[2 * D]) const {
#pragma unroll
    for (int k = 0; k < D; ++k) {
      out[k] = ds_add(ds_mul_f(ds_from_kahan(s1[r][k], c1[r][k]), kq),
                      ds_mul_f(ds_from_kahan(s2[r][k], c2[r][k]), -kappa));
      out[D + k] = ds_from_kahan(sB[r][k], cB[r][k]);
    }
  }
};

}  // namespace gs
