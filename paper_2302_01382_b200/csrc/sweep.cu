// Quantization-error sensitivity sweep (Eq. 2 of the paper): for every tensor and every bit
// width b in 2..8 the sum of squared differences between x and Q_b(x), in ONE pass over HBM.
//
// A row (output channel) is held in registers by a team of 32..256 threads: the row maximum,
// the 7 scale pairs and the 7 error sums all come from those registers, so every weight is
// read from HBM exactly once.  Per element and bit width the work is four FMA-pipe ops:
//   u = fma(x, inv_scale, 1.5*2^23)   (round-half-even of x*inv_scale in the low mantissa bits)
//   r = u - 1.5*2^23                  (the code as a float)
//   e = fma(-scale, r, x)             (x - Q(x))
//   acc = fma(e, e, acc)
// The clip of Eq. 1 is a no-op here because the scale comes from the row's own maximum.
//
// Work distribution: the rows of all tensors form one flat sequence, cut into as many pieces of equal
// cost as blocks stay resident on the device; a piece that crosses a tensor boundary becomes several
// segments.  Every block therefore starts once, streams the same amount and ends with the others,
// whatever the mix of row lengths (the 54 tensors of ResNet-50 took one launch per row length and
// one block for the 147-column stem: 144 us, now 46).
// Each segment writes its 7 sums and its maximum to its own slot; one block per tensor (the one that
// finishes its last segment, or a finalize kernel's) adds the tensor's slots in a fixed order, so the
// result does not depend on timing.
// Queues were slower: blocks taking items of an eighth of a piece 126 us against 94 for 80 M elements
// in rows of 768, single warps taking items 125 us.
//
// Sums: fp32 in two short stages, then fp64.  A thread's packed accumulators take at most
// kChainTerms squared errors each; they are then added into a second fp32 accumulator per bit width,
// which takes at most kChainSums such sums; that one is reduced over the warp in fp64 and added to the
// warp's sum in shared memory.  A sequential fp32 sum of n non-negative terms is within (n-1)*2^-24
// relative of the exact sum, so the two stages together stay within (23 + 1 + 15) * 2^-24 = 2.3e-6,
// inside the sweep's 1e-5 tolerance; no thread of these rows keeps fp64 accumulators in registers.
// Rows that are not whole aligned float4 go from the first stage to fp64, after one squared error below 512 columns and
// one per 256 columns beyond (64 x 147: mean error 4.5e-10 of the sum; through both fp32 stages 1.7e-9.  Four blocks of
// hidden size 701: 69.7 us against 59.3).
#include <cstring>
#include <type_traits>

#include "common.cuh"

namespace qcfg {

namespace {

constexpr int kThreads = 256;
constexpr int kNB = 7;                       // bit widths 2..8
constexpr float kMagic = 12582912.0f;        // 1.5 * 2^23
constexpr int kRing = 3;                     // shared-memory row stages per thread
constexpr int kBlocksPerSM = 3;
constexpr int kChainTerms = 24;              // terms per fp32 accumulator of the first stage
constexpr int kChainSums = 16;               // such sums per fp32 accumulator of the second stage
constexpr int64_t kMinBlockElems = 2 * 1024;   // do not cut the work finer than one round of a block's eight warps at 256 columns

// One run of whole rows of one tensor, processed by one block.
struct SweepSeg {
  const float* w;         // first row of the run
  int32_t rows;
  int32_t cols;
  int32_t tensor;         // index into the caller's tensor list
  int32_t team_log2;      // team size = 32 << team_log2
  int32_t slot;           // partial-result slot
  int16_t v;              // float4 per thread and row (1..8); 0: rows too long for the ring
  int16_t vec;            // rows are 16-byte aligned and whole float4
};
static_assert(sizeof(SweepSeg) == 32, "one segment is two 16-byte words");
struct SweepBlock { int32_t seg0, nseg; };
struct TensorSlots { int32_t slot0, slot1; unsigned done, pad; };   // done: segments finished; back at 0 after every call

__device__ __forceinline__ void scales_for_lane(float A, int lane, float& s, float& inv) {
  int b = 2 + (lane % kNB);
  float qm = (float)((1 << (b - 1)) - 1);
  s = 1.0f; inv = 1.0f;
  if (A != 0.0f) { s = __fdiv_rn(A, qm); inv = __fdiv_rn(qm, A); }
}

__device__ __forceinline__ void err4(float x, float s, float inv, float& acc) {
  float u = fmaf(x, inv, kMagic);
  float r = u - kMagic;
  float e = fmaf(-s, r, x);
  acc = fmaf(e, e, acc);
}

// Two elements per instruction: the four operations of one (element, b) evaluation as packed
// fp32 arithmetic (sm_100 fma.rn.f32x2 / add.rn.f32x2), which halves the issue slots they need.
// ns holds the negated scale in both halves.
__device__ __forceinline__ void err8(float2 x, float2 ns, float2 inv, float2& acc) {
  const float2 magic = make_float2(kMagic, kMagic), nmagic = make_float2(-kMagic, -kMagic);
  float2 u = __ffma2_rn(x, inv, magic);
  float2 r = __fadd2_rn(u, nmagic);
  float2 e = __ffma2_rn(ns, r, x);
  acc = __ffma2_rn(e, e, acc);
}

// The tensor's result from the slots of its segments, written by the block that finished the last of
// them: 32 groups of 8 threads stride over the slots (thread j of a group owns column j: 7 sums and
// the maximum), then thread j < 8 combines the 32 group results.  The order is that of the slots,
// whichever block does it, so the result does not depend on timing.
__device__ __forceinline__ void finalize_tensor(const double* __restrict__ partial, int slot0, int slot1, int t, int jlo, int nb,
                                                double* __restrict__ sse, float* __restrict__ absmax, int write_absmax,
                                                double (*sm)[8]) {
  const int j = threadIdx.x & 7, g = threadIdx.x >> 3;
  double v = 0.0;
  for (int i = slot0 + g; i < slot1; i += 32) {
    const double x = __ldcg(partial + (int64_t)i * 8 + j);      // other blocks wrote them: not through L1
    v = (j == 7) ? fmax(v, x) : v + x;
  }
  sm[g][j] = v;
  __syncthreads();
  if (threadIdx.x < 8) {
    double a = sm[0][j];
    for (int k = 1; k < 32; ++k) a = (j == 7) ? fmax(a, sm[k][j]) : a + sm[k][j];
    if (j == 7) {
      if (write_absmax) absmax[t] = (float)a;
    } else if (j >= jlo && j < jlo + nb) {
      sse[(int64_t)t * nb + (j - jlo)] = a;
    }
  }
  __syncthreads();
}

// What the bodies below keep in shared memory besides the ring, declared once by the kernel: with arrays of their own
// the nine bodies of a mixed plan took 5 KB, and where the ring is 72 KB only two of the three blocks per SM that the
// plan counts on were resident (four blocks of hidden size 701: 67 us, 59 this way).
struct SweepShared {
  float smax2[2][kThreads / 32];
  double swarp[kThreads / 32][8];             // per warp: 7 fp64 sums and the maximum
};

// One run of rows of up to 4*V*team elements, VEC: whole aligned float4, otherwise copied word by word.
// All 7 bit widths are always evaluated (a narrower request only selects columns at the end).
template <int V, bool VEC>
__device__ __forceinline__ void sweep_segment(const SweepSeg& d, int per_tensor, float A_tensor, float4* ring, SweepShared& sh,
                                              double* __restrict__ out) {
  // rows between two first-stage flushes: every row adds 2*V terms to each half of a packed accumulator
  constexpr int kFlushRows = (kChainTerms / (2 * V)) > 0 ? (kChainTerms / (2 * V)) : 1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int T = 32 << d.team_log2;
  const int nteams = kThreads >> (5 + d.team_log2);
  const int team = threadIdx.x >> (5 + d.team_log2);
  const int tl = threadIdx.x & (T - 1);
  const int n_iter = (d.rows + nteams - 1) / nteams;
  const int c4 = d.cols >> 2;
  int row_parity = 0;
  double (*swarp)[8] = sh.swarp;

  float2 facc[kNB];
  float f2[kNB];                              // VEC: the second fp32 stage
  double dacc[kNB];                           // otherwise: fp64 behind a first stage of `chain` terms
#pragma unroll
  for (int j = 0; j < kNB; ++j) { facc[j] = make_float2(0.0f, 0.0f); f2[j] = 0.0f; dacc[j] = 0.0; }
  const int chain = d.cols < 2 * kThreads ? 1 : d.cols / kThreads < kChainTerms ? d.cols / kThreads : kChainTerms;
  int terms = 0;
  if (lane < 8) swarp[warp][lane] = 0.0;
  float amax_blk = 0.0f;

  auto process_row = [&](const float4 (&cur)[V]) {
    float m = 0.0f;
#pragma unroll
    for (int v = 0; v < V; ++v)
      m = fmaxf(fmaxf(fmaxf(m, fabsf(cur[v].x)), fmaxf(fabsf(cur[v].y), fabsf(cur[v].z))), fabsf(cur[v].w));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (T > 32) {
      // the team's warps exchange their maxima through shared memory; a named barrier per team
      // keeps other teams running, and alternating slots make one barrier per row enough
      float* slot = sh.smax2[row_parity];
      if (lane == 0) slot[warp] = m;
      asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "r"(T) : "memory");
      const int w0 = team * (T >> 5);
      m = slot[w0];
      for (int w = 1; w < (T >> 5); ++w) m = fmaxf(m, slot[w0 + w]);
      row_parity ^= 1;
    }
    amax_blk = fmaxf(amax_blk, m);
    if (per_tensor) m = A_tensor;

    // the 7 scale pairs: two IEEE divisions in lanes 0..6, broadcast by shuffles
    float s_l, inv_l;
    scales_for_lane(m, lane, s_l, inv_l);
    float2 ns[kNB], inv[kNB];
#pragma unroll
    for (int j = 0; j < kNB; ++j) {
      const float sj = -__shfl_sync(0xffffffffu, s_l, j), ij = __shfl_sync(0xffffffffu, inv_l, j);
      ns[j] = make_float2(sj, sj);
      inv[j] = make_float2(ij, ij);
    }
    auto flush1 = [&]() {                       // !VEC
      if (++terms < chain) return;
      terms = 0;
#pragma unroll
      for (int j = 0; j < kNB; ++j) { dacc[j] += (double)facc[j].x + (double)facc[j].y; facc[j] = make_float2(0.0f, 0.0f); }
    };
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const float2 lo = make_float2(cur[v].x, cur[v].y), hi = make_float2(cur[v].z, cur[v].w);
      if (VEC) {
#pragma unroll
        for (int j = 0; j < kNB; ++j) {
          err8(lo, ns[j], inv[j], facc[j]);
          err8(hi, ns[j], inv[j], facc[j]);
        }
      } else {
#pragma unroll
        for (int j = 0; j < kNB; ++j) err8(lo, ns[j], inv[j], facc[j]);
        flush1();
#pragma unroll
        for (int j = 0; j < kNB; ++j) err8(hi, ns[j], inv[j], facc[j]);
        flush1();
      }
    }
  };
  // second stage, or the thread's fp64 sums -> the warp's fp64 sums
  auto flush2 = [&]() {
#pragma unroll
    for (int j = 0; j < kNB; ++j) {
      const double v = warp_sum(VEC ? (double)f2[j] : dacc[j]);
      if (lane == 0) swarp[warp][j] += v;
      f2[j] = 0.0f;
    }
  };

  // Rows stream through a three-stage ring in shared memory filled by cp.async, two rows ahead
  // of the one being processed: enough loads in flight to cover HBM latency without holding
  // future rows in registers.  Every thread copies and reads back only its own 16-byte slots, so
  // no barrier is needed between the copy and the read.  Rows that are not whole aligned float4
  // are copied word by word, consecutive lanes taking consecutive words; which element sits in
  // which slot does not matter to the sums.
  const float* rowp = d.w + (int64_t)team * d.cols + (VEC ? 4 * tl : tl);   // this thread's first element of its team's next row
  const int64_t row_step = (int64_t)nteams * d.cols;
  int fetch_row = team;
  const uint32_t ring0 = (uint32_t)__cvta_generic_to_shared(ring + threadIdx.x);
  auto issue_row = [&](int stage) {
    const uint32_t dst0 = ring0 + (uint32_t)(stage * V) * (kThreads * 16);
    const bool row_ok = fetch_row < d.rows;
    if (VEC) {
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const uint32_t dst = dst0 + v * (kThreads * 16);
        if (row_ok && tl + v * T < c4) {
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(reinterpret_cast<const float4*>(rowp) + v * T) : "memory");
        } else {
          asm volatile("st.shared.v4.f32 [%0], {%1, %1, %1, %1};" ::"r"(dst), "f"(0.0f) : "memory");
        }
      }
    } else {
#pragma unroll 4
      for (int e = 0; e < 4 * V; ++e) {
        const uint32_t dst = dst0 + (e >> 2) * (kThreads * 16) + (e & 3) * 4;
        if (row_ok && tl + e * T < d.cols) {
          asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(rowp + e * T) : "memory");
        } else {
          asm volatile("st.shared.f32 [%0], %1;" ::"r"(dst), "f"(0.0f) : "memory");
        }
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    rowp += row_step;
    fetch_row += nteams;
  };
  issue_row(0);
  issue_row(1);
  int stage = 0, n1 = 0, n2 = 0;
  for (int it = 0; it < n_iter; ++it) {
    int nxt = stage + 2; if (nxt >= kRing) nxt -= kRing;
    issue_row(nxt);                                                 // zeros past the end
    asm volatile("cp.async.wait_group 2;" ::: "memory");            // the row of this iteration has landed
    float4 cur[V];
#pragma unroll
    for (int v = 0; v < V; ++v) cur[v] = ring[(stage * V + v) * kThreads + threadIdx.x];
    process_row(cur);
    if (VEC && ++n1 == kFlushRows) {
#pragma unroll
      for (int j = 0; j < kNB; ++j) { f2[j] += facc[j].x + facc[j].y; facc[j] = make_float2(0.0f, 0.0f); }
      n1 = 0;
      if (++n2 == kChainSums - 1) { flush2(); n2 = 0; }
    }
    if (++stage == kRing) stage = 0;
  }
#pragma unroll
  for (int j = 0; j < kNB; ++j) {
    if (VEC) f2[j] += facc[j].x + facc[j].y;
    else dacc[j] += (double)facc[j].x + (double)facc[j].y;
  }
  flush2();
  asm volatile("cp.async.wait_group 0;" ::: "memory");
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) amax_blk = fmaxf(amax_blk, __shfl_xor_sync(0xffffffffu, amax_blk, o));
  if (lane == 0) swarp[warp][7] = (double)amax_blk;
  __syncthreads();
  if (threadIdx.x < 8) {                  // the warps' sums in a fixed order
    double v = swarp[0][threadIdx.x];
    for (int w = 1; w < kThreads / 32; ++w)
      v = (threadIdx.x == 7) ? fmax(v, swarp[w][7]) : v + swarp[w][threadIdx.x];
    out[threadIdx.x] = v;
  }
}

// Rows longer than the ring holds: the whole block works on one row at a time and reads it twice
// (the second read hits L1/L2).
__device__ __forceinline__ void sweep_segment_long(const SweepSeg& d, int per_tensor, float A_tensor, int jlo, int jhi, SweepShared& sh,
                                                   double* __restrict__ out) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* smax = sh.smax2[0];
  double (*swarp)[8] = sh.swarp;
  double dacc[kNB];
#pragma unroll
  for (int j = 0; j < kNB; ++j) dacc[j] = 0.0;
  float amax_blk = 0.0f;
  for (int row = 0; row < d.rows; ++row) {
    const float* p = d.w + (int64_t)row * d.cols;
    float m = 0.0f;
    for (int c = threadIdx.x; c < d.cols; c += kThreads) m = fmaxf(m, fabsf(__ldg(p + c)));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) smax[warp] = m;
    __syncthreads();
    m = smax[0];
    for (int w = 1; w < kThreads / 32; ++w) m = fmaxf(m, smax[w]);
    __syncthreads();
    amax_blk = fmaxf(amax_blk, m);
    if (per_tensor) m = A_tensor;
    float s_l, inv_l;
    scales_for_lane(m, lane, s_l, inv_l);
    float s[kNB], inv[kNB], facc[kNB];
#pragma unroll
    for (int j = 0; j < kNB; ++j) {
      s[j] = __shfl_sync(0xffffffffu, s_l, j);
      inv[j] = __shfl_sync(0xffffffffu, inv_l, j);
      facc[j] = 0.0f;
    }
    int terms = 0;
    for (int c = threadIdx.x; c < d.cols; c += kThreads) {
      float x = __ldg(p + c);
#pragma unroll
      for (int j = 0; j < kNB; ++j)
        if (j >= jlo && j <= jhi) err4(x, s[j], inv[j], facc[j]);
      if (++terms == kChainTerms) {            // very long rows: keep the fp32 chains short
#pragma unroll
        for (int j = 0; j < kNB; ++j) { dacc[j] += (double)facc[j]; facc[j] = 0.0f; }
        terms = 0;
      }
    }
#pragma unroll
    for (int j = 0; j < kNB; ++j) dacc[j] += (double)facc[j];
  }
#pragma unroll
  for (int j = 0; j < kNB; ++j) {
    double v = warp_sum(dacc[j]);
    if (lane == 0) swarp[warp][j] = v;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) amax_blk = fmaxf(amax_blk, __shfl_xor_sync(0xffffffffu, amax_blk, o));
  if (lane == 0) swarp[warp][7] = (double)amax_blk;
  __syncthreads();
  if (threadIdx.x < 8) {
    double v = swarp[0][threadIdx.x];
    for (int w = 1; w < kThreads / 32; ++w)
      v = (threadIdx.x == 7) ? fmax(v, swarp[w][7]) : v + swarp[w][threadIdx.x];
    out[threadIdx.x] = v;
  }
}

// All segments of a call.  KV: the float4 count per thread of every segment, all of them aligned, or 0
// when the plan mixes row lengths (the body is then chosen per segment, at the register count of the
// largest).  FUSED: the block that finishes a tensor's last segment also writes the tensor's result
// (plans that do not fill the device: 15.6 us for three tensors of 256 columns against 20.5 with a
// second launch); otherwise a finalize kernel follows (the counting costs every segment a round trip to
// L2: 110.4 against 106.3 us for 340 MB).
template <int KV, bool FUSED>
__global__ void __launch_bounds__(kThreads, kBlocksPerSM)
sweep_kernel(const SweepSeg* __restrict__ segs, const SweepBlock* __restrict__ blocks, TensorSlots* __restrict__ slots, int per_tensor,
             const float* __restrict__ tensor_absmax, int jlo, int nb, double* __restrict__ partial, double* __restrict__ sse,
             float* __restrict__ absmax) {
  // Programmatic dependent launch: the block is scheduled while the previous kernel of the stream
  // drains and waits here for that kernel's results (result slots, per-tensor maxima, and whatever
  // produced the weights).
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __shared__ double fin[32][8];
  __shared__ int last;
  __shared__ SweepShared sh;
  extern __shared__ float4 ring[];                       // [kRing][V][kThreads]
  const SweepBlock blk = blocks[blockIdx.x];
  for (int si = blk.seg0; si < blk.seg0 + blk.nseg; ++si) {
    const SweepSeg d = segs[si];
    const float A_tensor = per_tensor ? tensor_absmax[d.tensor] : 0.0f;
    double* out = partial + (int64_t)d.slot * 8;
    auto run = [&](auto v) {
      if (d.vec) sweep_segment<decltype(v)::value, true>(d, per_tensor, A_tensor, ring, sh, out);
      else sweep_segment<decltype(v)::value, false>(d, per_tensor, A_tensor, ring, sh, out);
    };
    if (KV > 0) sweep_segment<(KV > 0 ? KV : 1), true>(d, per_tensor, A_tensor, ring, sh, out);
    else switch (d.v) {
      case 0: sweep_segment_long(d, per_tensor, A_tensor, jlo, jlo + nb - 1, sh, out); break;
      case 1: run(std::integral_constant<int, 1>()); break;
      case 2: run(std::integral_constant<int, 2>()); break;
      case 3: run(std::integral_constant<int, 3>()); break;
      case 4: run(std::integral_constant<int, 4>()); break;
      case 5: run(std::integral_constant<int, 5>()); break;
      case 6: run(std::integral_constant<int, 6>()); break;
      case 7: run(std::integral_constant<int, 7>()); break;
      default: run(std::integral_constant<int, 8>()); break;
    }
    if (!FUSED) { __syncthreads(); continue; }
    // The eight values of the slot become visible before the segment is counted; the counter wraps
    // to zero with the tensor's last segment, so the next call finds it as this one did.
    if (threadIdx.x < 8) __threadfence();
    __syncthreads();
    const int slot0 = slots[d.tensor].slot0, slot1 = slots[d.tensor].slot1;
    if (threadIdx.x == 0) {
      const unsigned n = (unsigned)(slot1 - slot0);
      last = atomicInc(&slots[d.tensor].done, n - 1) == n - 1;
      __threadfence();
    }
    __syncthreads();
    if (last) finalize_tensor(partial, slot0, slot1, d.tensor, jlo, nb, sse, absmax, per_tensor ? 0 : 1, fin);
  }
}
__global__ void __launch_bounds__(kThreads)
sweep_finalize_kernel(const TensorSlots* __restrict__ slots, int write_absmax, int jlo, int nb, const double* __restrict__ partial,
                      double* __restrict__ sse, float* __restrict__ absmax) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");     // the slots come from the kernel before
  __shared__ double fin[32][8];
  const int t = blockIdx.x;
  finalize_tensor(partial, slots[t].slot0, slots[t].slot1, t, jlo, nb, sse, absmax, write_absmax, fin);
}

// Per-tensor maxima for the per-tensor grids, over the same segments: integer max of |x| bit patterns.
__global__ void __launch_bounds__(kThreads)
sweep_absmax_kernel(const SweepSeg* __restrict__ segs, const SweepBlock* __restrict__ blocks, unsigned* __restrict__ absmax) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __shared__ unsigned sm[kThreads / 32];
  const SweepBlock blk = blocks[blockIdx.x];
  for (int si = blk.seg0; si < blk.seg0 + blk.nseg; ++si) {
    const SweepSeg d = segs[si];
    const int64_t n = (int64_t)d.rows * d.cols;
    unsigned m = 0;
    auto fold = [&](float x) { const unsigned a = abs_bits(x); m = m > a ? m : a; };
    if (d.vec) {
      const float4* p = reinterpret_cast<const float4*>(d.w);
#pragma unroll 4
      for (int64_t i = threadIdx.x; i < (n >> 2); i += kThreads) { const float4 x = __ldg(p + i); fold(x.x); fold(x.y); fold(x.z); fold(x.w); }
    } else {
#pragma unroll 4
      for (int64_t i = threadIdx.x; i < n; i += kThreads) fold(__ldg(d.w + i));
    }
    m = warp_max_u(m);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x < 32) {
      m = warp_max_u(threadIdx.x < kThreads / 32 ? sm[threadIdx.x] : 0u);
      if (threadIdx.x == 0 && m) atomicMax(absmax + d.tensor, m);
    }
    __syncthreads();
  }
}

// Launch configuration with programmatic stream serialization: the kernel may start while its
// predecessor in the stream drains; it orders itself with griddepcontrol.wait.
inline cudaLaunchConfig_t pdl_config(cudaLaunchAttribute* attr, int blocks, size_t smem, cudaStream_t st) {
  attr->id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr->val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3((unsigned)kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

using SweepKernel = void (*)(const SweepSeg*, const SweepBlock*, TensorSlots*, int, const float*, int, int, double*, double*, float*);
constexpr SweepKernel kSweepKernels[9] = {sweep_kernel<0, false>, sweep_kernel<1, false>, sweep_kernel<2, false>,
                                          sweep_kernel<3, false>, sweep_kernel<4, false>, sweep_kernel<5, false>,
                                          sweep_kernel<6, false>, sweep_kernel<7, false>, sweep_kernel<8, false>};
constexpr SweepKernel kSweepFused = sweep_kernel<0, true>;

constexpr size_t ring_bytes(int v) { return (size_t)kRing * v * kThreads * sizeof(float4); }

// ------------------------------------------------------------------ planning (host)

// Capacity of the tables a plan is written into.  Segments never exceed blocks + tensors.
struct PlanTables {
  SweepSeg* segs; int max_segs;
  SweepBlock* blocks; int max_blocks;
  TensorSlots* slots; int max_tensors;
};
struct Plan {
  int n_segs = 0, n_blocks = 0;
  int max_v = 0;             // largest float4 count per thread and row: sizes the ring
  int one_v = 0;             // that count if all rows have it and are aligned, else 0
  bool fused = false;        // fewer blocks than the device keeps resident: one launch
};

// How a tensor's rows are processed, and what one row costs (relative).
struct RowPlan { int v, team_log2, vec; int64_t cost; };
// A row takes T = 32 << team_log2 threads with V float4 each.  Measured on long runs of one row length
// (80 M elements, ns per row over the whole device): T = 32 costs 0.14 (V + 0.5) for V = 1..8, and
// every doubling of the team about 5 % more per warp (barrier between its warps).  V up to 8 fits
// the ring with two blocks per SM, V up to 6 with three; two are enough where all rows are that
// long (1024 columns: 1.27 ns as V = 8 against 1.39 as two warps with V = 4), three serve a mixed plan.
constexpr int kMaxV = 6;
inline RowPlan plan_rows(const float* w, int64_t cols, int max_v) {
  RowPlan best{0, 0, 0, 0};
  best.vec = ((uintptr_t)w % 16 == 0) && (cols % 4 == 0);
  const int64_t c4 = (cols + 3) / 4;
  for (int tl = 0; tl <= 3; ++tl) {
    const int64_t v = (c4 + (32 << tl) - 1) / (32 << tl);
    if (v > (tl == 3 ? 8 : max_v)) continue;
    const int64_t cost = ((int64_t)1 << tl) * (2 * v + 1) * (20 + tl);
    if (best.v == 0 || cost < best.cost) { best.v = (int)v; best.team_log2 = tl; best.cost = cost; }
  }
  if (best.v == 0) best.cost = (cols / 128 + 16) * 80;      // whole block per row, read twice
  else if (!best.vec) best.cost *= 2;                       // word-wise copies (147 columns: 0.46 against 0.21 ns per row of 128)
  return best;
}

// Cuts the rows of all tensors into pieces of equal cost, one per block.  Returns false when a table is
// too small.  Segments of one tensor get consecutive slots; a tensor without elements gets one empty
// segment, whose zeros become its result.
bool plan_sweep(const float* const* w, const int64_t* rows, const int64_t* cols, int32_t n_tensors, int sms,
                const PlanTables& T, Plan* P) {
  if (n_tensors > T.max_tensors) return false;
  int64_t total = 0, elems = 0;
  int limit = 8;
  for (int pass = 0; pass < 2; ++pass) {       // rows of one kind only: V up to 8; otherwise plan again with the mixed plan's limit
    total = elems = 0;
    P->max_v = 0;
    for (int t = 0; t < n_tensors; ++t) {
      if (rows[t] * cols[t] == 0) continue;
      const RowPlan r = plan_rows(w[t], cols[t], limit);
      P->one_v = r.vec && (elems == 0 || r.v == P->one_v) ? r.v : 0;
      if (r.v > P->max_v) P->max_v = r.v;
      total += rows[t] * r.cost;
      elems += rows[t] * cols[t];
    }
    if (P->one_v || P->max_v <= kMaxV) break;
    limit = kMaxV;
  }
  if (P->max_v < 1) P->max_v = 1;
  const int resident = sms * (P->max_v > kMaxV ? 2 : kBlocksPerSM);
  int64_t nblk = (elems + kMinBlockElems - 1) / kMinBlockElems;
  if (nblk > resident) nblk = resident;
  if (nblk < 1) nblk = 1;
  P->fused = nblk < resident;
  if (nblk > T.max_blocks) return false;
  const int64_t quota = (total + nblk - 1) / nblk;             // cost per block
  int blk = 0;
  int64_t room = quota;
  T.blocks[0].seg0 = 0; T.blocks[0].nseg = 0;
  for (int t = 0; t < n_tensors; ++t) {
    const bool empty = rows[t] * cols[t] == 0;
    const RowPlan r = empty ? RowPlan{P->one_v ? P->one_v : 1, 0, 0, 1} : plan_rows(w[t], cols[t], limit);
    const int64_t nt = r.v ? kThreads / (32 << r.team_log2) : 1;
    T.slots[t].slot0 = P->n_segs;
    T.slots[t].done = 0; T.slots[t].pad = 0;
    const int64_t n_rows = empty ? 0 : rows[t];
    int64_t row = 0;
    do {
      int64_t take = (room + r.cost - 1) / r.cost;              // whole rows filling the block's quota
      if (take < 8 * nt) take = (take + nt - 1) / nt * nt;      // few rounds of the block's teams: whole ones
      if (blk == nblk - 1) take = n_rows - row;                 // the last block takes what is left
      if (take < nt) take = nt;
      if (take > n_rows - row) take = n_rows - row;
      if (take > 0x40000000) take = 0x40000000;
      if (P->n_segs >= T.max_segs) return false;
      SweepSeg& s = T.segs[P->n_segs];
      s.w = empty ? nullptr : w[t] + row * cols[t]; s.rows = (int32_t)take; s.cols = empty ? 0 : (int32_t)cols[t]; s.tensor = t;
      s.team_log2 = r.team_log2; s.slot = P->n_segs; s.v = (int16_t)r.v; s.vec = (int16_t)r.vec;
      P->n_segs++;
      T.blocks[blk].nseg++;
      row += take;
      room -= take * r.cost;
      if (room <= 0 && blk < nblk - 1) {
        ++blk;
        T.blocks[blk].seg0 = P->n_segs; T.blocks[blk].nseg = 0;
        room += quota;                                          // what this block took beyond its quota the next one takes less
        if (room < quota / 2) room = quota / 2;
      }
    } while (row < n_rows);
    T.slots[t].slot1 = P->n_segs;
  }
  P->n_blocks = blk + (T.blocks[blk].nseg > 0 ? 1 : 0);        // a last block left without a segment is not launched
  return true;
}

// Enqueues the sweep's kernels for a plan whose tables are on the device already.
int run_plan(Ctx* ctx, const Plan& P, const SweepSeg* segs, const SweepBlock* blocks, TensorSlots* slots, double* partial,
             int32_t n_tensors, int per_tensor, int b_lo, int b_hi, double* sse, float* absmax, cudaStream_t st) {
  cudaLaunchAttribute attr;
  if (per_tensor) {
    cudaError_t e = cudaMemsetAsync(absmax, 0, (size_t)n_tensors * sizeof(float), st);
    if (e != cudaSuccess) return check_cuda(ctx, e, "memset absmax");
    cudaLaunchConfig_t cfg = pdl_config(&attr, P.n_blocks, 0, st);
    prof_begin(ctx, 2, st);
    e = cudaLaunchKernelEx(&cfg, sweep_absmax_kernel, segs, blocks, reinterpret_cast<unsigned*>(absmax));
    prof_end(ctx, 2, 0.0, st);
    if (e != cudaSuccess) return check_cuda(ctx, e, "sweep absmax launch");
    count_launch(ctx);
  }
  cudaLaunchConfig_t cfg = pdl_config(&attr, P.n_blocks, ring_bytes(P.max_v), st);
  prof_begin(ctx, 2, st);
  cudaError_t e = cudaLaunchKernelEx(&cfg, P.fused ? kSweepFused : kSweepKernels[P.one_v], segs, blocks, slots, per_tensor,
                                     (const float*)absmax, b_lo - 2, b_hi - b_lo + 1, partial, sse, absmax);
  prof_end(ctx, 2, 0.0, st);
  if (e != cudaSuccess) return check_cuda(ctx, e, "sweep launch");
  count_launch(ctx);
  if (!P.fused) {
    cfg = pdl_config(&attr, n_tensors, 0, st);
    e = cudaLaunchKernelEx(&cfg, sweep_finalize_kernel, (const TensorSlots*)slots, per_tensor ? 0 : 1, b_lo - 2, b_hi - b_lo + 1,
                           (const double*)partial, sse, absmax);
    if (e != cudaSuccess) return check_cuda(ctx, e, "sweep finalize launch");
    count_launch(ctx);
  }
  return check_cuda(ctx, cudaGetLastError(), "sweep launch");
}

inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

}  // namespace

// The shared-memory opt-in of a kernel is a per-device attribute: set for every variant whenever a
// context is created (the context's device is current then).
int sweep_init(Ctx* ctx) {
  cudaError_t e = cudaSuccess;
  for (int v = 0; v <= 8 && e == cudaSuccess; ++v)
    e = cudaFuncSetAttribute(kSweepKernels[v], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ring_bytes(v ? v : 8));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(kSweepFused, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ring_bytes(8));
  return check_cuda(ctx, e, "sweep smem attribute");
}

int launch_sweep(Ctx* ctx, const float* const* w, const int64_t* rows, const int64_t* cols, int32_t n_tensors,
                 int granularity, int b_lo, int b_hi, double* sse, float* absmax, cudaStream_t st) {
  if (n_tensors == 0) return QCFG_OK;
  const int max_blocks = sm_count(ctx) * kBlocksPerSM, max_segs = max_blocks + n_tensors;
  // host tables in one context-owned buffer: tensor slot ranges | blocks | segments
  const size_t slot_bytes = align_up((size_t)n_tensors * sizeof(TensorSlots), 16);
  const size_t blk_bytes = align_up((size_t)max_blocks * sizeof(SweepBlock), 16);
  const size_t seg_bytes = (size_t)max_segs * sizeof(SweepSeg);
  char* host = static_cast<char*>(host_scratch(ctx, slot_bytes + blk_bytes + seg_bytes));
  if (!host) return set_error(ctx, QCFG_ENOMEM, "sweep: host tables");
  memset(host + slot_bytes, 0, blk_bytes);                       // entries of unused blocks take part in the comparison below
  PlanTables T{reinterpret_cast<SweepSeg*>(host + slot_bytes + blk_bytes), max_segs,
               reinterpret_cast<SweepBlock*>(host + slot_bytes), max_blocks, reinterpret_cast<TensorSlots*>(host), n_tensors};
  Plan P;
  if (!plan_sweep(w, rows, cols, n_tensors, sm_count(ctx), T, &P)) return set_error(ctx, QCFG_EINVAL, "sweep: planning failed");
  const size_t used = slot_bytes + blk_bytes + (size_t)P.n_segs * sizeof(SweepSeg);

  // device scratch: partials | the same three tables
  const size_t partial_bytes = align_up((size_t)max_segs * 8 * sizeof(double), 256);
  char* base = static_cast<char*>(scratch(ctx, partial_bytes + slot_bytes + blk_bytes + seg_bytes));
  if (!base) return set_error(ctx, QCFG_ENOMEM, "sweep scratch (%zu bytes)", partial_bytes + slot_bytes + blk_bytes + seg_bytes);
  char* tab = base + partial_bytes;
  // the tables only depend on the tensor list: a repeated sweep of the same tensors (same scratch
  // buffer) finds them on the device already, the counters back at zero
  if (!sweep_tables_cached(ctx, base, st, host, used)) {
    const cudaError_t e = cudaMemcpyAsync(tab, host, used, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return check_cuda(ctx, e, "sweep table upload");
  }
  return run_plan(ctx, P, reinterpret_cast<const SweepSeg*>(tab + slot_bytes + blk_bytes),
                  reinterpret_cast<const SweepBlock*>(tab + slot_bytes), reinterpret_cast<TensorSlots*>(tab),
                  reinterpret_cast<double*>(base), n_tensors, granularity == QCFG_PER_TENSOR, b_lo, b_hi, sse, absmax, st);
}


// ------------------------------------------------------------------ sweep without allocation
//
// Same sweep, for callers that must not allocate device memory at call time: the segment
// partials and the tables live in a fixed device array that is part of the loaded library image
// (about 0.6 MiB on every GPU that loads the library, until the process exits).

constexpr int kStaticMaxTensors = 1024;
constexpr int kStaticMaxBlocks = 4096;                                  // 3 per SM
constexpr int kStaticMaxSegs = kStaticMaxBlocks + kStaticMaxTensors;
constexpr int64_t kStaticMaxElems = (int64_t)1 << 35;                   // elements per call

struct StaticSweepScratch {
  double partial[kStaticMaxSegs * 8];
  SweepSeg segs[kStaticMaxSegs];
  SweepBlock blocks[kStaticMaxBlocks];
  TensorSlots slots[kStaticMaxTensors];
};

static __device__ __align__(256) unsigned char g_static_sweep_scratch[sizeof(StaticSweepScratch)];

// Device address of the array above, per device ordinal.  In host code the array's name is only a
// handle for the runtime; the address a kernel can use comes from cudaGetSymbolAddress, asked
// once per device while that device is current.
constexpr int kMaxDevices = 64;
static void* g_static_sweep_addr[kMaxDevices] = {nullptr};

int launch_sweep_static(Ctx* ctx, const float* const* w, const int64_t* rows, const int64_t* cols,
                        int32_t n_tensors, int granularity, int b_lo, int b_hi, double* sse, float* absmax,
                        cudaStream_t st) {
  if (n_tensors == 0) return QCFG_OK;
  if (n_tensors > kStaticMaxTensors)
    return set_error(ctx, QCFG_ENOMEM, "static sweep: %d tensors exceed the fixed scratch (at most %d per call)",
                     n_tensors, kStaticMaxTensors);
  int64_t total = 0;
  for (int t = 0; t < n_tensors; ++t) {
    if (rows[t] > kStaticMaxElems || (cols[t] > 0 && rows[t] > kStaticMaxElems / cols[t])) total = kStaticMaxElems + 1;
    else total += rows[t] * cols[t];
    if (total > kStaticMaxElems)
      return set_error(ctx, QCFG_ENOMEM, "static sweep: more than 2^35 elements in one call; split the tensors over several calls");
  }
  if (sm_count(ctx) * kBlocksPerSM > kStaticMaxBlocks)
    return set_error(ctx, QCFG_ENOMEM, "static sweep: the device has more SMs than the fixed tables are sized for");

  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return check_cuda(ctx, e, "static sweep: cudaGetDevice");
  if (dev != device_of(ctx) || dev < 0 || dev >= kMaxDevices)
    return set_error(ctx, QCFG_ESTATE, "static sweep: the context's device (%d) must be the current device (%d)",
                     device_of(ctx), dev);
  if (!g_static_sweep_addr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_static_sweep_scratch);
    if (e != cudaSuccess || !p) return check_cuda(ctx, e == cudaSuccess ? cudaErrorInvalidSymbol : e, "static sweep: cudaGetSymbolAddress");
    g_static_sweep_addr[dev] = p;
  }
  StaticSweepScratch* S = static_cast<StaticSweepScratch*>(g_static_sweep_addr[dev]);

  // the plan is written into a host buffer the context owns (no large arrays on the caller's stack)
  const size_t seg_bytes = sizeof(S->segs), blk_bytes = sizeof(S->blocks), slot_bytes = sizeof(S->slots);
  char* host = static_cast<char*>(host_scratch(ctx, seg_bytes + blk_bytes + slot_bytes));
  if (!host) return set_error(ctx, QCFG_ENOMEM, "static sweep: host tables");
  PlanTables T{reinterpret_cast<SweepSeg*>(host), kStaticMaxSegs, reinterpret_cast<SweepBlock*>(host + seg_bytes), kStaticMaxBlocks,
               reinterpret_cast<TensorSlots*>(host + seg_bytes + blk_bytes), kStaticMaxTensors};
  Plan P;
  if (!plan_sweep(w, rows, cols, n_tensors, sm_count(ctx), T, &P))
    return set_error(ctx, QCFG_ENOMEM, "static sweep: the plan does not fit the fixed tables");

  // Every segment overwrites all 8 values of its own slot and the finalize kernel reads only the
  // slots of this call, so nothing left in the array by an earlier call needs clearing.  The copies
  // come from pageable host memory, so they have left the host buffer when the calls return.
  e = cudaMemcpyAsync(S->segs, T.segs, (size_t)P.n_segs * sizeof(SweepSeg), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(S->blocks, T.blocks, (size_t)P.n_blocks * sizeof(SweepBlock), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(S->slots, T.slots, (size_t)n_tensors * sizeof(TensorSlots), cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return check_cuda(ctx, e, "static sweep: table upload");
  return run_plan(ctx, P, S->segs, S->blocks, S->slots, S->partial, n_tensors,
                  granularity == QCFG_PER_TENSOR, b_lo, b_hi, sse, absmax, st);
}

}  // namespace qcfg
