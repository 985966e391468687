// The stem of a convolutional table at 16 bit: a stride-2 convolution of an image with few channels, its
// activation, and the 3x3/2 max-pool its consumers read, in one kernel.
//
// As separate steps (patch matrix, GEMM, max-pool) the 7x7 stem of 128 images of 224 x 224 x 3 took
// 620 us, nearly all of it moving a 514 MB patch matrix and a 411 MB fp32 output that only the pool
// reads; here 77 MB come in and 103 MB go out.
//
// A tile is one output row: up to 128 pixels are the M rows of a tcgen05.mma (bf16, fp32 accumulators), the
// reduction is the patch in (kh, kw, cin) order exactly as in the general path, sixteen elements per instruction,
// so both paths give the same bits.
//   warps 0..7  producers: bring input rows to shared memory as bf16 (a ring of sixteen, zeros left and right
//               of the image; two new rows per output row, loaded one output row ahead) and build the patch
//               matrix of the output row from them, a lane owning two neighbouring elements of the patch: its
//               source positions are fixed but for the pixel, so there is nothing to divide or test, and with the
//               channel count known every address of a pixel is an immediate (12 instructions per pixel and warp;
//               with 16-bit loads and computed addresses the kernel took 358 us, 302 us this way).
//   warp  8     MMA issuer: one of two patch tiles into one of four accumulators.
//   warps 9..16 epilogue: activation, running maximum over output rows in registers; every second row the
//               maxima of the row triple cross lanes through shared memory, and the pooled row leaves in 16-byte
//               stores, with its readers' int8 codes beside it (a quantize launch per reader took 19 us each).
// What bounds it (128 images of 224 x 224 x 3: 233 us from the end of the kernel in front to the last CTA's end, 299 before the
// row pitch and the second epilogue warp per quadrant): the producers.  With clocks read in the kernel (243 us, 1.84 GHz) a
// CTA of 105 output rows takes 446000 cycles: 220000 patch copies through shared memory, 126000 storing the two rows an
// output row adds and issuing the next loads, 24000 waiting for the tensor core, 34000 first rows of bands, 40000 weights,
// barriers and exit.  The epilogue is busy for 2250 of the 4100 cycles per output row.  Seven pixels per batch, predicated
// loads and an unrolled MMA loop changed nothing.
// Work items are bands of pooled rows of one image; a band repeats one output row of its neighbour.
#include "common.cuh"
#include "ptx.cuh"

namespace qcfg {

namespace {

constexpr int kProducers = 8;                 // warps
// Two epilogue warps per lane quadrant, 32 channels each.  With one (64 running maxima in registers, spilled) the producers
// waited for it: an evaluation of ResNet-50 at batch 128 2272 us, 2201 with two.
constexpr int kEpiWarps = 8;
constexpr int kStemThreads = 32 * (kProducers + 1 + kEpiWarps);
constexpr int kRows = 16;                     // input rows held (power of two)
constexpr int kMaxKh = 8, kMaxW = 256;
constexpr int kMaxK = 192, kKBlocks = kMaxK / 64;      // 128-byte k-blocks of 64 elements
constexpr int kLeft = 16;                     // elements in front of an input row's first one: the left padding ends there
// One input row of up to four channels with what its last window reads beyond; rows lie that far apart plus as many words as a
// window of one kernel row takes (StemParams::row_bytes), so that the 64 patch elements a warp reads at once, three or
// four windows of as many rows, come from as many banks.  Rows a multiple of 128 bytes apart have all windows on the same
// eleven (an evaluation of ResNet-50 at batch 128: 2282 us, 2262 this way).
constexpr int kRowBytes = (kLeft + kMaxW * 4 + 48) * 2, kMaxRowPitch = kRowBytes + 31 * 4;
constexpr int kTileBytes = kKBlocks * 128 * 128;
constexpr int kTiles = 2;
constexpr int kMaxN = 64;
constexpr int kWBytes = kMaxN * 128;          // weights of one k-block
constexpr int kAccs = 4;                      // accumulators of 64 columns
constexpr int kPoolPitch = kMaxN + 4;         // floats per pixel of a row of maxima: 16-byte writes of eight lanes on different banks
constexpr int kStemSmem = 1024 + 1024 + kTiles * kTileBytes + kKBlocks * kWBytes + 2 * 128 * kPoolPitch * 4 + kRows * kMaxRowPitch;
static_assert(kStemSmem <= 232448, "shared memory of one CTA");

struct StemParams {
  const float* x;              // [images, H, W, C]
  const __nv_bfloat16* w;      // [n, ldk] in (kh, kw, cin) order
  float* y;                    // [images * OH * OW, n] or null
  float* pool;                 // [images * PH * PW, n] or null
  int32_t H, W, C, kh, kw, pad, OH, OW, PH, PW, n, ldk, act;
  CodeSlot codes[kStemSlots];  // int8 codes of the pooled tensor for its readers (kind 1; 0: unused)
  int32_t bands, band_rows, items, row_bytes;
  unsigned* err;
  unsigned long long* stamp;
};

// one band: pooled rows p0..p1-1, output rows oh0..oh1
struct Band { int img, p0, p1, oh0, oh1; };
__device__ __forceinline__ Band band_of(const StemParams& p, int item) {
  Band b;
  b.img = item / p.bands;
  b.p0 = (item - b.img * p.bands) * p.band_rows;
  b.p1 = b.p0 + p.band_rows < p.PH ? b.p0 + p.band_rows : p.PH;
  b.oh0 = 2 * b.p0 - 1 > 0 ? 2 * b.p0 - 1 : 0;
  b.oh1 = 2 * b.p1 - 1 < p.OH - 1 ? 2 * b.p1 - 1 : p.OH - 1;
  return b;
}

// CC: channels, or 0 for any number up to four.  With CC set input rows are read four elements at a time (whole
// aligned groups of four in every row).
template <int CC>
__global__ void __launch_bounds__(kStemThreads, 1) stem_kernel(const __grid_constant__ StemParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem);           // full[2] empty[2] tfull[4] tempty[4]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + 512);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + 516);
  uint8_t* tiles = smem + 1024;
  uint8_t* wts = tiles + kTiles * kTileBytes;
  float* pool_rows = reinterpret_cast<float*>(wts + kKBlocks * kWBytes);
  uint8_t* in_rows = reinterpret_cast<uint8_t*>(pool_rows + 2 * 128 * kPoolPitch);
  const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * kTiles, tfull0 = empty0 + 8 * kTiles, tempty0 = tfull0 + 8 * kAccs;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int kwC = p.kw * p.C, K = p.kh * kwC;

  if (threadIdx.x == 0) {
    for (int i = 0; i < kTiles; ++i) { mbar_init(full0 + 8 * i, kProducers); mbar_init(empty0 + 8 * i, 1); }
    for (int i = 0; i < kAccs; ++i) { mbar_init(tfull0 + 8 * i, 1); mbar_init(tempty0 + 8 * i, kEpiWarps); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kProducers) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kAccs * 64) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // what nobody writes later stays zero: patch elements behind the last, pixels behind the last, image borders
  for (int i = threadIdx.x; i < (kTiles * kTileBytes + kKBlocks * kWBytes) / 16; i += kStemThreads)
    reinterpret_cast<uint4*>(tiles)[i] = make_uint4(0, 0, 0, 0);
  for (int i = threadIdx.x; i < kRows * kMaxRowPitch / 16; i += kStemThreads) reinterpret_cast<uint4*>(in_rows)[i] = make_uint4(0, 0, 0, 0);
  __syncthreads();
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (p.stamp && threadIdx.x == 32) atomicMin(p.stamp, (unsigned long long)global_timer());
  for (int i = threadIdx.x; i < p.n * K; i += kStemThreads) {
    const int n = i / K, k = i - n * K, w = (k & 63) >> 1;
    *reinterpret_cast<__nv_bfloat16*>(wts + (k >> 6) * kWBytes + n * 128 + (((w >> 2) ^ (n & 7)) << 4) + (w & 3) * 4 + (k & 1) * 2) =
        p.w[(int64_t)n * p.ldk + k];
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const uint32_t tmem_base = *tmem_slot;

  if (warp < kProducers) {
    // ------------------------------------------------------------------ producers
    // The warps meet at a named barrier, so none may leave early: after a wait that gave up they go through the
    // motions (shared memory only).
    constexpr int kThreadsP = 32 * kProducers;
    constexpr int kVec = CC ? 4 : 1;                          // elements per load
    constexpr int kAhead = (2 * kMaxW * (CC ? CC : 4) / kVec + kThreadsP - 1) / kThreadsP;   // loads of two input rows per thread
    const int C = CC ? CC : p.C;
    const int tid = threadIdx.x;
    const int row_elems = p.W * C, row_vecs = row_elems / kVec;
    const uint32_t rows0 = smem_u32(in_rows), tiles0 = smem_u32(tiles);
    // the lane's patch elements, 64 kb + 2 lane and the next one: kernel row, the word of an input row that holds each
    // at pixel 0, and how the two halves come together
    int dy[kKBlocks][2], word[kKBlocks][2];
    uint32_t pick[kKBlocks], mask[kKBlocks];
#pragma unroll
    for (int kb = 0; kb < kKBlocks; ++kb) {
      const int k = 64 * kb + 2 * lane;
      uint32_t half[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        dy[kb][e] = k + e < K ? (k + e) / kwC : 0;
        const int at = k + e < K ? kLeft - p.pad * C + (k + e) - dy[kb][e] * kwC : 0;     // element of the stored row
        word[kb][e] = (at >> 1) * 4;
        half[e] = at & 1;
      }
      pick[kb] = (half[0] ? 0x32u : 0x10u) | ((half[1] ? 0x76u : 0x54u) << 8);
      mask[kb] = k + 1 < K ? 0xffffffffu : k < K ? 0xffffu : 0u;
    }
    struct Vec { float v[kVec]; };
    auto put = [&](uint32_t slot, int f, const Vec& q) {       // load f of the input row in ring place `slot`
      uint8_t* row = in_rows + slot * p.row_bytes + (kLeft + f * kVec) * 2;
      if (CC) {
        __nv_bfloat162 h0 = __floats2bfloat162_rn(q.v[0], q.v[1 % kVec]), h1 = __floats2bfloat162_rn(q.v[2 % kVec], q.v[3 % kVec]);
        reinterpret_cast<uint32_t*>(row)[0] = *reinterpret_cast<uint32_t*>(&h0);       // rows start on four bytes
        reinterpret_cast<uint32_t*>(row)[1] = *reinterpret_cast<uint32_t*>(&h1);
      } else {
        *reinterpret_cast<__nv_bfloat16*>(row) = __float2bfloat16_rn(q.v[0]);
      }
    };
    uint32_t seq = 0, t = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < p.items; item += gridDim.x) {
      const Band b = band_of(p, item);
      const int ih0 = 2 * b.oh0 - p.pad, nr = b.oh1 - b.oh0 + 1;
      const float* img = p.x + (int64_t)b.img * p.H * row_elems;
      auto get = [&](int j, int f) {                         // load f of row j of the band (zeros outside the image)
        const int ih = ih0 + j;
        Vec q;
        if (ih >= 0 && ih < p.H) {
          const float* src = img + (int64_t)ih * row_elems + f * kVec;
          if (CC) {
            const float4 x4 = __ldg(reinterpret_cast<const float4*>(src));
            q.v[0] = x4.x; q.v[1 % kVec] = x4.y; q.v[2 % kVec] = x4.z; q.v[3 % kVec] = x4.w;
          } else {
            q.v[0] = __ldg(src);
          }
        } else {
#pragma unroll
          for (int i = 0; i < kVec; ++i) q.v[i] = 0.0f;
        }
        return q;
      };
      // all warps have built the previous band's last tile before its rows are overwritten
      asm volatile("bar.sync 2, %0;" ::"n"(kThreadsP) : "memory");
#pragma unroll 4
      for (int g = tid; g < p.kh * row_vecs; g += kThreadsP) {
        const int j = g / row_vecs, f = g - j * row_vecs;
        put((seq + j) & (kRows - 1), f, get(j, f));
      }
      Vec ahead[kAhead];
      auto load_two = [&](int j0) {
#pragma unroll
        for (int i = 0; i < kAhead; ++i) {
          const int g = tid + i * kThreadsP, second = g >= row_vecs;
          if (g < 2 * row_vecs) ahead[i] = get(j0 + second, g - second * row_vecs);
        }
      };
      if (nr > 1) load_two(p.kh);
      for (int r = 0; r < nr; ++r, ++t) {
        if (r > 0) {                                         // the two rows this output row adds
#pragma unroll
          for (int i = 0; i < kAhead; ++i) {
            const int g = tid + i * kThreadsP, second = g >= row_vecs;
            if (g < 2 * row_vecs) put((seq + p.kh + 2 * (r - 1) + second) & (kRows - 1), g - second * row_vecs, ahead[i]);
          }
          if (r + 1 < nr) load_two(p.kh + 2 * r);
        }
        asm volatile("bar.sync 2, %0;" ::"n"(kThreadsP) : "memory");
        const uint32_t a = t & (kTiles - 1);
        if (ok && !mbar_wait(empty0 + 8 * a, ((t / kTiles) & 1u) ^ 1u, abort_flag, p.err)) ok = false;
        ok = __all_sync(0xffffffffu, ok);
        if (ok) {
          uint32_t src[kKBlocks][2];
#pragma unroll
          for (int kb = 0; kb < kKBlocks; ++kb)
#pragma unroll
            for (int e = 0; e < 2; ++e)
              src[kb][e] = rows0 + ((seq + 2 * r + dy[kb][e]) & (kRows - 1)) * p.row_bytes + word[kb][e] + warp * 4 * C;
          // pixels warp, warp + 8, ...: the swizzle of the tile's row is the same for all of them
          uint32_t dst = tiles0 + a * kTileBytes + warp * 128 + (lane & 3) * 4 + (((lane >> 2) ^ (warp & 7)) << 4);
          // four at a time: all their loads are in flight before the first store needs one
          constexpr int kPix = 4;
          for (int ow0 = warp; ow0 < p.OW; ow0 += kPix * kProducers) {
            uint32_t w[kPix][kKBlocks][2];
#pragma unroll
            for (int i = 0; i < kPix; ++i)
#pragma unroll
              for (int kb = 0; kb < kKBlocks; ++kb)
#pragma unroll
                for (int e = 0; e < 2; ++e)
                  if (ow0 + i * kProducers < p.OW)
                    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(w[i][kb][e]) : "r"(src[kb][e] + i * kProducers * 4 * C) : "memory");
                  else
                    w[i][kb][e] = 0u;
#pragma unroll
            for (int i = 0; i < kPix; ++i)
#pragma unroll
              for (int kb = 0; kb < kKBlocks; ++kb) {
                const uint32_t v = __byte_perm(w[i][kb][0], w[i][kb][1], pick[kb]) & mask[kb];
                if (ow0 + i * kProducers < p.OW)
                  asm volatile("st.shared.b32 [%0], %1;" ::"r"(dst + i * kProducers * 128 + kb * (128 * 128)), "r"(v) : "memory");
              }
#pragma unroll
            for (int kb = 0; kb < kKBlocks; ++kb) { src[kb][0] += kPix * kProducers * 4 * C; src[kb][1] += kPix * kProducers * 4 * C; }
            dst += kPix * kProducers * 128;
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(full0 + 8 * a);
        }
      }
      seq += (uint32_t)(2 * (nr - 1) + p.kh);
    }
  } else if (warp == kProducers) {
    // ------------------------------------------------------------------ MMA issuer
    constexpr uint32_t kHi = (uint32_t)(1024 >> 4) | (1u << 14) | (2u << 29);      // 128B swizzle, 8-row groups 1024 bytes apart
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(p.n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
    const uint32_t a0 = smem_u32(tiles) >> 4, w0 = smem_u32(wts) >> 4;
    const bool elected = elect_one();
    const int steps = (K + 15) / 16;
    uint32_t t = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < p.items && ok; item += gridDim.x) {
      const Band b = band_of(p, item);
      for (int oh = b.oh0; oh <= b.oh1; ++oh, ++t) {
        const uint32_t a = t & (kAccs - 1), s = t & (kTiles - 1);
        if (!mbar_wait_warp(tempty0 + 8 * a, ((t / kAccs) & 1u) ^ 1u, abort_flag, p.err)) { ok = false; break; }
        if (!mbar_wait_warp(full0 + 8 * s, (t / kTiles) & 1u, abort_flag, p.err)) { ok = false; break; }
        tc_fence_after();
        if (elected) {
          for (int k = 0; k < steps; ++k) {
            const uint32_t la = a0 + s * (kTileBytes >> 4) + (k >> 2) * (128 * 128 >> 4) + 2 * (k & 3);
            const uint32_t lb = w0 + (k >> 2) * (kWBytes >> 4) + 2 * (k & 3);
            tc_mma<true>(tmem_base + a * 64, ((uint64_t)kHi << 32) | (uint64_t)((la & 0x3FFFu) | (1u << 16)),
                         ((uint64_t)kHi << 32) | (uint64_t)((lb & 0x3FFFu) | (1u << 16)), idesc, k ? 1u : 0u);
          }
          tc_commit(empty0 + 8 * s);
          tc_commit(tfull0 + 8 * a);
        }
        __syncwarp();
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue
    // The warps meet at a named barrier, so none of them may leave early: after a wait that gave up
    // they go through the motions without touching memory.
    constexpr int kThreadsE = 32 * kEpiWarps;
    const int quad = warp & 3, h = (warp - kProducers - 1) >> 2;      // lane quadrant and half of the channels
    const int ow = quad * 32 + lane;
    const int et = (warp - kProducers - 1) * 32 + lane;
    const float ninf = __int_as_float(0xff800000);
    const int n4 = p.n >> 2, pooled4 = p.PW * n4;
    uint32_t t = 0, emitted = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < p.items; item += gridDim.x) {
      const Band b = band_of(p, item);
      float m[32];                                        // maximum over the rows of the open triple
#pragma unroll
      for (int c = 0; c < 32; ++c) m[c] = ninf;
      for (int oh = b.oh0; oh <= b.oh1; ++oh, ++t) {
        const uint32_t a = t & (kAccs - 1);
        if (ok && !mbar_wait(tfull0 + 8 * a, (t / kAccs) & 1u, abort_flag, p.err)) ok = false;
        ok = __all_sync(0xffffffffu, ok);
        if (ok) tc_fence_after();
        // rows 2q - 1, 2q, 2q + 1 make pooled row q: an odd row closes one triple and opens the next
        const bool odd = oh & 1;
        const int q = oh >> 1;
        const bool emit = p.pool && (odd || oh == p.OH - 1) && q >= b.p0 && q < b.p1;
        float* stage = pool_rows + (emitted & 1u) * (128 * kPoolPitch) + ow * kPoolPitch;
        uint32_t v[32];
        if (ok) {
          tmem_ld32_issue(tmem_base + ((uint32_t)(quad * 32) << 16) + a * 64 + 32 * h, v);
          tmem_ld_wait();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(tempty0 + 8 * a);
        } else {
#pragma unroll
          for (int c = 0; c < 32; ++c) v[c] = 0u;
        }
        if (p.y && ok && ow < p.OW) {
          if (p.act == QCFG_ACT_RELU) {
#pragma unroll
            for (int c = 0; c < 32; ++c) v[c] = __float_as_uint(fmaxf(__uint_as_float(v[c]), 0.0f));
          }
          float* dst = p.y + (((int64_t)b.img * p.OH + oh) * p.OW + ow) * p.n + 32 * h;
#pragma unroll
          for (int c = 0; c < 32; c += 4)
            if (32 * h + c < p.n) *reinterpret_cast<uint4*>(dst + c) = make_uint4(v[c], v[c + 1], v[c + 2], v[c + 3]);
        }
        if (emit && ow < p.OW) {
#pragma unroll
          for (int c = 0; c < 32; c += 4)
            if (32 * h + c < p.n)
              *reinterpret_cast<float4*>(stage + 32 * h + c) =
                  make_float4(fmaxf(m[c], __uint_as_float(v[c])), fmaxf(m[c + 1], __uint_as_float(v[c + 1])),
                              fmaxf(m[c + 2], __uint_as_float(v[c + 2])), fmaxf(m[c + 3], __uint_as_float(v[c + 3])));
        }
#pragma unroll
        for (int c = 0; c < 32; ++c) m[c] = odd ? __uint_as_float(v[c]) : fmaxf(m[c], __uint_as_float(v[c]));
        if (!emit) continue;
        // two stages in turn: whoever writes a stage again has passed the barrier that follows its last reads
        asm volatile("bar.sync 1, %0;" ::"n"(kThreadsE) : "memory");
        if (ok) {
          const float* row = pool_rows + (emitted & 1u) * (128 * kPoolPitch);
          float* dst = p.pool + ((int64_t)b.img * p.PH + q) * p.PW * p.n;
          for (int i = et; i < pooled4; i += kThreadsE) {
            const int j = i / n4, c = (i - j * n4) * 4;
            float4 r = *reinterpret_cast<const float4*>(row + 2 * j * kPoolPitch + c);
            if (j > 0) {
              const float4 l = *reinterpret_cast<const float4*>(row + (2 * j - 1) * kPoolPitch + c);
              r.x = fmaxf(r.x, l.x); r.y = fmaxf(r.y, l.y); r.z = fmaxf(r.z, l.z); r.w = fmaxf(r.w, l.w);
            }
            if (2 * j + 1 < p.OW) {
              const float4 l = *reinterpret_cast<const float4*>(row + (2 * j + 1) * kPoolPitch + c);
              r.x = fmaxf(r.x, l.x); r.y = fmaxf(r.y, l.y); r.z = fmaxf(r.z, l.z); r.w = fmaxf(r.w, l.w);
            }
            if (p.act == QCFG_ACT_RELU) {                  // of the maximum: the same value as the maximum of the activated ones
              r.x = fmaxf(r.x, 0.0f); r.y = fmaxf(r.y, 0.0f); r.z = fmaxf(r.z, 0.0f); r.w = fmaxf(r.w, 0.0f);
            }
            *reinterpret_cast<float4*>(dst + (int64_t)i * 4) = r;
#pragma unroll
            for (int s = 0; s < kStemSlots; ++s) {         // as the quantize kernel rounds: clamp, half to even
              const CodeSlot& o = p.codes[s];
              if (!o.kind) break;
              auto code = [&](float x) {
                return __float_as_uint(__fadd_rn(fminf(fmaxf(__fmul_rn(x, o.inv_scale), -o.qmax), o.qmax), 12582912.0f));
              };
              const uint32_t lo = __byte_perm(code(r.x), code(r.y), 0x0040), hi = __byte_perm(code(r.z), code(r.w), 0x0040);
              *reinterpret_cast<uint32_t*>(reinterpret_cast<uint8_t*>(o.ptr) + (((int64_t)b.img * p.PH + q) * p.PW + j) * o.ld + c) = __byte_perm(lo, hi, 0x5410);
            }
          }
        }
        ++emitted;
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (p.stamp && threadIdx.x == 32) atomicMax(p.stamp + 1, (unsigned long long)global_timer());
  if (warp == kProducers) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kAccs * 64) : "memory");
  }
}

}  // namespace

int stem_init(Ctx* ctx) {
  cudaError_t e = cudaFuncSetAttribute(stem_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, kStemSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(stem_kernel<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, kStemSmem);
  return check_cuda(ctx, e, "stem smem attribute");
}

bool stem_capable(int64_t n, int in_h, int in_w, int in_c, int kh, int kw, int stride, int pad, int act) {
  if (kh < 1 || kh > kMaxKh || stride != 2 || in_c < 1 || in_c > 4 || pad < 0 || pad * in_c > kLeft || kw < 1 || kh * kw * in_c > kMaxK) return false;
  if (n < 16 || n > kMaxN || n % 16 || (act != QCFG_ACT_NONE && act != QCFG_ACT_RELU)) return false;
  if (in_h + 2 * pad < kh || in_w + 2 * pad < kw || in_w > kMaxW) return false;
  const int ow = (in_w + 2 * pad - kw) / 2 + 1;
  return ow >= 1 && ow <= 128;
}

int launch_stem(Ctx* ctx, const float* x, int64_t images, int H, int W, int C, const void* w_bf16, int64_t ldk, int64_t n, int kh, int kw,
                int pad, int act, float* y, float* pool, const CodeSlot* codes, cudaStream_t st) {
  if (images == 0) return QCFG_OK;
  StemParams p{};
  for (int s = 0; s < kStemSlots; ++s) p.codes[s] = codes[s];
  p.x = x; p.w = reinterpret_cast<const __nv_bfloat16*>(w_bf16); p.y = y; p.pool = pool;
  p.H = H; p.W = W; p.C = C; p.kh = kh; p.kw = kw; p.pad = pad; p.n = (int32_t)n; p.ldk = (int32_t)ldk; p.act = act;
  p.OH = (H + 2 * pad - kh) / 2 + 1; p.OW = (W + 2 * pad - kw) / 2 + 1;
  p.PH = (p.OH - 1) / 2 + 1; p.PW = (p.OW - 1) / 2 + 1;
  p.row_bytes = kRowBytes + ((kw * C + 1) / 2 % 32) * 4;
  p.err = err_word(ctx);
  if (((uintptr_t)y & 15) || ((uintptr_t)pool & 15)) return set_error(ctx, QCFG_EALIGN, "stem: outputs must be 16-byte aligned");
  // bands per image: the fewest output rows on the busiest CTA (a band of r pooled rows takes 2r + 1)
  const int64_t sms = sm_count(ctx);
  int64_t best = -1;
  for (int nb = 1; nb <= p.PH; ++nb) {
    const int rows = (p.PH + nb - 1) / nb, used = (p.PH + rows - 1) / rows;
    const int64_t cost = ((images * used + sms - 1) / sms) * (2 * rows + 1);
    if (best < 0 || cost < best) { best = cost; p.bands = used; p.band_rows = rows; }
  }
  if (images * p.bands > 0x7fffffff) return set_error(ctx, QCFG_ESHAPE, "stem: too many images");
  p.items = (int32_t)(images * p.bands);
  const double ops = 2.0 * (double)images * p.OH * p.OW * (double)n * kh * kw * C;
  p.stamp = prof_stamp(ctx, 1, ops);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(p.items < sms ? p.items : sms));
  cfg.blockDim = dim3(kStemThreads);
  cfg.dynamicSmemBytes = kStemSmem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  prof_begin(ctx, 1, st);
  const bool rgb = C == 3 && W % 4 == 0 && (uintptr_t)x % 16 == 0;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, rgb ? stem_kernel<3> : stem_kernel<0>, p);
  prof_end(ctx, 1, ops, st);
  if (e != cudaSuccess) return check_cuda(ctx, e, "stem launch");
  count_launch(ctx);
  return check_cuda(ctx, cudaGetLastError(), "stem launch");
}

}  // namespace qcfg
