// Quantized GEMM of a configuration evaluation: int8 x int8 -> int32 (tcgen05 kind::i8) and
// bf16 x bf16 -> fp32 (kind::f16) for 16-bit layers, with the dequantize / shortcut /
// activation / re-quantize epilogue fused in (Eq. 1's rescale 2^-(b-1)*gamma for both operands;
// the "Evaluate f(x, w)" step of Algorithms 1 and 2).
//
// Structure (one persistent CTA per SM, 576 threads):
//   warp 0      TMA producer: 128-byte-swizzled K-major tiles of A [128 x 128 B] and
//               B [BN x 128 B] into a ring of shared-memory stages (mbarrier full/empty).
//   warp 1      MMA issuer: one thread issues tcgen05.mma (M=128, N=BN, K=32 B per instruction)
//               from shared-memory descriptors into one of two TMEM accumulator buffers
//               (2 x 256 columns), and commits stage-release / accumulator-ready barriers.
//   warps 2..17 epilogue: tcgen05.ld of the accumulator (one row per thread, 16 or 32 columns per
//               load), rescale, shortcut add, activation, stores of fp32 and/or the consumer's
//               int8 / bf16 codes through shared-memory staging and TMA stores; overlaps the next
//               tile's main loop.
//   warps 18,19 (convolution launches only, 640 threads) gather the A tile of an implicit-GEMM
//               convolution from the NHWC codes of the layer's input with cp.async.
//   warps 18,19 (chained launches only, 640 threads) publish finished tiles (18) and clear tiles
//               whose input rows are complete (19): a chain runs up to 16 consecutive GEMMs of a
//               forward pass as one cooperative launch (see the kernel).
// Every wait (mbarrier, counter in shared or global memory) is bounded: after ~2 s it sets the
// context's error word and the CTA leaves through the normal teardown (TMEM is freed).
#include <cuda.h>

#include <cstring>
#include <mutex>
#include <new>
#include <unordered_map>

#include "common.cuh"
#include "ptx.cuh"

namespace qcfg {

namespace {

constexpr int BM = 128;               // rows per tile (UMMA M, cta_group::1)
constexpr int kStageKBytes = 128;     // bytes of K per stage row = one 128B swizzle atom
constexpr int kUmmaKBytes = 32;       // bytes of K per tcgen05.mma
constexpr int kEpiWarps = 16;
constexpr int kGemmThreads = 64 + 32 * kEpiWarps;
constexpr int kGatherWarps = 2;       // convolution launches only: build the A tile from the NHWC source
constexpr int kGemmThreadsConv = kGemmThreads + 32 * kGatherWarps;
constexpr int kGatherDepth = 2;       // k-blocks a gather warp keeps in flight
constexpr int kTmemCols = 512;
constexpr int kAccCols = 256;         // columns per accumulator buffer
constexpr int kMaxStages = 8;
constexpr int kSmemHeader = 1024;     // barriers and bookkeeping
constexpr int kResBarOffset = 512;    // in the header: two barriers per epilogue warp for shortcut blocks
constexpr int kShortcutBytes = 2 * 4096 + 1024;   // per epilogue warp: two 32 x 32 fp32 blocks and one of codes
constexpr int kCsBytes = kEpiWarps * 64 * 4;   // per epilogue warp: rescale factors of its 64 columns
constexpr int kSmemMax = 232448;      // 227 KB

constexpr int kNumOuts = 2 + kMaxSlots;   // raw accumulators, fp32 output, consumer code slots

struct OutDesc {
  int32_t kind;       // 0 none, 1 int8 codes, 2 bf16 codes, 3 fp32, 4 int32
  int32_t tma;        // 1: staged through shared memory and written by a TMA store
  void* ptr;
  int64_t ld;         // elements
  float inv_scale, qmax;
};
// One launch runs up to kMaxGroups GEMMs of equal m, k, operand type and tile shape ("groups":
// layers that are ready at the same time, e.g. the three projections reading one input).  Their
// column tiles are numbered one after the other, so the persistent CTAs work through all of them
// and only the first tile's main loop and the last tile's epilogue stay unoverlapped.
constexpr int kMaxGroups = 3;
// Tensor maps of a record sit in a pool; per group an index row says where its A and B operand
// maps, the map of the output a fast epilogue body writes and the maps of its outputs are.
constexpr int kMapsPerGroup = 3 + kNumOuts;
enum : int { MAP_A = 0, MAP_B = 1, MAP_FAST = 2, MAP_OUT = 3 };
constexpr int kPoolAll = kMaxGroups * kMapsPerGroup;   // a launch of its own: every map has its place
constexpr int kPoolChain = 8;                          // a record of a chain: the (distinct) maps it really uses
// Epilogue bodies.  The general one handles any combination of outputs with run-time branches; the
// common combinations have straight-line bodies (same arithmetic, same order).
enum : int32_t { EPI_GENERAL = 0, EPI_CODES1 = 1, EPI_Y = 2, EPI_SHORTCUT = 3, EPI_CODES32 = 4, EPI_BF16 = 5, EPI_Y32 = 6 };
// Fast bodies (256-column tiles only): EPI_CODES1 writes each warp's 32 x 64 int8 block with one
// TMA store (64-byte rows, 64B swizzle), EPI_Y each 32 x 32 fp32 block with one (128-byte rows,
// 128B swizzle), EPI_BF16 each warp's 32 x 64 bf16 block with one (128-byte rows, 128B swizzle), taking the maximum
// of what it writes along in the calibration forward.  EPI_SHORTCUT (int8, one CTA per tile, at most 128 columns): fp32 shortcut in, fp32 matrix and
// up to two int8 code matrices out.  EPI_CODES32 (one CTA per tile, fewer than 256 columns): one int8 code matrix.
// EPI_Y32 (int8, fewer than 256 columns, not a lone GEMM in CTA pairs): the fp32 matrix.
struct GroupDesc {
  int32_t n, tn_begin;        // columns; first column-tile index of the group in the launch's numbering
  int32_t act;
  int32_t need_y;             // anything besides raw accumulators to produce
  int32_t mode;               // EPI_*: which epilogue body serves this group
  // chains number a record's tiles group by group (column tile fastest inside a group):
  int32_t gtiles_n, tile_first;   // column tiles of this group; record-local index of its first tile (unused: INT32_MAX)
  int32_t signal;             // a later record of the launch reads this group's output rows
  float scale_x;
  const float* scale_w;
  const float* residual; int64_t ldr;
  unsigned* amax;             // optional: bit pattern of max |output| over the whole matrix (general body only)
  OutDesc outs[kNumOuts];     // [0] raw accumulators, [1] fp32 output, [2..] consumer codes
};
// Implicit-GEMM convolution: the A operand is not a matrix in memory but the NHWC code tensor of the
// layer's input; row (b, oh, ow) of the k-block (tap, channel chunk) is gathered from pixel
// (b, oh*stride - pad + dy, ow*stride - pad + dx), zero outside the image.
// How the operand gets into shared memory: gather warps (any multiple of 16 bytes of channels), or TMA in its
// im2col mode, where one load brings a chunk of channels of 128 consecutive output pixels at one tap:
// 128-byte chunks (channels a multiple of 128 bytes; the usual 128B-swizzled tile), or two 64-byte chunks
// per k-block (a multiple of 64 bytes; two half tiles of 64-byte rows, 64B swizzle).  CONV_SLAB: see SlabDesc.
enum : int32_t { CONV_NONE = 0, CONV_GATHER = 1, CONV_TMA128 = 2, CONV_TMA64 = 3, CONV_SLAB = 4 };
struct ConvDesc {
  int32_t on, H, W, C, kh, kw, stride, pad, OH, OW, esz, K;
  int64_t img_bytes;          // bytes of one image (H * W * C * esz)
  const uint8_t* src;
};
// Stride-1 3x3 convolutions whose only output is one int8 code matrix read their input once per tile, not once per tap: a
// tile is tw x rows output pixels of `imgs` images, and one tiled TMA load per channel chunk brings all input pixels
// its taps touch (a slab of `pitch` pixels per row, zeros outside the image).  The A operand of tap (dy, dx) is
// then simply the 128 slab pixels from dy * pitch + dx on: row r of the tile is the output pixel at linear slab position r, and
// positions that are no output pixel (the halo at the right of a row, the rows between two images) are
// computed and not stored.  A whole-width tile shares the halo: the zeros left of a row stand right of the row before
// (right of the last row: zeros the kernel puts behind each slab once).
struct SlabDesc {
  int32_t pitch, tw, rows, imgs;        // slab pixels per row; output columns, rows and images of a tile
  int32_t img_pitch;                    // slab pixels per image
  int32_t tiles_w, tiles_h, images;
  int32_t chunk, chunks;                // channel bytes per load (64 or 128), loads per tile
  int32_t bytes, tx_bytes, count;       // slab size in the ring (whole 1024 bytes, also what the last tap reads), bytes loaded, slabs in the ring
  int32_t resident;                     // one chunk, one column tile: all weights stay in shared memory, a stage (and barrier) per tap
};
constexpr int kMaxSlabs = 4;
constexpr int kSlabRoom = kSmemMax - kSmemHeader - kCsBytes - 1024;      // shared memory for slabs and weights
constexpr int kMaxDeps = 4;
struct GemmParams {
  int32_t m, k_blocks, bn, tiles_m, tiles_n, stages, is_bf16;   // tiles_n: column tiles of all groups together
  int32_t epi_bytes;          // staging bytes per epilogue warp
  int32_t alternate;          // tiles of 64 columns: half of the epilogue warps take the even tiles, half the odd ones
  uint32_t idesc;
  GroupDesc grp[kMaxGroups];  // unused groups have tn_begin = INT32_MAX
  unsigned* err;
  unsigned long long* stamp;  // optional [2]: earliest start / latest end of the launch's CTAs (%globaltimer, ns)
  ConvDesc conv;              // conv.on: A comes from the gather warps (single-group launches only)
  SlabDesc slab;
  // chains: records of the same launch whose output rows this record reads (-1: none), and
  // whether a later record of the launch reads this one's
  uint8_t mi[kMaxGroups][kMapsPerGroup];   // pool indices of the groups' tensor maps
  int32_t deps[kMaxDeps];
  int32_t need;               // finished tiles per row tile and CTA rank that make this record's rows complete for its readers
};
// What one launch gets: one record, or a chain of them (see the kernel).
constexpr int kChainMax = 16;
template <int POOL> struct Rec { CUtensorMap m[POOL]; GemmParams p; };
template <bool CHAIN> struct LaunchArgs {
  Rec<CHAIN ? kPoolChain : kPoolAll> rec[CHAIN ? kChainMax : 1];
  int32_t n;             // records in use
  int32_t total_tiles;   // tiles of all records together
  int32_t flag_stride;   // counters per record (two per row tile: one per CTA of the pair)
  unsigned* flags;       // [n x flag_stride], zero when the launch starts
};
static_assert(sizeof(LaunchArgs<true>) <= 32764, "kernel parameters are limited to 32764 bytes");

// ---------------------------------------------------------------------------- PTX wrappers

// Chains: waits until a counter of finished tiles has reached `need`.  Bounded like every other wait.
__device__ __forceinline__ bool flag_wait(const unsigned* flag, uint32_t need, volatile int* abort_flag, unsigned* err,
                                          uint64_t limit_ns = kWaitLimitNs) {
  uint64_t t0 = 0;
  for (uint32_t it = 1;; ++it) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(flag) : "memory");
    if (v >= need) return true;
    __nanosleep(100);        // the warp that polls is ahead of the producer; it need not spin at full rate
    if ((it & 63u) == 0) {
      if (*abort_flag) return false;
      const uint64_t now = global_timer();
      if (t0 == 0) t0 = now;
      else if (now - t0 > limit_ns) {
        atomicOr(err, ERR_TIMEOUT);
        *abort_flag = 1;
        return false;
      }
    }
  }
}

// Chains: waits until the CTA's dependency warp has cleared `need` tiles (a counter in shared memory).
__device__ __forceinline__ bool cleared_wait(uint32_t addr, uint32_t need, volatile int* abort_flag, unsigned* err,
                                             uint64_t limit_ns = kWaitLimitNs) {
  uint64_t t0 = 0;
  for (uint32_t it = 1;; ++it) {
    uint32_t v;
    asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    if (v >= need) return true;
    __nanosleep(40);
    if ((it & 1023u) == 0) {
      if (*abort_flag) return false;
      const uint64_t now = global_timer();
      if (t0 == 0) t0 = now;
      else if (now - t0 > limit_ns) {
        atomicOr(err, ERR_TIMEOUT);
        *abort_flag = 1;
        return false;
      }
    }
  }
}

// Chains: waits (whole warp) until every epilogue warp has reported `need` tiles; lane w reads warp w's counter.
__device__ __forceinline__ bool reported_wait(uint32_t rep0, uint32_t need, int lane, volatile int* abort_flag, unsigned* err,
                                              uint64_t limit_ns = kWaitLimitNs) {
  uint64_t t0 = 0;
  for (uint32_t it = 1;; ++it) {
    uint32_t v = need;
    if (lane < kEpiWarps) asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(rep0 + 4 * lane) : "memory");
    if (__all_sync(0xffffffffu, v >= need)) return true;
    __nanosleep(40);
    if ((it & 1023u) == 0) {
      bool give_up = *abort_flag != 0;
      const uint64_t now = global_timer();
      if (t0 == 0) t0 = now;
      else if (now - t0 > limit_ns) {
        if (lane == 0) { atomicOr(err, ERR_TIMEOUT); *abort_flag = 1; }
        give_up = true;
      }
      if (__any_sync(0xffffffffu, give_up)) return false;
    }
  }
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int32_t x, int32_t y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y) : "memory");
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int32_t c, int32_t w, int32_t h, int32_t n) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c), "r"(w), "r"(h), "r"(n) : "memory");
}
// im2col loads: (w, h) is the first pixel's corner of the filter window, (dx, dy) the tap
__device__ __forceinline__ void tma_load_im2col(uint32_t dst, const CUtensorMap* map, uint32_t bar, int32_t c, int32_t w, int32_t h, int32_t n,
                                                int dx, int dy) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.im2col.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2], {%7, %8};"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c), "r"(w), "r"(h), "r"(n), "h"((uint16_t)dx), "h"((uint16_t)dy) : "memory");
}

// Pair flavour (two CTAs of a cluster work on one 256-row tile, cta_group::2): the load of either
// CTA reports its bytes to the barrier of the pair's first CTA; shared-memory addresses of the
// two CTAs differ in bit 24 of the shared::cluster window.
constexpr uint32_t kPeerBitMask = 0xFEFFFFFFu;
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar, int32_t x, int32_t y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar & kPeerBitMask), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void tma_load_4d_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar, int32_t c, int32_t w, int32_t h, int32_t n) {
  asm volatile(
      "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar & kPeerBitMask), "r"(c), "r"(w), "r"(h), "r"(n) : "memory");
}
__device__ __forceinline__ void tma_load_im2col_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar, int32_t c, int32_t w, int32_t h,
                                                     int32_t n, int dx, int dy) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.im2col.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%3, %4, %5, %6}], [%2], {%7, %8};"
      ::"r"(dst), "l"(map), "r"(bar & kPeerBitMask), "r"(c), "r"(w), "r"(h), "r"(n), "h"((uint16_t)dx), "h"((uint16_t)dy) : "memory");
}
__device__ __forceinline__ void mbar_arrive_leader(uint32_t bar) {   // arrive on the first CTA's copy of the barrier
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar & kPeerBitMask) : "memory");
}
__device__ __forceinline__ void tc_commit_pair(uint32_t bar) {       // arrives on this barrier in both CTAs
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(bar), "h"((uint16_t)3) : "memory");
}
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <bool BF16>
__device__ __forceinline__ void tc_mma_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  if (BF16) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
  } else {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::i8 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
  }
}

__device__ __forceinline__ void tmem_ld16_issue(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr));
}
// Shared-memory matrix descriptors used by the MMA issuer: K-major tile of 128-byte rows, 128B
// swizzle, groups of 8 rows 1024 bytes apart (the layout a 128B-swizzled TMA box produces).
// Bits 0-13 start address in 16-byte units, bit 16 leading byte offset (unused for swizzled
// K-major), bits 32-45 stride byte offset between 8-row groups (1024 >> 4), bit 46 descriptor
// version of sm_100, bits 61-63 layout type 2 = SWIZZLE_128B.

// ---------------------------------------------------------------------------- epilogue math

// int8 code of Eq. 1 in the low byte of the returned word: clamp, then add 1.5*2^23 (a
// round-half-even at integer granularity); the low mantissa byte is the two's-complement code.
__device__ __forceinline__ uint32_t code_word(float y, float inv_scale, float qmax) {
  const float t = __fmul_rn(y, inv_scale);
  // clamp to [-qmax, qmax] in one instruction: magnitude min(|t|, qmax), sign of t (qmax > 0)
  float c;
  asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(c) : "f"(t), "f"(qmax));
  return __float_as_uint(__fadd_rn(c, 12582912.0f));
}
// low bytes of four words -> one word (byte i from word i)
__device__ __forceinline__ uint32_t pack4(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  return __byte_perm(__byte_perm(a, b, 0x0040), __byte_perm(c, d, 0x0040), 0x5410);
}

__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int32_t x, int32_t y) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
               ::"l"(map), "r"(src), "r"(x), "r"(y) : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// Writes one warp's 32-row x 32-column piece of an output.  Each thread holds its row's 32
// elements packed into WORDS 32-bit words (32: fp32 / int32, 16: bf16, 8: int8).
// Staged path: the warp lays the piece out in one of its two shared-memory slots and one lane
// issues a TMA store, which writes whole rows and clips at the matrix edge.  Outputs TMA cannot write
// (pointer or row pitch not 16-byte aligned): 4-byte elements are turned in the staging buffer and
// stored row by row, narrower ones go out from each lane's registers.
template <int WORDS>
__device__ __forceinline__ void store_piece(const OutDesc& o, const CUtensorMap* map, const uint32_t (&w)[WORDS],
                                            bool row_ok, int ncols, int64_t row, int row0, int col0,
                                            uint32_t stage, uint32_t stage_bytes, uint32_t& cursor, int lane) {
  constexpr int kRowBytes = WORDS * 4;
  constexpr int kElemBytes = kRowBytes / 32;
  if (o.tma) {
    // The warp's buffer holds two slots used alternately: before a slot is rewritten only the
    // store issued two pieces ago must have been read by the TMA engine (at most one store
    // stays pending).  4-byte outputs go out as two 16-column pieces of 64-byte rows (64B
    // swizzle: the 16-byte writes of eight lanes then cover all banks).
    const uint32_t slot_bytes = stage_bytes >> 1;
    constexpr int kHalves = (WORDS == 32) ? 2 : 1;
#pragma unroll
    for (int h = 0; h < kHalves; ++h) {
      if (h == 1 && ncols <= 16) break;                 // warp-uniform: the second half lies outside
      if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
      __syncwarp();
      const uint32_t base = stage + (cursor & 1u) * slot_bytes;
      ++cursor;
      if (WORDS == 32) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int js = j ^ ((lane >> 1) & 3);
          st_shared_v4(base + lane * 64 + js * 16, w[16 * h + 4 * j], w[16 * h + 4 * j + 1], w[16 * h + 4 * j + 2], w[16 * h + 4 * j + 3]);
        }
      } else {
#pragma unroll
        for (int j = 0; j < WORDS / 4; ++j)
          st_shared_v4(base + lane * kRowBytes + j * 16, w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) tma_store_2d(map, base, col0 + 16 * h, row0);
    }
    return;
  }
  if constexpr (WORDS == 32) {
    // A 4-byte output TMA cannot write (row pitch not a multiple of 16 bytes); every launch with one has 4 KB of staging.  The lanes hold one
    // row each, so stores straight from registers would touch 32 rows per instruction; instead the
    // piece is turned in the warp's staging buffer (16-byte chunks swizzled by the row, no bank
    // conflicts either way) and goes out row by row, 32 consecutive words per instruction.
    // 4099 x 3085 x 771, quantize and GEMM together: 93.8 us with per-lane rows, 32.4 us this way (rows unrolled by
    // sixteen; by eight 33.4).
    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // other outputs' stores read the same buffer
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 8; ++j)
      st_shared_v4(stage + lane * 128 + ((j ^ (lane & 7)) << 4), w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
    const int nrows = __popc(__ballot_sync(0xffffffffu, row_ok));
    __syncwarp();
    uint32_t* out = reinterpret_cast<uint32_t*>(o.ptr) + (int64_t)row0 * o.ld + col0 + lane;
#pragma unroll 16
    for (int i = 0; i < nrows; ++i) {
      uint32_t x;
      asm volatile("ld.shared.b32 %0, [%1];" : "=r"(x) : "r"(stage + i * 128 + (((lane >> 2) ^ (i & 7)) << 4) + (lane & 3) * 4) : "memory");
      if (lane < ncols) *out = x;
      out += o.ld;
    }
    __syncwarp();
  } else {
    if (!row_ok) return;
    uint8_t* dst = reinterpret_cast<uint8_t*>(o.ptr) + (row * o.ld + col0) * kElemBytes;
    if (ncols >= 32 && (reinterpret_cast<uintptr_t>(dst) & 15) == 0) {
#pragma unroll
      for (int j = 0; j < WORDS / 4; ++j)
        reinterpret_cast<uint4*>(dst)[j] = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
    } else {
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        if (i < ncols) {
          if (kElemBytes == 2) reinterpret_cast<uint16_t*>(dst)[i] = (uint16_t)(w[i >> 1] >> (16 * (i & 1)));
          else dst[i] = (uint8_t)(w[i >> 2] >> (8 * (i & 3)));
        }
      }
    }
  }
}

// ---- fast epilogue bodies -------------------------------------------------------------------
// Two values at a time with packed fp32 instructions (same roundings as the scalar forms: each
// half is an independent round-to-nearest operation).
__device__ __forceinline__ float2 gelu_tanh2(float2 y) {
  const float2 c1 = make_float2(-2.302208198f, -2.302208198f), c3 = make_float2(-0.1029432396f, -0.1029432396f);
  const float2 y2 = __fmul2_rn(y, y);
  const float2 t = __fmul2_rn(y, __ffma2_rn(c3, y2, c1));
  float2 e;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.x) : "f"(t.x));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.y) : "f"(t.y));
  const float2 d = __fadd2_rn(e, make_float2(1.0f, 1.0f));
  float2 r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(d.x));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(d.y));
  return __fmul2_rn(y, r);
}
// Rescaled and activated values of 16 accumulator columns of one row.  cs points to the 16
// rescale factors of these columns in shared memory (every lane reads the same addresses).
template <bool BF16>
__device__ __forceinline__ void sub_values(float2 (&y)[8], const uint32_t (&v)[16], const float* cs, int act) {
  if (BF16) {
#pragma unroll
    for (int i = 0; i < 8; ++i) y[i] = make_float2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 c = *reinterpret_cast<const float4*>(cs + 4 * q);
      y[2 * q] = __fmul2_rn(make_float2((float)(int32_t)v[4 * q], (float)(int32_t)v[4 * q + 1]), make_float2(c.x, c.y));
      y[2 * q + 1] = __fmul2_rn(make_float2((float)(int32_t)v[4 * q + 2], (float)(int32_t)v[4 * q + 3]), make_float2(c.z, c.w));
    }
  }
  if (act == QCFG_ACT_RELU) {
#pragma unroll
    for (int i = 0; i < 8; ++i) y[i] = make_float2(fmaxf(y[i].x, 0.0f), fmaxf(y[i].y, 0.0f));
  } else if (act == QCFG_ACT_GELU_TANH) {
#pragma unroll
    for (int i = 0; i < 8; ++i) y[i] = gelu_tanh2(y[i]);
  }
}
// int8 codes of Eq. 1 for two values, each in the low byte of its word
__device__ __forceinline__ float2 code_words2(float2 y, float2 inv2, float qmax) {
  const float2 t = __fmul2_rn(y, inv2);
  float2 c;
  asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(c.x) : "f"(t.x), "f"(qmax));
  asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(c.y) : "f"(t.y), "f"(qmax));
  return __fadd2_rn(c, make_float2(12582912.0f, 12582912.0f));
}

// One warp's share of a 256-column tile (32 rows x 64 columns) in four pieces of 16 columns.
// The accumulator load of the next piece is in flight while the current one is processed; the
// accumulator buffer is released as soon as the last piece sits in registers.
// OUT = EPI_CODES1: one int8 matrix, the warp's 32 x 64 block staged in 64-byte rows (64B swizzle) and
// written by one TMA store.  EPI_BF16: one bf16 matrix, the block staged in 128-byte rows (128B swizzle), one
// store; with amax set its range as well (rows and columns outside the matrix are zero and do not
// count).  Calibration of a 12-block BERT-base stack, whose GEMMs mostly write that way: 2121 us in the
// general body, 2046 us here.
// EPI_Y: the fp32 matrix, each 32 x 32 block staged in 128-byte
// rows (128B swizzle), one TMA store per block; the single staging slot is reused once the
// previous store has read it.
// rep_addr (chains, else 0): this warp's report counter in shared memory, set to rep_val once the
// stores the warp issued for its previous tile have completed; that is checked after this tile's
// first piece, a quarter of an epilogue after they were issued.
template <bool BF16, bool PAIR, int OUT>
__device__ __forceinline__ void epilogue_tile_fast(const GroupDesc& G, const CUtensorMap* fmap, uint32_t tbase,
                                                   const float* cs, uint32_t stage, int row0, int col0, int lane,
                                                   uint32_t tempty_bar, uint32_t rep_addr, uint32_t rep_val) {
  constexpr bool CODES = OUT == EPI_CODES1, Y = OUT == EPI_Y;
  const int act = G.act;
  unsigned mx = 0;
  const float qmax = G.outs[2].qmax;
  const float2 inv2 = make_float2(G.outs[2].inv_scale, G.outs[2].inv_scale);
  uint32_t va[16], vb[16];
  if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // the slot's last store was a tile ago
  __syncwarp();
  tmem_ld16_issue(tbase, va);
  auto piece = [&](const uint32_t (&v)[16], int s) {
    float2 y[8];
    sub_values<BF16>(y, v, cs + 16 * s, act);
    if (CODES) {
      uint32_t w[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float2 a = code_words2(y[2 * j], inv2, qmax), b = code_words2(y[2 * j + 1], inv2, qmax);
        w[j] = pack4(__float_as_uint(a.x), __float_as_uint(a.y), __float_as_uint(b.x), __float_as_uint(b.y));
      }
      st_shared_v4(stage + lane * 64 + ((s ^ ((lane >> 1) & 3)) << 4), w[0], w[1], w[2], w[3]);
    } else if (OUT == EPI_BF16) {
      if (G.amax) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const unsigned a0 = abs_bits(y[j].x), a1 = abs_bits(y[j].y), a = a0 > a1 ? a0 : a1;
          mx = mx > a ? mx : a;
        }
      }
      uint32_t w[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        __nv_bfloat162 h = __floats2bfloat162_rn(y[j].x, y[j].y);
        w[j] = *reinterpret_cast<uint32_t*>(&h);
      }
      st_shared_v4(stage + lane * 128 + (((2 * s) ^ (lane & 7)) << 4), w[0], w[1], w[2], w[3]);
      st_shared_v4(stage + lane * 128 + (((2 * s + 1) ^ (lane & 7)) << 4), w[4], w[5], w[6], w[7]);
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int p16 = 4 * (s & 1) + j;
        st_shared_v4(stage + lane * 128 + ((p16 ^ (lane & 7)) << 4), __float_as_uint(y[2 * j].x), __float_as_uint(y[2 * j].y),
                     __float_as_uint(y[2 * j + 1].x), __float_as_uint(y[2 * j + 1].y));
      }
    }
  };
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    tmem_ld_wait();
    tmem_ld16_issue(tbase + 32 * h + 16, vb);
    if (Y && h == 1) {   // the first block's store must have read the slot before it is refilled
      if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
      __syncwarp();
    }
    piece(va, 2 * h);
    if (h == 0 && rep_addr && lane == 0) {    // a quarter of a tile after the previous tile's last store
      asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
      asm volatile("st.release.cta.shared::cta.u32 [%0], %1;" ::"r"(rep_addr), "r"(rep_val) : "memory");
    }
    tmem_ld_wait();
    if (h == 0) {
      tmem_ld16_issue(tbase + 32, va);
    } else {          // every column of this warp is in registers: the accumulator buffer is free
      tc_fence_before();
      __syncwarp();
      if (lane == 0) { if (PAIR) mbar_arrive_leader(tempty_bar); else mbar_arrive(tempty_bar); }
    }
    piece(vb, 2 * h + 1);
    if (Y) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0 && col0 + 32 * h < G.n) tma_store_2d(fmap, stage, col0 + 32 * h, row0);
    }
  }
  if (!Y) {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
    if (lane == 0) tma_store_2d(fmap, stage, col0, row0);
  }
  if (OUT == EPI_BF16 && G.amax) {
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0 && mx) atomicMax(G.amax, mx);
  }
}

// One 32-column chunk of one accumulator row (all 32 lanes of the warp call this together).
template <bool BF16, bool CHAIN>
__device__ __forceinline__ void epilogue_chunk(const GroupDesc& p, const CUtensorMap* pool, const uint8_t* mi, int m, uint32_t epi_bytes,
                                               uint32_t (&v)[32], float cs_lane,
                                               int64_t row, int row0, int col0, uint32_t stage, uint32_t& cursor, int lane) {
  const int ncols = p.n - col0;                    // valid columns in this chunk (may be <= 0 or > 32)
  if (ncols <= 0 || row0 >= m) return;             // warp-uniform: the piece lies outside the matrix
  const bool row_ok = row < m;
  const bool full = ncols >= 32;

  if (!BF16 && p.outs[0].kind) store_piece<32>(p.outs[0], &pool[mi[MAP_OUT]], v, row_ok, ncols, row, row0, col0, stage, epi_bytes, cursor, lane);
  if (!p.need_y) return;

  float y[32];
  if (BF16) {
#pragma unroll
    for (int i = 0; i < 32; ++i) y[i] = __uint_as_float(v[i]);
  } else {
    // lane i holds scale_x * scale_w[col0 + i] (loaded before the accumulator was ready)
#pragma unroll
    for (int i = 0; i < 32; ++i)
      y[i] = __fmul_rn((float)(int32_t)v[i], __shfl_sync(0xffffffffu, cs_lane, i));
  }
  if (p.residual && row_ok) {
    // In a chain another SM may have written the shortcut earlier in this launch, so it is read
    // with ordinary loads, not through the read-only path.  (A stale L1 line is impossible: within a
    // launch every address is written at most once and read only after that write has been seen.)
    const float* r = p.residual + row * p.ldr + col0;
    if (full && (p.ldr & 3) == 0 && (((uintptr_t)p.residual) & 15) == 0) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 r4 = CHAIN ? *(reinterpret_cast<const float4*>(r) + i) : __ldg(reinterpret_cast<const float4*>(r) + i);
        y[4 * i + 0] = __fadd_rn(y[4 * i + 0], r4.x);
        y[4 * i + 1] = __fadd_rn(y[4 * i + 1], r4.y);
        y[4 * i + 2] = __fadd_rn(y[4 * i + 2], r4.z);
        y[4 * i + 3] = __fadd_rn(y[4 * i + 3], r4.w);
      }
    } else {
#pragma unroll
      for (int i = 0; i < 32; ++i) if (i < ncols) y[i] = __fadd_rn(y[i], CHAIN ? r[i] : __ldg(r + i));
    }
  }
  if (p.act == QCFG_ACT_RELU) {
#pragma unroll
    for (int i = 0; i < 32; ++i) y[i] = fmaxf(y[i], 0.0f);
  } else if (p.act == QCFG_ACT_GELU_TANH) {
#pragma unroll
    for (int i = 0; i < 32; ++i) y[i] = gelu_tanh(y[i]);
  }
  if (p.amax) {     // calibration: the range of what the consumers will read (bit patterns, exact in any order)
    unsigned mx = 0;
    if (row_ok) {
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        const unsigned a = __float_as_uint(y[i]) & 0x7fffffffu;
        if (i < ncols) mx = mx > a ? mx : a;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned other = __shfl_xor_sync(0xffffffffu, mx, o);
      mx = mx > other ? mx : other;
    }
    if (lane == 0 && mx) atomicMax(p.amax, mx);
  }
  if (p.outs[1].kind) {
    uint32_t w[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) w[i] = __float_as_uint(y[i]);
    store_piece<32>(p.outs[1], &pool[mi[MAP_OUT + 1]], w, row_ok, ncols, row, row0, col0, stage, epi_bytes, cursor, lane);
  }
#pragma unroll
  for (int s = 0; s < kMaxSlots; ++s) {
    const OutDesc& o = p.outs[2 + s];
    if (o.kind == 1) {
      uint32_t w[8];
#pragma unroll
      for (int i = 0; i < 8; ++i)
        w[i] = pack4(code_word(y[4 * i], o.inv_scale, o.qmax), code_word(y[4 * i + 1], o.inv_scale, o.qmax),
                     code_word(y[4 * i + 2], o.inv_scale, o.qmax), code_word(y[4 * i + 3], o.inv_scale, o.qmax));
      store_piece<8>(o, &pool[mi[MAP_OUT + 2 + s]], w, row_ok, ncols, row, row0, col0, stage, epi_bytes, cursor, lane);
    } else if (o.kind == 2) {
      uint32_t w[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        __nv_bfloat162 h = __floats2bfloat162_rn(y[2 * i], y[2 * i + 1]);
        w[i] = *reinterpret_cast<uint32_t*>(&h);
      }
      store_piece<16>(o, &pool[mi[MAP_OUT + 2 + s]], w, row_ok, ncols, row, row0, col0, stage, epi_bytes, cursor, lane);
    }
  }
}

// One warp's 32 x 32 block of a layer whose only output is one int8 code matrix, in tiles narrower than 256
// columns (the convolutions of 64 and 128 channels and the 1x1 layers in front of them).  One accumulator
// load, broadcast scales, one TMA store of 32-byte rows; tiles of 64 columns are taken by one half of the epilogue
// warps or the other in turn.  401408 x 64 x 256: 40.7 us in the general body, 25.1 us here; 100352 x 128 x 512:
// 20.0 -> 16.8 us.
template <bool BF16>
__device__ __forceinline__ void epilogue_codes32(const GroupDesc& G, const CUtensorMap* map, uint32_t tbase, const float* cs, uint32_t stage,
                                                 int row0, int col0, bool inside, int lane, uint32_t tempty_bar) {
  uint32_t v[32];
  tmem_ld32_issue(tbase, v);
  tmem_ld_wait();
  tc_fence_before();
  __syncwarp();
  if (lane == 0) mbar_arrive(tempty_bar);
  const float2 inv2 = make_float2(G.outs[2].inv_scale, G.outs[2].inv_scale);
  const float qmax = G.outs[2].qmax;
  uint32_t w[8];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t part[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) part[i] = v[16 * h + i];
    float2 y[8];
    sub_values<BF16>(y, part, cs + 16 * h, G.act);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float2 a = code_words2(y[2 * j], inv2, qmax), b = code_words2(y[2 * j + 1], inv2, qmax);
      w[4 * h + j] = pack4(__float_as_uint(a.x), __float_as_uint(a.y), __float_as_uint(b.x), __float_as_uint(b.y));
    }
  }
  if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // the last tile's store has read the slot
  __syncwarp();
  st_shared_v4(stage + lane * 32, w[0], w[1], w[2], w[3]);
  st_shared_v4(stage + lane * 32 + 16, w[4], w[5], w[6], w[7]);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncwarp();
  if (lane == 0 && inside) tma_store_2d(map, stage, col0, row0);
}

// One warp's 32 x 32 block of an int8 layer whose only output is the fp32 matrix, in tiles narrower than 256 columns (launches
// of one tile per CTA, whose epilogue nothing hides): broadcast scales, one TMA store of 128-byte rows.  The general body
// shuffles a scale per element and stores twice; 3072 x 768 x 3072 took 2.7 us there from the last product to the last store.
// Two blocks of 768 at 384 rows: 60.5 us there, 59.1 here; ResNet-50 of 16 images of 64 x 64 225.8 / 221.8.  16-bit layers
// need no scales and gain nothing.  A lone GEMM in CTA pairs keeps the general body: it gains 0.05 us from this one, whose code
// in that kernel, the one of the plain 256-column launches, cost every launch 0.25 (4096 x 1024 x 1024 with its quantize 12.97
// and 12.62 us, three such layers 28.1 and 27.2).  In groups of pairs it stays (a block at 3072 rows with its q and k
// outputs: 45.6 us without, 45.3 with).
template <bool PAIR>
__device__ __forceinline__ void epilogue_y32(const GroupDesc& G, const CUtensorMap* map, uint32_t tbase, const float* cs, uint32_t stage,
                                             int row0, int col0, bool inside, int lane, uint32_t tempty_bar) {
  uint32_t v[32];
  tmem_ld32_issue(tbase, v);
  if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // the last tile's store has read the slot
  tmem_ld_wait();
  tc_fence_before();
  __syncwarp();
  if (lane == 0) { if (PAIR) mbar_arrive_leader(tempty_bar); else mbar_arrive(tempty_bar); }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t part[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) part[i] = v[16 * h + i];
    float2 y[8];
    sub_values<false>(y, part, cs + 16 * h, G.act);
#pragma unroll
    for (int j = 0; j < 4; ++j)
      st_shared_v4(stage + lane * 128 + (((4 * h + j) ^ (lane & 7)) << 4), __float_as_uint(y[2 * j].x), __float_as_uint(y[2 * j].y),
                   __float_as_uint(y[2 * j + 1].x), __float_as_uint(y[2 * j + 1].y));
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncwarp();
  if (lane == 0 && inside) tma_store_2d(map, stage, col0, row0);
}

// One warp's 32 x 32 block of a shortcut layer.  The shortcut block has been brought into `block` by TMA (128-byte
// rows, 128B swizzle) while the previous tile was worked on; the sum goes back to the same place and out
// from there, so the block is both the staging of the load and of the store, and no global load sits on the
// tile's path: with per-lane loads of a row each (32 rows per instruction, waited for in every chunk) the warps
// spent ten cycles per issued instruction on them.  ResNet-50 at batch 128, sixteen such layers: 3844 us per
// evaluation before, 3492 us this way.
// Arithmetic and order are those of epilogue_chunk.
__device__ __forceinline__ void epilogue_shortcut(const GroupDesc& G, const CUtensorMap* pool, const uint8_t* mi, uint32_t tbase, const float* cs,
                                                  uint32_t block, uint32_t codes, int row0, int col0, int lane, uint32_t tempty_bar,
                                                  uint32_t res_bar, uint32_t res_parity, bool inside, volatile int* abort_flag, unsigned* err, bool& ok) {
  uint32_t v[32];
  tmem_ld32_issue(tbase, v);
  tmem_ld_wait();
  tc_fence_before();
  __syncwarp();
  if (lane == 0) mbar_arrive(tempty_bar);
  if (!mbar_wait(res_bar, res_parity, abort_flag, err)) ok = false;
  if (!__all_sync(0xffffffffu, ok)) { ok = false; return; }
  const int act = G.act;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const uint32_t at = block + lane * 128 + ((j ^ (lane & 7)) << 4);
    float4 r;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(r.x), "=f"(r.y), "=f"(r.z), "=f"(r.w) : "r"(at) : "memory");
    const float4 c = *reinterpret_cast<const float4*>(cs + 4 * j);
    float y0 = __fadd_rn(__fmul_rn((float)(int32_t)v[4 * j], c.x), r.x), y1 = __fadd_rn(__fmul_rn((float)(int32_t)v[4 * j + 1], c.y), r.y);
    float y2 = __fadd_rn(__fmul_rn((float)(int32_t)v[4 * j + 2], c.z), r.z), y3 = __fadd_rn(__fmul_rn((float)(int32_t)v[4 * j + 3], c.w), r.w);
    if (act == QCFG_ACT_RELU) {
      y0 = fmaxf(y0, 0.0f); y1 = fmaxf(y1, 0.0f); y2 = fmaxf(y2, 0.0f); y3 = fmaxf(y3, 0.0f);
    } else if (act == QCFG_ACT_GELU_TANH) {
      y0 = gelu_tanh(y0); y1 = gelu_tanh(y1); y2 = gelu_tanh(y2); y3 = gelu_tanh(y3);
    }
    v[4 * j] = __float_as_uint(y0); v[4 * j + 1] = __float_as_uint(y1); v[4 * j + 2] = __float_as_uint(y2); v[4 * j + 3] = __float_as_uint(y3);
    st_shared_v4(at, v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
  }
  bool y_out = G.outs[1].kind != 0;
#pragma unroll 1
  for (int s = 0; s < 2; ++s) {
    const OutDesc& o = G.outs[2 + s];
    if (s == 1 && !o.kind) break;
    if (s == 1) {                                // the second matrix takes the place of the first one's codes
      if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
      __syncwarp();
    }
    if (o.kind) {
      uint32_t w[8];
#pragma unroll
      for (int i = 0; i < 8; ++i)
        w[i] = pack4(code_word(__uint_as_float(v[4 * i]), o.inv_scale, o.qmax), code_word(__uint_as_float(v[4 * i + 1]), o.inv_scale, o.qmax),
                     code_word(__uint_as_float(v[4 * i + 2]), o.inv_scale, o.qmax), code_word(__uint_as_float(v[4 * i + 3]), o.inv_scale, o.qmax));
      st_shared_v4(codes + lane * 32, w[0], w[1], w[2], w[3]);
      st_shared_v4(codes + lane * 32 + 16, w[4], w[5], w[6], w[7]);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
    if (lane == 0 && inside) {
      if (y_out) tma_store_2d(&pool[mi[MAP_FAST]], block, col0, row0);
      if (o.kind) tma_store_2d(&pool[mi[MAP_OUT + 2 + s]], codes, col0, row0);
    }
    y_out = false;
  }
}

// One warp's 32 rows x (32 * nch) columns of a slab convolution: codes go from the registers to the rows' pixels, 32 bytes
// per lane and chunk (whole sectors), because the 32 rows are no box of the output matrix.  dst: this lane's row at
// the warp's first column, or null where the row is no output pixel.
template <bool PAIR>
__device__ __forceinline__ void epilogue_slab(const GroupDesc& G, uint32_t tbase, const float* cs, int nch, uint8_t* dst, int lane, uint32_t tempty_bar) {
  const float2 inv2 = make_float2(G.outs[2].inv_scale, G.outs[2].inv_scale);
  const float qmax = G.outs[2].qmax;
  const int act = G.act;
  uint32_t v[32];
#pragma unroll 1
  for (int c = 0; c < nch; ++c) {
    tmem_ld32_issue(tbase + 32 * c, v);
    tmem_ld_wait();
    if (c == nch - 1) {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) { if (PAIR) mbar_arrive_leader(tempty_bar); else mbar_arrive(tempty_bar); }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      uint32_t part[16], w[4];
#pragma unroll
      for (int i = 0; i < 16; ++i) part[i] = v[16 * h + i];
      float2 y[8];
      sub_values<false>(y, part, cs + 32 * c + 16 * h, act);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float2 a = code_words2(y[2 * j], inv2, qmax), b = code_words2(y[2 * j + 1], inv2, qmax);
        w[j] = pack4(__float_as_uint(a.x), __float_as_uint(a.y), __float_as_uint(b.x), __float_as_uint(b.y));
      }
      if (dst) *reinterpret_cast<uint4*>(dst + 32 * c + 16 * h) = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
}

// 256-column tiles of an fp32 matrix whose row pitch TMA cannot write (the only output).  The four warps of a lane quadrant
// turn 32 rows x 128 columns together, 32 columns each, and every warp writes eight of the rows, cut where 128-byte lines
// begin: of a row's seventeen sectors only the first and the last are written in part.  With 32 columns at a time two of five
// were, and L2 takes those slowly (12000 x 4001 x 500 with its quantize: 99.5 us, 64 this way).
// The warps meet at a named barrier, so after a wait that gave up (ok false) they go through the motions.
template <bool BF16, bool PAIR>
__device__ __forceinline__ void epilogue_rows(const GroupDesc& G, uint32_t tbase, const float* cs, uint32_t stage, uint32_t slot0, uint32_t slot_step, int quad,
                                              int colgrp, int m, int row0, int col0, int lane, uint32_t tempty_bar, bool ok) {
  const OutDesc& o = G.outs[1];
  const int act = G.act;
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    uint32_t v[32];
    if (ok) {
      tmem_ld32_issue(tbase + 32 * (4 * h + colgrp), v);
      tmem_ld_wait();
      if (h == 1) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) { if (PAIR) mbar_arrive_leader(tempty_bar); else mbar_arrive(tempty_bar); }
      }
    }
    asm volatile("bar.sync %0, 128;" ::"r"(1 + quad) : "memory");      // the rows turned last have been read
    if (ok) {
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        uint32_t part[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) part[i] = v[16 * p + i];
        float2 y[8];
        sub_values<BF16>(y, part, cs + 32 * h + 16 * p, act);
#pragma unroll
        for (int j = 0; j < 4; ++j)
          st_shared_v4(stage + lane * 128 + (((4 * p + j) ^ (lane & 7)) << 4), __float_as_uint(y[2 * j].x), __float_as_uint(y[2 * j].y),
                       __float_as_uint(y[2 * j + 1].x), __float_as_uint(y[2 * j + 1].y));
      }
    }
    asm volatile("bar.sync %0, 128;" ::"r"(1 + quad) : "memory");
    const int left = G.n - col0 - 128 * h, ncols = left < 128 ? left : 128;
    if (!ok || ncols <= 0) continue;
    // Two rows at a time: all their reads, then all their stores (a store behind every read waited for the read each time:
    // 83 us for the matrix above)
    constexpr int kBatch = 2;
#pragma unroll 1
    for (int i = 8 * colgrp; i < 8 * colgrp + 8; i += kBatch) {
      uint32_t x[kBatch][5];
      // a lane's words of a row are 32 apart, counted from the line's beginning: one place in each of the four warps' slots,
      // begun in the slot before for lanes whose first word lies in front of the row
      uint32_t* out = reinterpret_cast<uint32_t*>(o.ptr) + (int64_t)(row0 + i) * o.ld + col0 + 128 * h;
#pragma unroll
      for (int b = 0; b < kBatch; ++b) {
        const int c0 = lane - (int)(((uintptr_t)(out + b * o.ld) >> 2) & 31), w = c0 & 31;
        const uint32_t src = slot0 + (i + b) * 128 + (((w >> 2) ^ ((i + b) & 7)) << 4) + (w & 3) * 4 - (c0 < 0 ? slot_step : 0u);
#pragma unroll
        for (int j = 0; j < 5; ++j)
          if (j == 0 ? c0 >= 0 : j < 4 || c0 < 0) asm volatile("ld.shared.b32 %0, [%1];" : "=r"(x[b][j]) : "r"(src + j * slot_step));
      }
#pragma unroll
      for (int b = 0; b < kBatch; ++b) {
        if (row0 + i + b >= m) break;
        const int c0 = lane - (int)(((uintptr_t)(out + b * o.ld) >> 2) & 31);
        uint32_t* at = out + b * o.ld + c0;
#pragma unroll
        for (int j = 0; j < 5; ++j)
          if (c0 + 32 * j >= 0 && c0 + 32 * j < ncols) at[32 * j] = x[b][j];
      }
    }
  }
}

// ---------------------------------------------------------------------------- the kernel

// One launch runs one GEMM record or, in the CHAIN flavour, up to kChainMax records one after the
// other: consecutive layers of a model, each reading what an earlier one wrote.  The tiles of all
// records form one sequence (record after record, group after group, column tile fastest) that the
// CTA pairs deal out round-robin, so a pair that runs out of tiles of one record goes on with the
// next: no pipeline fill and drain, no idle last round and no kernel boundary between layers.
// A tile may start when the row tiles it reads are complete: every finished tile adds one to a
// counter of its (record, row tile, CTA rank) -- a warp of its own does that once the tile's stores
// have completed -- and another warp, ahead of the producer, waits for the counters of the records
// a tile's record names and clears the tile for loading.
// Waits only ever point at earlier tiles of the sequence and the launch is cooperative (all CTAs
// resident), so the first unfinished tile can always proceed.  The records of a chain share tile
// shape, operand type, stage count, staging size, rows and grid.
// FL: what the single-GEMM flavours carry besides the plain matrix product.  Convolutions and shortcut layers have
// instantiations of their own: their code inside the plain kernel slowed its short launches by a tenth to a fifth
// (100352 x 128 x 512: 20.0 -> 24.5 us).
enum : int { FL_PLAIN = 0, FL_CONV = 1, FL_SHORTCUT = 2, FL_SLAB = 3, FL_SLAB64 = 4, FL_ROWS = 5 };
template <bool BF16, bool PAIR, bool GROUPED, bool CHAIN, int FL = FL_PLAIN>
__global__ void __launch_bounds__(FL == FL_CONV || CHAIN ? kGemmThreadsConv : kGemmThreads, 1)
gemm_kernel(const __grid_constant__ LaunchArgs<CHAIN> L) {
  const GemmParams& p = L.rec[0].p;        // what all records of the launch have in common is read here
  const GemmParams* q = &L.rec[0].p;       // the record this thread's role is working on
  const CUtensorMap* mp = L.rec[0].m;      // its pool of tensor maps
  extern __shared__ uint8_t smem_raw[];
  // 1024-byte alignment for the 128B swizzle atoms
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem);           // full[8] empty[8] tfull[2] tempty[2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + 256);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + 260);
  const uint32_t cleared_addr = smem_u32(smem + 264);            // chains: tiles of this CTA whose inputs are complete
  float* cs_all = reinterpret_cast<float*>(smem + kSmemHeader);  // kEpiWarps x 64 rescale factors
  uint8_t* epi_stage = smem + kSmemHeader + kCsBytes;            // kEpiWarps x epi_bytes, 1024-aligned
  uint8_t* stage_base = epi_stage + kEpiWarps * p.epi_bytes;

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  // Pair flavour: the two CTAs of a cluster share one 256-row tile.  Each loads its own 128 rows
  // of A and its own half of the tile's B rows; the first CTA issues the MMAs for both
  // (cta_group::2), each CTA's TMEM receives the accumulators of its 128 rows.  p.tiles_m then
  // counts 256-row tiles.
  const int rank = PAIR ? (int)cluster_ctarank() : 0;
  const int b_rows = PAIR ? (p.bn >> 1) : p.bn;                  // B rows held per stage by this CTA
  constexpr bool kSlab = FL == FL_SLAB || FL == FL_SLAB64;       // stages hold weights only, the input's slabs have a ring of their own
  constexpr int kChunk = FL == FL_SLAB64 ? 64 : 128;             // ... and the slab's channel bytes
  const uint32_t stage_bytes = kSlab ? (uint32_t)(b_rows * kChunk) : (uint32_t)(BM + b_rows) * kStageKBytes;
  const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * kMaxStages;
  const uint32_t tfull0 = empty0 + 8 * kMaxStages, tempty0 = tfull0 + 16;
  // chains: per epilogue warp, the number of its tiles whose stores have completed (counters, not
  // phase barriers: the warp that reads them may fall any number of tiles behind)
  const uint32_t rep0 = smem_u32(smem + 320);
  const int tile0 = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;       // first tile of this CTA (pair)
  const int tile_step = PAIR ? (int)(gridDim.x >> 1) : (int)gridDim.x;
  const int rows_per_tile = PAIR ? 2 * BM : BM;
  // group of a column tile (a single-GEMM launch has only group 0, known at compile time)
  auto group_of = [&](int tn) -> int {
    return GROUPED ? (int)(tn >= q->grp[1].tn_begin) + (int)(tn >= q->grp[2].tn_begin) : 0;
  };
  auto tile_in_group = [&](int tn, int g) -> int { return GROUPED ? tn - q->grp[g].tn_begin : tn; };
  // Tiles are numbered with the row-tile index fastest, in shortcut layers with the column tile fastest: they are bound by
  // what they move, and the column tiles of a row tile then read and write whole rows together (ResNet-50 at batch 128,
  // sixteen such layers: 2397 us per evaluation with the row tile fastest, 2288 this way; plain and convolution launches
  // do not differ).  Each role walks its tiles by adding the
  // stride split into (row tiles, column tiles) once here: a division per tile would sit on the
  // epilogue's and the producer's path.
  constexpr bool kColFast = FL == FL_SHORTCUT;
  int num_tiles, step_tn, step_tm, tm0, tn0;
  auto set_record = [&](int li) {
    q = &L.rec[CHAIN ? li : 0].p;
    mp = L.rec[CHAIN ? li : 0].m;
    num_tiles = q->tiles_m * q->tiles_n;
    if (kColFast) {
      step_tm = tile_step / q->tiles_n; step_tn = tile_step - step_tm * q->tiles_n;
      tn0 = tile0 % q->tiles_n; tm0 = tile0 / q->tiles_n;
      return;
    }
    step_tn = tile_step / q->tiles_m; step_tm = tile_step - step_tn * q->tiles_m;
    tm0 = tile0 % q->tiles_m; tn0 = tile0 / q->tiles_m;
  };
  // after both coordinates have been advanced by their shares of a step
  auto wrap = [&](int& tm_, int& tn_) {
    if (kColFast) { if (tn_ >= q->tiles_n) { tn_ -= q->tiles_n; ++tm_; } }
    else if (tm_ >= q->tiles_m) { tm_ -= q->tiles_m; ++tn_; }
  };
  set_record(0);
  // chains: position in the launch's tile sequence
  struct Cur { int li, first, ntiles; const GemmParams* q; const CUtensorMap* mp; };
  auto cur_seek = [&](Cur& c, int g) {       // g < L.total_tiles
    while (g >= c.first + c.ntiles) {
      c.first += c.ntiles; ++c.li;
      c.q = &L.rec[CHAIN ? c.li : 0].p; c.mp = L.rec[CHAIN ? c.li : 0].m;
      c.ntiles = c.q->tiles_m * c.q->tiles_n;
    }
  };
  Cur cur{0, 0, num_tiles, q, mp};
  // record-local tile index -> group, row tile, column tile (column tiles numbered over all groups)
  auto locate = [&](const GemmParams* qq, int T, int& gi, int& tm, int& tn) {
    gi = (int)(T >= qq->grp[1].tile_first) + (int)(T >= qq->grp[2].tile_first);
    const GroupDesc& G = qq->grp[gi];
    const int Tl = T - G.tile_first;
    tm = Tl / G.gtiles_n;
    tn = G.tn_begin + (Tl - tm * G.gtiles_n);
  };
  const int total_tiles = CHAIN ? L.total_tiles : num_tiles;

  // producer state (thread 0 only): next k-block to load
  // The producer and the MMA issuer share their scheduler with four epilogue warps that almost
  // always have an instruction ready, so every instruction these two threads need per k-block
  // costs them many cycles of waiting for an issue slot: their loops keep all addresses and
  // coordinates in registers and update them incrementally.
  int ld_tile = tile0, ld_kb = 0, ld_s = 0;
  uint32_t ld_ph = 0;
  const int k_elems = BF16 ? kStageKBytes / 2 : kStageKBytes;
  const uint32_t slab0 = smem_u32(stage_base);                   // kSlab: the slabs, then the stages
  const uint32_t stage0 = slab0 + (kSlab ? (uint32_t)(p.slab.count * p.slab.bytes) : 0u);
  const uint32_t sfull0 = smem_u32(smem + kResBarOffset), sempty0 = sfull0 + 8 * kMaxSlabs;
  uint32_t ld_dst = stage0, ld_bar = full0;      // stage address and its full barrier
  int ld_x = 0, ld_ya = 0, ld_yb = 0;            // TMA coordinates of the next k-block
  int ld_tm = tm0, ld_tn = tn0;
  const CUtensorMap* ld_map_a = &mp[q->mi[0][MAP_A]];
  const CUtensorMap* ld_map_b = &mp[q->mi[0][MAP_B]];
  constexpr bool kConv = FL == FL_CONV;
  const bool conv_tma = kConv && p.conv.on >= CONV_TMA128;
  int cv_n = 0, cv_h = 0, cv_w = 0;              // TMA convolutions: corner of the tile's first pixel
  int cv_c = 0, cv_dx = 0, cv_dy = 0;            // channel and tap of the next chunk
  auto set_tile_coords = [&]() {
    const int g = group_of(ld_tn);
    if (GROUPED) { ld_map_a = &mp[q->mi[g][MAP_A]]; ld_map_b = &mp[q->mi[g][MAP_B]]; }
    ld_ya = ld_tm * rows_per_tile + rank * BM;
    ld_yb = tile_in_group(ld_tn, g) * p.bn + rank * b_rows;
    if (conv_tma) {
      const int opix = p.conv.OH * p.conv.OW;
      cv_n = ld_ya / opix;
      const int pix = ld_ya - cv_n * opix, oh = pix / p.conv.OW;
      cv_h = oh * p.conv.stride - p.conv.pad;
      cv_w = (pix - oh * p.conv.OW) * p.conv.stride - p.conv.pad;
      cv_c = 0; cv_dx = 0; cv_dy = 0;
    }
  };
  if (warp == 0) set_tile_coords();
  const bool elected = elect_one();    // the lane of a converged warp that issues TMA / MMA instructions
  const bool conv_on = kConv && p.conv.on == CONV_GATHER;
  // one 128-row column of patches per call; chunks behind the last tap come from behind the last channel, which reads as
  // zeros (the B tile is zero there too, but zero times an infinity would not be)
  auto load_patches = [&]() {
    const int chunk = (p.conv.on == CONV_TMA64 ? 64 : 128) / (BF16 ? 2 : 1);
    const int loads = p.conv.on == CONV_TMA64 ? 2 : 1;
    for (int h = 0; h < loads; ++h) {
      const bool past = cv_dy == p.conv.kh;
      if (elected) {
        const uint32_t dst = ld_dst + h * (BM * 64);
        if (PAIR) tma_load_im2col_pair(dst, ld_map_a, ld_bar, past ? p.conv.C : cv_c, cv_w, cv_h, cv_n, past ? 0 : cv_dx, past ? 0 : cv_dy);
        else tma_load_im2col(dst, ld_map_a, ld_bar, past ? p.conv.C : cv_c, cv_w, cv_h, cv_n, past ? 0 : cv_dx, past ? 0 : cv_dy);
      }
      if (!past) {
        cv_c += chunk;
        if (cv_c >= p.conv.C) { cv_c = 0; if (++cv_dx == p.conv.kw) { cv_dx = 0; ++cv_dy; } }
      }
    }
  };
  // bytes the TMA loads of one CTA put into a stage (the A tile is gathered in convolution launches)
  const uint32_t tma_bytes = conv_on ? (uint32_t)b_rows * kStageKBytes : stage_bytes;
  auto issue_load = [&]() {   // whole warp 0; the stage's empty barrier must already have been passed
    if (elected) {
    if (PAIR) {
      // the first CTA's barrier collects the bytes of both CTAs' loads
      if (rank == 0) mbar_expect_tx(ld_bar, 2 * tma_bytes);
      if (!kConv || !(conv_on || conv_tma)) tma_load_2d_pair(ld_dst, ld_map_a, ld_bar, ld_x, ld_ya);
      tma_load_2d_pair(ld_dst + BM * kStageKBytes, ld_map_b, ld_bar, ld_x, ld_yb);
    } else {
      mbar_expect_tx(ld_bar, tma_bytes);
      if (!kConv || !(conv_on || conv_tma)) tma_load_2d(ld_dst, ld_map_a, ld_bar, ld_x, ld_ya);
      tma_load_2d(ld_dst + BM * kStageKBytes, ld_map_b, ld_bar, ld_x, ld_yb);
    }
    }
    if (kConv && conv_tma) load_patches();
    ld_dst += stage_bytes; ld_bar += 8; ld_x += k_elems;
    if (++ld_s == p.stages) { ld_s = 0; ld_ph ^= 1; ld_dst = stage0; ld_bar = full0; }
    if (++ld_kb == q->k_blocks) {
      ld_kb = 0; ld_x = 0; ld_tile += tile_step;
      ld_tm += step_tm; ld_tn += step_tn;
      wrap(ld_tm, ld_tn);
      set_tile_coords();
    }
  };

  if (threadIdx.x == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(&mp[q->mi[0][MAP_A]]) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&mp[q->mi[0][MAP_B]]) : "memory");
    const uint32_t full_count = 1 + (conv_on ? kGatherWarps * (PAIR ? 2 : 1) : 0);   // the TMA thread, plus one arrival per gather warp
    if (kSlab) {
      for (int s = 0; s < 2 * kMaxStages; ++s) mbar_init(full0 + 8 * s, 1);     // ring, or one per resident k-block
      for (int s = 0; s < 2 * kMaxSlabs; ++s) mbar_init(sfull0 + 8 * s, 1);
    } else
    for (int s = 0; s < p.stages; ++s) { mbar_init(full0 + 8 * s, full_count); mbar_init(empty0 + 8 * s, 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(tfull0 + 8 * a, 1); mbar_init(tempty0 + 8 * a, PAIR ? 2 * kEpiWarps : p.alternate ? kEpiWarps / 2 : kEpiWarps); }
    if (FL == FL_SHORTCUT) for (int a = 0; a < 2 * kEpiWarps; ++a) mbar_init(smem_u32(smem + kResBarOffset) + 8 * a, 1);
    if (CHAIN) for (int a = 0; a < kEpiWarps; ++a) *reinterpret_cast<volatile uint32_t*>(smem + 320 + 4 * a) = 0u;
    *abort_flag = 0;
    *reinterpret_cast<volatile uint32_t*>(smem + 264) = 0u;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (kSlab) {      // behind what the loads write: zeros
    const int quads = (p.slab.bytes - p.slab.tx_bytes) >> 4;
    for (int i = threadIdx.x; i < quads * p.slab.count; i += kGemmThreads)
      st_shared_v4(slab0 + (uint32_t)((i / quads) * p.slab.bytes + p.slab.tx_bytes + (i % quads) * 16), 0u, 0u, 0u, 0u);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    if (PAIR) {   // the same warp of both CTAs allocates for the pair
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kTmemCols) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kTmemCols) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  if (PAIR) {     // both CTAs' barriers exist before either one's loads or arrivals can reach them
    __syncthreads();
    cluster_sync_all();
  }
  // Everything above touches no global memory, so under programmatic dependent launch it
  // overlaps the tail of the previous kernel in the stream; from here on its results are needed.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (p.stamp && threadIdx.x == 32) atomicMin(p.stamp, (unsigned long long)global_timer());
  if (warp == 0) {
    // the ring is empty: fill it before the block-wide barrier so the first tiles are in flight
    if (!CHAIN && !kSlab) for (int i = 0; i < p.stages && ld_tile < num_tiles; ++i) issue_load();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    bool ok = true;
    if (CHAIN) {
      // The dependency warp clears tiles ahead of time (see there); here only a counter in shared
      // memory is read, so no device-scope fence sits between two tiles' loads.
      uint32_t t_ld = 0;
      for (int g = tile0; g < total_tiles && ok; g += tile_step) {
        cur_seek(cur, g);
        const GemmParams* cq = cur.q;
        int gi, tm, tn;
        locate(cq, g - cur.first, gi, tm, tn);
        if (!cleared_wait(cleared_addr, ++t_ld, abort_flag, p.err)) { ok = false; break; }
        const CUtensorMap* ma = &cur.mp[cq->mi[gi][MAP_A]];
        const CUtensorMap* mb = &cur.mp[cq->mi[gi][MAP_B]];
        const int ya = tm * rows_per_tile + rank * BM;
        const int yb = (tn - cq->grp[gi].tn_begin) * p.bn + rank * b_rows;
        int x = 0;
        for (int kb = 0; kb < cq->k_blocks; ++kb) {
          if (!mbar_wait_warp(ld_bar + 8 * kMaxStages, ld_ph ^ 1, abort_flag, p.err)) { ok = false; break; }
          if (elected) {
            if (rank == 0) mbar_expect_tx(ld_bar, 2 * stage_bytes);
            tma_load_2d_pair(ld_dst, ma, ld_bar, x, ya);
            tma_load_2d_pair(ld_dst + BM * kStageKBytes, mb, ld_bar, x, yb);
          }
          ld_dst += stage_bytes; ld_bar += 8; x += k_elems;
          if (++ld_s == p.stages) { ld_s = 0; ld_ph ^= 1; ld_dst = stage0; ld_bar = full0; }
        }
      }
    } else if (kSlab) {
      // Slabs run one ahead of the weights, so that the next chunk's pixels are under way while the ring waits for the
      // tensor core; with resident weights the ring of slabs is all there is to keep full.
      const SlabDesc& sd = p.slab;
      int f_tile = tile0, f_chunk = 0, f_s = 0, f_w = 0, f_h = 0, f_n = 0;
      uint32_t f_ph = 0;
      auto fetch_slab = [&]() -> bool {
        if (f_tile >= num_tiles) return true;
        if (!mbar_wait_warp(sempty0 + 8 * f_s, f_ph ^ 1, abort_flag, p.err)) return false;
        if (f_chunk == 0) {
          const int tm = f_tile % p.tiles_m, mt = PAIR ? 2 * tm + rank : tm;
          const int wh = sd.tiles_w * sd.tiles_h, ng = mt / wh, q2 = mt - ng * wh, th = q2 / sd.tiles_w;
          f_n = ng * sd.imgs;
          f_h = th * sd.rows - p.conv.pad;
          f_w = (q2 - th * sd.tiles_w) * sd.tw - p.conv.pad;
        }
        if (elected) {
          const uint32_t dst = slab0 + (uint32_t)(f_s * sd.bytes), bar = sfull0 + 8 * f_s;
          if (rank == 0) mbar_expect_tx(bar, (uint32_t)((PAIR ? 2 : 1) * sd.tx_bytes));
          if (PAIR) tma_load_4d_pair(dst, ld_map_a, bar, f_chunk * kChunk, f_w, f_h, f_n);
          else tma_load_4d(dst, ld_map_a, bar, f_chunk * kChunk, f_w, f_h, f_n);
        }
        if (++f_s == sd.count) { f_s = 0; f_ph ^= 1; }
        if (++f_chunk == sd.chunks) { f_chunk = 0; f_tile += tile_step; }
        return true;
      };
      ok = fetch_slab();
      if (sd.resident) {
        for (int t = 0; t < 9; ++t, ld_bar += 8, ld_dst += stage_bytes)
          if (elected) {
            mbar_expect_tx(ld_bar, stage_bytes);
            tma_load_2d(ld_dst, ld_map_b, ld_bar, t * p.conv.C, 0);
          }
        while (ok && f_tile < num_tiles) ok = fetch_slab();
      } else {
        for (int tile = tile0; tile < num_tiles && ok; tile += tile_step) {
          const int yb = tile / p.tiles_m * p.bn + rank * b_rows;
          for (int c = 0; c < sd.chunks && ok; ++c) {
            ok = fetch_slab();
            int x = c * kChunk;
            for (int t = 0; t < 9 && ok; ++t, x += p.conv.C) {
              if (!mbar_wait_warp(ld_bar + 8 * kMaxStages, ld_ph ^ 1, abort_flag, p.err)) { ok = false; break; }
              if (elected) {
                if (rank == 0) mbar_expect_tx(ld_bar, (PAIR ? 2 : 1) * stage_bytes);
                if (PAIR) tma_load_2d_pair(ld_dst, ld_map_b, ld_bar, x, yb);
                else tma_load_2d(ld_dst, ld_map_b, ld_bar, x, yb);
              }
              ld_dst += stage_bytes; ld_bar += 8;
              if (++ld_s == p.stages) { ld_s = 0; ld_ph ^= 1; ld_dst = stage0; ld_bar = full0; }
            }
          }
        }
      }
      // as below for the stages: the pair's first CTA still releases this CTA's slabs
      if (PAIR)
        for (int i = 0; i < sd.count && ok; ++i) {
          if (!mbar_wait_warp(sempty0 + 8 * f_s, f_ph ^ 1, abort_flag, p.err)) ok = false;
          if (++f_s == sd.count) { f_s = 0; f_ph ^= 1; }
        }
    } else {
      while (ld_tile < num_tiles) {
        if (!mbar_wait_warp(ld_bar + 8 * kMaxStages, ld_ph ^ 1, abort_flag, p.err)) { ok = false; break; }
        issue_load();
      }
    }
    if (PAIR && ok) {
      // the peer's MMA completions still arrive on this CTA's stage barriers: drain them all
      // before this CTA may exit (a stage never filled passes at once)
      for (int i = 0; i < p.stages && ok; ++i) {
        if (!mbar_wait_warp(empty0 + 8 * ld_s, ld_ph ^ 1, abort_flag, p.err)) ok = false;
        if (++ld_s == p.stages) { ld_s = 0; ld_ph ^= 1; }
      }
    }
    if (!ok) {
      // give copies already in flight a bounded time to land before the CTA exits
      const uint64_t t0 = global_timer();
      while (global_timer() - t0 < 200000ull) {}
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    if (kSlab && rank == 0) {
      // Per channel chunk one slab and one block of weights per tap; a tap moves the A operand's start by whole slab pixels.
      // The swizzle pattern stays where the TMA load put it (it follows the address), so the start may be any row.
      // The taps are written out: an instruction for 64 columns keeps the tensor core for 48 cycles only, and with the taps
      // in loops issuing one took 240 (56 x 56 x 64, 128 images: 69 us, 32 this way).
      const SlabDesc& sd = p.slab;
      constexpr uint32_t kPx = (uint32_t)kChunk >> 4;                  // one slab pixel, in the descriptor's 16-byte units
      constexpr uint32_t kHi = kChunk == 64 ? (uint32_t)(512 >> 4) | (1u << 14) | (4u << 29) : (uint32_t)(1024 >> 4) | (1u << 14) | (2u << 29);
      const uint32_t pitch = (uint32_t)sd.pitch * kPx;
      const uint32_t alo0 = ((slab0 >> 4) & 0x3FFFu) | (1u << 16), a_step = (uint32_t)sd.bytes >> 4;
      const uint32_t blo0 = ((stage0 >> 4) & 0x3FFFu) | (1u << 16), b_step = stage_bytes >> 4;
      uint32_t alo = alo0, sfb = sfull0, sph = 0;
      int ss = 0, t = 0;
      bool ok = true;
      auto mma_tap = [&](uint32_t d_tmem, int tap, uint32_t bl, uint32_t acc) {      // elected lane
        const uint32_t al = alo + (uint32_t)(tap / 3) * pitch + (uint32_t)(tap % 3) * kPx;
#pragma unroll
        for (int k = 0; k < kChunk / kUmmaKBytes; ++k) {
          const uint64_t da = ((uint64_t)kHi << 32) | (uint64_t)(al + 2u * k), db = ((uint64_t)kHi << 32) | (uint64_t)(bl + 2u * k);
          if (PAIR) tc_mma_pair<BF16>(d_tmem, da, db, p.idesc, k == 0 ? acc : 1u);
          else tc_mma<BF16>(d_tmem, da, db, p.idesc, k == 0 ? acc : 1u);
        }
      };
      auto acc_wait = [&](int at) { return mbar_wait_warp(tempty0 + 8 * (at & 1), ((at >> 1) & 1) ^ 1, abort_flag, p.err); };
      auto next_slab = [&]() {
        alo += a_step; sfb += 8;
        if (++ss == sd.count) { ss = 0; sph ^= 1; alo = alo0; sfb = sfull0; }
      };
      if (!PAIR && sd.resident) {
        // one chunk, all weights in shared memory: no wait and no branch between a tile's taps
        for (int tile = tile0; tile < num_tiles && ok; tile += tile_step, ++t) {
          if (!acc_wait(t) || !mbar_wait_warp(sfb, sph, abort_flag, p.err)) { ok = false; break; }
          tc_fence_after();
          const uint32_t d_tmem = tmem_base + (uint32_t)(t & 1) * kAccCols;
          if (t == 0) {                                    // the weights arrive tap by tap
#pragma unroll
            for (int tap = 0; tap < 9; ++tap) {
              if (ok && !mbar_wait_warp(full0 + 8 * tap, 0, abort_flag, p.err)) ok = false;
              tc_fence_after();
              if (ok && elected) mma_tap(d_tmem, tap, blo0 + (uint32_t)tap * b_step, tap > 0);
            }
            if (!ok) break;
          } else if (elected) {
#pragma unroll
            for (int tap = 0; tap < 9; ++tap) mma_tap(d_tmem, tap, blo0 + (uint32_t)tap * b_step, tap > 0);
          }
          if (elected) { tc_commit(sfb + 8 * kMaxSlabs); tc_commit(tfull0 + 8 * (t & 1)); }
          next_slab();
        }
      } else {
        uint32_t blo = blo0, fb = full0, ph = 0;
        int s = 0;
        for (int tile = tile0; tile < num_tiles && ok; tile += tile_step, ++t) {
          if (!acc_wait(t)) { ok = false; break; }
          tc_fence_after();
          const uint32_t d_tmem = tmem_base + (uint32_t)(t & 1) * kAccCols;
          for (int c = 0; c < sd.chunks && ok; ++c) {
            if (!mbar_wait_warp(sfb, sph, abort_flag, p.err)) { ok = false; break; }
            tc_fence_after();
#pragma unroll
            for (int tap = 0; tap < 9; ++tap) {
              if (!ok || !mbar_wait_warp(fb, ph, abort_flag, p.err)) { ok = false; break; }
              tc_fence_after();
              if (elected) {
                mma_tap(d_tmem, tap, blo, c + tap > 0);
                if (PAIR) tc_commit_pair(fb + 8 * kMaxStages); else tc_commit(fb + 8 * kMaxStages);
              }
              blo += b_step; fb += 8;
              if (++s == p.stages) { s = 0; ph ^= 1; blo = blo0; fb = full0; }
            }
            if (ok && elected) { if (PAIR) tc_commit_pair(sfb + 8 * kMaxSlabs); else tc_commit(sfb + 8 * kMaxSlabs); }
            next_slab();
          }
          if (ok && elected) { if (PAIR) tc_commit_pair(tfull0 + 8 * (t & 1)); else tc_commit(tfull0 + 8 * (t & 1)); }
        }
      }
    } else if (!kSlab && rank == 0) {
      // Descriptor low words (start address field, 16-byte units) of the four K steps of the
      // current stage's A and B tiles; the high word is the same for all.
      constexpr uint32_t kDescHi = (uint32_t)(1024 >> 4) | (1u << 14) | (2u << 29);
      const uint32_t lo0 = ((stage0 >> 4) & 0x3FFFu) | (1u << 16);
      const uint32_t lo_step = stage_bytes >> 4;
      constexpr uint32_t kBOff = (uint32_t)(BM * kStageKBytes) >> 4;
      uint32_t lo = lo0, fb = full0;
      int s = 0; uint32_t ph = 0;
      bool ok = true;
      int t = 0;
      // A tiles of two 64-byte halves: 64B swizzle (layout type 4), 8-row groups 512 bytes apart, the
      // second half BM * 64 bytes behind the first
      const bool halves = kConv && p.conv.on == CONV_TMA64;
      const uint32_t a_hi = halves ? (uint32_t)(512 >> 4) | (1u << 14) | (4u << 29) : kDescHi;
      const uint32_t a_half = halves ? (uint32_t)((BM * 64) >> 4) - 4u : 0u;
      auto mma4 = [&](uint32_t d_tmem, uint32_t first_acc) {
        if (!elected) return;
#pragma unroll
        for (int k4 = 0; k4 < kStageKBytes / kUmmaKBytes; ++k4) {
          // advancing the start address by 32 bytes (2 units) steps along K inside the swizzle atom
          const uint64_t da = ((uint64_t)(kConv ? a_hi : kDescHi) << 32) | (uint64_t)(lo + 2u * k4 + (kConv && k4 >= 2 ? a_half : 0u));
          const uint64_t db = ((uint64_t)kDescHi << 32) | (uint64_t)(lo + kBOff + 2u * k4);
          const uint32_t acc = k4 == 0 ? first_acc : 1u;
          if (PAIR) tc_mma_pair<BF16>(d_tmem, da, db, p.idesc, acc);
          else tc_mma<BF16>(d_tmem, da, db, p.idesc, acc);
        }
      };
      for (int tile = tile0; tile < total_tiles && ok; tile += tile_step, ++t) {
        if (CHAIN) { cur_seek(cur, tile); q = cur.q; }
        const int a = t & 1;
        if (!mbar_wait_warp(tempty0 + 8 * a, ((t >> 1) & 1) ^ 1, abort_flag, p.err)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)a * kAccCols;
        for (int kb = 0; kb < q->k_blocks; ++kb) {
          if (!mbar_wait_warp(fb, ph, abort_flag, p.err)) { ok = false; break; }
          tc_fence_after();
          mma4(d_tmem, kb != 0);
          // stage reusable once these MMAs have read it
          if (elected) { if (PAIR) tc_commit_pair(fb + 8 * kMaxStages); else tc_commit(fb + 8 * kMaxStages); }
          lo += lo_step; fb += 8;
          if (++s == p.stages) { s = 0; ph ^= 1; lo = lo0; fb = full0; }
        }
        if (ok && elected) { if (PAIR) tc_commit_pair(tfull0 + 8 * a); else tc_commit(tfull0 + 8 * a); }   // accumulator complete
      }
    }
  } else if (CHAIN && warp >= 2 + kEpiWarps) {
    // ------------------------------------------------------------------ signal warp (chains)
    // For each of this CTA's tiles in order: once all epilogue warps have seen their stores of
    // the tile complete (the bulk-group wait makes the TMA writes visible to the waiting thread,
    // whose barrier arrival this warp has acquired), publish it with a release at device scope:
    // one is added to the counter of its record, row tile and CTA rank.
    if (warp == 2 + kEpiWarps) {
      int t = 0;
      for (int g = tile0; g < total_tiles; g += tile_step, ++t) {
        cur_seek(cur, g);
        if (!reported_wait(rep0, (uint32_t)t + 1u, lane, abort_flag, p.err)) break;
        int gi, tm, tn;
        locate(cur.q, g - cur.first, gi, tm, tn);
        if (elected && cur.q->grp[gi].signal) {
          asm volatile("red.release.gpu.global.add.u32 [%0], 1;"
                       ::"l"(L.flags + (size_t)cur.li * L.flag_stride + 2 * tm + rank) : "memory");
        }
      }
    } else if (warp == 3 + kEpiWarps) {
      // ---------------------------------------------------------------- dependency warp (chains)
      // Walks this CTA's tiles ahead of the producer.  For each, lane d waits (acquire at device
      // scope, bounded) until the counter of dependency d says the rows the tile reads are
      // complete; then one lane orders the asynchronous proxy after that and publishes the tile
      // count in shared memory, which is all the producer looks at.  The two device-scope fences
      // cost about a microsecond each under load, and here they delay nobody.
      uint32_t t_clear = 0;
      for (int g = tile0; g < total_tiles; g += tile_step) {
        cur_seek(cur, g);
        int gi, tm, tn;
        locate(cur.q, g - cur.first, gi, tm, tn);
        const int dep = lane < kMaxDeps ? cur.q->deps[lane] : -1;
        bool failed = false;
        if (dep >= 0)
          failed = !flag_wait(L.flags + (size_t)dep * L.flag_stride + 2 * tm + rank, (uint32_t)L.rec[dep].p.need, abort_flag, p.err);
        const bool had = __any_sync(0xffffffffu, dep >= 0);
        if (__any_sync(0xffffffffu, failed)) break;
        ++t_clear;
        __syncwarp();
        if (elected) {
          if (had) asm volatile("fence.proxy.async;" ::: "memory");
          asm volatile("st.release.cta.shared::cta.u32 [%0], %1;" ::"r"(cleared_addr), "r"(t_clear) : "memory");
        }
      }
    }
  } else if (kConv && warp >= 2 + kEpiWarps) {
    // ------------------------------------------------------------------ gather warps (convolutions)
    // Each lane owns two rows of the CTA's 128-row A tile.  Per k-block it copies the rows' eight
    // 16-byte chunks from the NHWC source (cp.async with zero fill outside the image, beyond the
    // reduction length and past the last row) to where a 128B-swizzled TMA box would have put them.
    // kGatherDepth k-blocks stay in flight; when the oldest has landed the lane makes its writes
    // visible to the tensor core (fence.proxy.async) and one lane per warp arrives on the stage's
    // full barrier (the pair's first CTA's).
    const ConvDesc& cv = p.conv;
    const int gw = warp - (2 + kEpiWarps);
    const int epc = 16 / cv.esz;                       // elements per 16-byte chunk
    const int opix = cv.OH * cv.OW;
    int s = 0, as = 0, inflight = 0;
    uint32_t ph = 0;
    int tm = tm0, tn = tn0;
    bool ok = true;
    auto landed = [&]() {                              // the oldest group in flight has landed
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) { if (PAIR) mbar_arrive_leader(full0 + 8 * as); else mbar_arrive(full0 + 8 * as); }
      if (++as == p.stages) as = 0;
      --inflight;
    };
    for (int tile = tile0; tile < num_tiles && ok; tile += tile_step) {
      int ih0[2], iw0[2];
      const uint8_t* img[2];
      bool rv[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int64_t pm = (int64_t)tm * rows_per_tile + rank * BM + gw * 64 + i * 32 + lane;
        rv[i] = pm < p.m;
        const int q = rv[i] ? (int)pm : 0;
        const int b = q / opix, pix = q - b * opix;
        const int oh = pix / cv.OW, ow = pix - oh * cv.OW;
        ih0[i] = oh * cv.stride - cv.pad;
        iw0[i] = ow * cv.stride - cv.pad;
        img[i] = cv.src + (int64_t)b * cv.img_bytes;
      }
      int dy = 0, dx = 0, c = 0, ke = 0;
      for (int kb = 0; kb < p.k_blocks && ok; ++kb) {
        if (!mbar_wait_warp(empty0 + 8 * s, ph ^ 1, abort_flag, p.err)) { ok = false; break; }
        const uint32_t a_dst = stage0 + (uint32_t)s * stage_bytes + (uint32_t)(gw * 64 + lane) * 128;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const bool kin = ke < cv.K;
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int ih = ih0[i] + dy, iw = iw0[i] + dx;
            const bool valid = rv[i] && kin && (unsigned)ih < (unsigned)cv.H && (unsigned)iw < (unsigned)cv.W;
            const uint8_t* src = valid ? img[i] + ((int64_t)(ih * cv.W + iw) * cv.C + c) * cv.esz : cv.src;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                         ::"r"(a_dst + i * 32 * 128 + ((j ^ (lane & 7)) << 4)), "l"(src), "r"(valid ? 16 : 0) : "memory");
          }
          ke += epc; c += epc;
          if (c >= cv.C) { c = 0; if (++dx == cv.kw) { dx = 0; ++dy; } }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        if (++s == p.stages) { s = 0; ph ^= 1; }
        if (++inflight > kGatherDepth) {
          asm volatile("cp.async.wait_group %0;" ::"n"(kGatherDepth) : "memory");
          landed();
        }
      }
      tm += step_tm; tn += step_tn;
      wrap(tm, tn);
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    while (inflight > 0) landed();
  } else {
    // ------------------------------------------------------------------ epilogue
    constexpr bool kRowsOut = FL == FL_ROWS;
    const int ew = warp - 2;
    const int quad = warp & 3;                 // TMEM lanes 32*quad .. 32*quad+31 belong to this warp
    const bool alternate = !PAIR && !GROUPED && !CHAIN && FL != FL_SHORTCUT && p.alternate;
    const int colgrp = alternate ? (ew >> 2) & 1 : ew >> 2;    // four warp sets share the tile's columns (alternate: two, on every other tile)
    const int chunks = p.bn >> 5;
    const int cpg = chunks >= 4 ? (chunks >> 2) : 1;
    const int c_begin = colgrp * cpg;
    const int c_end = c_begin < chunks ? c_begin + cpg : c_begin;
    const uint32_t stage = smem_u32(epi_stage + ew * p.epi_bytes);
    float* cs_tab = cs_all + ew * 64;
    uint32_t cursor = 0;
    bool prev_fast = false;
    bool ok = true;
    // this warp's walk through the CTA's tiles: all of them, or every other one
    int t = 0, tile = tile0, tm = tm0, tn = tn0;
    int e_step = tile_step, e_tm = step_tm, e_tn = step_tn;
    if (alternate) {
      if (ew >> 3) {
        t = 1; tile += tile_step; tm += step_tm; tn += step_tn;
        wrap(tm, tn);
      }
      e_step = 2 * tile_step; e_tm = 2 * step_tm; e_tn = 2 * step_tn;
      wrap(e_tm, e_tn);
    }
    // Weight scales of this warp's chunks, one column per lane and chunk.  They are fetched one
    // tile ahead: when the epilogue is the longer phase the accumulator is already waiting at
    // the top of the loop, and a load issued there would put its whole latency on the tile.
    auto load_scales = [&](const GemmParams* qq, bool valid, int tile_tn, float (&w)[2]) {
      w[0] = 0.f; w[1] = 0.f;
      if (BF16 || !valid) return;
      const int gi = GROUPED ? (int)(tile_tn >= qq->grp[1].tn_begin) + (int)(tile_tn >= qq->grp[2].tn_begin) : 0;
      const GroupDesc& G = qq->grp[gi];
      if (!G.need_y) return;
      const int cb = (GROUPED ? tile_tn - G.tn_begin : tile_tn) * p.bn + (kRowsOut ? colgrp : c_begin) * 32;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int col = cb + j * (kRowsOut ? 128 : 32) + lane;
        if (c_begin + j < c_end && col < G.n) w[j] = __ldg(G.scale_w + col);
      }
    };
    float sw_next[2];
    // shortcut blocks: brought in one tile ahead, into the two blocks in turn
    const bool shortcut = FL == FL_SHORTCUT && c_begin < c_end;
    const uint32_t res_bar0 = smem_u32(smem + kResBarOffset) + 16 * ew;
    auto fetch_shortcut = [&](int which, int ftm, int ftn) {      // lane 0
      const uint32_t bar = res_bar0 + 8 * which;
      mbar_expect_tx(bar, 4096);
      tma_load_2d(stage + which * 4096, &mp[q->mi[0][MAP_OUT]], bar, ftn * p.bn + c_begin * 32, ftm * BM + quad * 32);
    };
    if (shortcut && lane == 0 && tile0 < num_tiles) fetch_shortcut(0, tm0, tn0);
    // slabs: where this lane's tile row lies among the tile's images, rows and columns (pix_ok: an output pixel at all)
    int pix_i = 0, pix_h = 0, pix_w = 0;
    bool pix_ok = false;
    if (kSlab) {
      const int r = quad * 32 + lane;
      pix_i = r / p.slab.img_pitch;
      pix_h = (r - pix_i * p.slab.img_pitch) / p.slab.pitch;
      pix_w = r - pix_i * p.slab.img_pitch - pix_h * p.slab.pitch;
      pix_ok = pix_i < p.slab.imgs && pix_h < p.slab.rows && pix_w < p.slab.tw;
    }
    if (CHAIN) {
      if (tile0 < total_tiles) {
        cur_seek(cur, tile0);
        int gi0, tm_0, tn_0;
        locate(cur.q, tile0 - cur.first, gi0, tm_0, tn_0);
        load_scales(cur.q, true, tn_0, sw_next);
      }
    } else {
      load_scales(q, tile < num_tiles, tn, sw_next);
    }
    for (; tile < total_tiles && (ok || kRowsOut); tile += e_step, t += alternate ? 2 : 1) {
      if (CHAIN) {     // record of this tile, column tile fastest inside it
        cur_seek(cur, tile); q = cur.q; mp = cur.mp;
        int gi_;
        locate(q, tile - cur.first, gi_, tm, tn);
      }
      const int a = t & 1, a_ph = (t >> 1) & 1;
      const int row0 = tm * rows_per_tile + rank * BM + quad * 32;
      const int g = group_of(tn);
      const GroupDesc& G = q->grp[g];
      const int col_base = tile_in_group(tn, g) * p.bn + c_begin * 32;
      const float cs[2] = {__fmul_rn(G.scale_x, sw_next[0]), __fmul_rn(G.scale_x, sw_next[1])};
      int tm_next = tm + e_tm, tn_next = tn + e_tn;
      if (CHAIN) {
        const int nt = tile + tile_step;
        Cur c2 = cur;
        if (nt < total_tiles) cur_seek(c2, nt);
        int gi2 = 0, tm2 = 0, tn2 = 0;
        if (nt < total_tiles) locate(c2.q, nt - c2.first, gi2, tm2, tn2);
        load_scales(c2.q, nt < total_tiles, tn2, sw_next);
      } else {
        wrap(tm_next, tn_next);
        load_scales(q, tile + e_step < num_tiles, tn_next, sw_next);
      }
      // Chains: the previous tile is reported once its stores have completed.  When this tile's
      // accumulator is already there the check is left to the body (after its first piece, when
      // the old stores have landed); when it is not, this tile may itself be waiting for
      // rows other CTAs produce, and they for the report, so the report goes out now.
      uint32_t rep_addr = (CHAIN && t > 0) ? rep0 + 4 * ew : 0u;
      const bool fast_inside = G.mode != EPI_GENERAL && !(row0 >= q->m || col_base >= G.n);
      if (rep_addr && !(fast_inside && __all_sync(0xffffffffu, mbar_try_wait(tfull0 + 8 * a, a_ph)))) {
        if (lane == 0) {
          asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
          asm volatile("st.release.cta.shared::cta.u32 [%0], %1;" ::"r"(rep_addr), "r"((uint32_t)t) : "memory");
        }
        __syncwarp();
        rep_addr = 0;
      }
      if (shortcut) {       // the previous tile's stores have read their block: the next tile's shortcut may come in there
        if (lane == 0) {
          asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
          if (tile + tile_step < num_tiles) fetch_shortcut((t & 1) ^ 1, tm_next, tn_next);
        }
        __syncwarp();
      }
      uint8_t* slab_dst = nullptr;     // slabs: this lane's output pixel
      if (kSlab) {
        const SlabDesc& sd = p.slab;
        const int mt = PAIR ? 2 * tm + rank : tm;
        const int wh = sd.tiles_w * sd.tiles_h, ng = mt / wh, q2 = mt - ng * wh, th = q2 / sd.tiles_w;
        const int img = ng * sd.imgs + pix_i, oh = th * sd.rows + pix_h, ow = (q2 - th * sd.tiles_w) * sd.tw + pix_w;
        if (pix_ok && img < sd.images && oh < p.conv.OH && ow < p.conv.OW)
          slab_dst = reinterpret_cast<uint8_t*>(G.outs[2].ptr) + (((int64_t)img * p.conv.OH + oh) * p.conv.OW + ow) * G.outs[2].ld + col_base;
        cs_tab[lane] = cs[0];
        cs_tab[32 + lane] = cs[1];
        __syncwarp();
      }
      if (!mbar_wait(tfull0 + 8 * a, a_ph, abort_flag, p.err)) { ok = false; if (!kRowsOut) break; }
      tc_fence_after();
      const uint32_t tbase = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(a * kAccCols + c_begin * 32);
      const int nch = c_end - c_begin;           // 0, 1 or 2
      const int64_t row = (int64_t)row0 + lane;
      const uint32_t tempty_bar = tempty0 + 8 * a;
      if (kRowsOut) {
        ok = __all_sync(0xffffffffu, ok);
        cs_tab[lane] = cs[0];
        cs_tab[32 + lane] = cs[1];
        __syncwarp();
        if (row0 < q->m)
          epilogue_rows<BF16, PAIR>(G, tbase - (uint32_t)(c_begin * 32), cs_tab, stage, smem_u32(epi_stage + (ew & 3) * p.epi_bytes), (uint32_t)(4 * p.epi_bytes), quad,
                                    colgrp, q->m, row0, tn * p.bn, lane, tempty_bar, ok);
        else if (ok) {
          __syncwarp();
          if (lane == 0) { if (PAIR) mbar_arrive_leader(tempty_bar); else mbar_arrive(tempty_bar); }
        }
        __syncwarp();
      } else if (kSlab) {
        if (nch == 0 || col_base >= G.n) {
          __syncwarp();
          if (lane == 0) { if (PAIR) mbar_arrive_leader(tempty_bar); else mbar_arrive(tempty_bar); }
        } else {
          const int left = (G.n - col_base) >> 5;         // whole chunks (n is a multiple of 32)
          epilogue_slab<PAIR>(G, tbase, cs_tab, nch < left ? nch : left, slab_dst, lane, tempty_bar);
          __syncwarp();
        }
      } else if (FL == FL_SHORTCUT) {
        if (nch == 0) {
          __syncwarp();
          if (lane == 0) mbar_arrive(tempty_bar);
        } else {
          cs_tab[lane] = cs[0];
          __syncwarp();
          epilogue_shortcut(G, mp, q->mi[0], tbase, cs_tab, stage + (t & 1) * 4096, stage + 2 * 4096, row0, col_base, lane, tempty_bar,
                            res_bar0 + 8 * (t & 1), (uint32_t)(t >> 1) & 1u, row0 < q->m && col_base < G.n, abort_flag, p.err, ok);
        }
      } else if (!PAIR && !GROUPED && !CHAIN && G.mode == EPI_CODES32) {
        if (nch == 0) {
          __syncwarp();
          if (lane == 0) mbar_arrive(tempty_bar);
        } else {
          if (!BF16) {
            cs_tab[lane] = cs[0];
            __syncwarp();
          }
          epilogue_codes32<BF16>(G, &mp[q->mi[0][MAP_OUT + 2]], tbase, cs_tab, stage, row0, col_base, row0 < q->m && col_base < G.n, lane, tempty_bar);
        }
      } else if (!BF16 && FL == FL_PLAIN && !CHAIN && (!PAIR || GROUPED) && G.mode == EPI_Y32) {
        if (nch == 0) {
          __syncwarp();
          if (lane == 0) { if (PAIR) mbar_arrive_leader(tempty_bar); else mbar_arrive(tempty_bar); }
        } else {
          cs_tab[lane] = cs[0];
          __syncwarp();
          epilogue_y32<PAIR>(G, &mp[q->mi[g][MAP_FAST]], tbase, cs_tab, stage, row0, col_base, row0 < q->m && col_base < G.n, lane, tempty_bar);
        }
        prev_fast = true;
      } else if (G.mode != EPI_GENERAL) {
        // fast bodies: 256-column tiles, so this warp owns 64 columns starting at col_base
        if (!fast_inside) {
          __syncwarp();
          if (lane == 0) { if (PAIR) mbar_arrive_leader(tempty_bar); else mbar_arrive(tempty_bar); }
        } else {
          if (!BF16) {   // rescale factors of the 64 columns, read back by every lane
            cs_tab[lane] = cs[0];
            cs_tab[32 + lane] = cs[1];
            __syncwarp();
          }
          if (G.mode == EPI_CODES1)
            epilogue_tile_fast<BF16, PAIR, EPI_CODES1>(G, &mp[q->mi[g][MAP_FAST]], tbase, cs_tab, stage, row0, col_base, lane, tempty_bar, rep_addr, (uint32_t)t);
          else if (G.mode == EPI_BF16)
            epilogue_tile_fast<BF16, PAIR, EPI_BF16>(G, &mp[q->mi[g][MAP_FAST]], tbase, cs_tab, stage, row0, col_base, lane, tempty_bar, rep_addr, (uint32_t)t);
          else
            epilogue_tile_fast<BF16, PAIR, EPI_Y>(G, &mp[q->mi[g][MAP_FAST]], tbase, cs_tab, stage, row0, col_base, lane, tempty_bar, rep_addr, (uint32_t)t);
        }
        prev_fast = true;
      } else {
        if (prev_fast) {    // a fast body's last store reads the whole staging buffer: let it finish
          if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
          __syncwarp();
          prev_fast = false;
        }
        uint32_t v[32];
        // one copy of the chunk code, looped: keeps the instruction footprint small
#pragma unroll 1
        for (int c = 0; c < nch; ++c) {
          tmem_ld32_issue(tbase + 32 * c, v);
          tmem_ld_wait();
          if (c == nch - 1) {   // the accumulator buffer is free again once this warp's columns sit in registers
            tc_fence_before();
            __syncwarp();
            if (lane == 0) { if (PAIR) mbar_arrive_leader(tempty_bar); else mbar_arrive(tempty_bar); }
          }
          const float csl = c ? cs[1] : cs[0];
          epilogue_chunk<BF16, CHAIN>(G, mp, q->mi[g], q->m, (uint32_t)p.epi_bytes, v, csl, row, row0, col_base + 32 * c, stage, cursor, lane);
        }
        if (nch == 0) {
          __syncwarp();
          if (lane == 0) { if (PAIR) mbar_arrive_leader(tempty_bar); else mbar_arrive(tempty_bar); }
        }
      }
      if (!CHAIN) { tm = tm_next; tn = tn_next; }
    }
    if (CHAIN && t > 0 && ok) {       // the last tile: report it as soon as its stores have completed
      if (lane == 0) {
        asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        asm volatile("st.release.cta.shared::cta.u32 [%0], %1;" ::"r"(rep0 + 4 * ew), "r"((uint32_t)t) : "memory");
      }
    }
    // all TMA stores of this warp must have completed before the CTA's shared memory goes away
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  }

  tc_fence_before();
  __syncthreads();
  if (p.stamp && threadIdx.x == 32) atomicMax(p.stamp + 1, (unsigned long long)global_timer());
  if (PAIR) cluster_sync_all();     // the peer no longer signals this CTA's barriers nor uses its TMEM
  if (warp == 1) {
    tc_fence_after();
    if (PAIR) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
    else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
  }
}

// ---------------------------------------------------------------------------- host side

// Host state of the chain being collected (one per context).
struct Span { const uint8_t* lo; const uint8_t* hi; };      // byte range [lo, hi) of a matrix
struct ChainRecInfo { Span in[2 * kMaxGroups]; int n_in; Span out[kNumOuts * kMaxGroups]; int out_grp[kNumOuts * kMaxGroups]; int n_out; };
constexpr size_t kFlagRingBytes = 8u << 20;
constexpr int kChainMaxTilesM = 2048;
struct ChainState {
  LaunchArgs<true> args;          // args.n records collected so far
  // the first record once more, set up as a launch of its own: a chain that ends with one record
  // goes out that way (the cooperative launch only pays when tiles of several GEMMs can overlap)
  LaunchArgs<false> solo;
  int solo_grid = 0, solo_grouped = 0;
  size_t solo_smem = 0;
  ChainRecInfo info[kChainMax];
  double ops = 0.0;
  unsigned* ring = nullptr;       // device counters, handed out front to back and cleared when used up
  unsigned* zero = nullptr;       // a device word that stays zero (self-test of the bounded waits)
  size_t ring_used = 0;           // bytes
  bool open = false;              // a forward pass is running: eligible launches may be deferred
  bool bf16 = false;
  int grid = 0;
  int64_t m = 0;
  size_t smem = 0;
  cudaStream_t st = nullptr;
  const void* ready[32];          // kernels whose shared-memory limit this context has raised (make_ready)
  int n_ready = 0;
  ChainState() { memset(&args, 0, sizeof(args)); memset(&solo, 0, sizeof(solo)); }
};

// Raises a kernel's shared-memory limit when a context first launches it, which also loads the kernel.  With all 22 flavours
// loaded when a context is made, the first one of a process took 12.0 ms, 6.4 this way; with a block's noise table (8.9 ms in
// place of 4.7), calibration and evaluation behind it 23.1, 21.8 this way.
cudaError_t make_ready(ChainState* cs, const void* kern) {
  for (int i = 0; i < cs->n_ready; ++i) if (cs->ready[i] == kern) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
  if (e == cudaSuccess && cs->n_ready < 32) cs->ready[cs->n_ready++] = kern;
  return e;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn g_encode = nullptr;
typedef CUresult (*EncodeIm2colFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const int*,
                                   const int*, cuuint32_t, cuuint32_t, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeIm2colFn g_encode_im2col = nullptr;

// A two-dimensional tiled tensor map.  Encoding one costs a driver call of a microsecond or two and
// an evaluation needs a couple of hundred, always the same ones (a map depends only on address,
// shape, pitch, box, type and swizzle), so encoded maps are kept in a process-wide table.
struct MapKey {
  const void* ptr; uint64_t d0, d1, pitch; uint32_t b0, b1, dt, swz, promo;
  bool operator==(const MapKey& o) const {
    return ptr == o.ptr && d0 == o.d0 && d1 == o.d1 && pitch == o.pitch && b0 == o.b0 && b1 == o.b1 && dt == o.dt &&
           swz == o.swz && promo == o.promo;
  }
};
struct MapKeyHash {
  size_t operator()(const MapKey& k) const {
    uint64_t h = (uint64_t)(uintptr_t)k.ptr * 0x9E3779B97F4A7C15ull;
    auto mix = [&](uint64_t v) { h ^= v + 0x9E3779B97F4A7C15ull + (h << 6) + (h >> 2); };
    mix(k.d0); mix(k.d1); mix(k.pitch); mix(((uint64_t)k.b0 << 32) | k.b1); mix(((uint64_t)k.dt << 40) | ((uint64_t)k.swz << 20) | k.promo);
    return (size_t)h;
  }
};
std::mutex g_map_mutex;
std::unordered_map<MapKey, CUtensorMap, MapKeyHash> g_map_cache;
constexpr size_t kMapCacheMax = 16384;

bool encode_2d(CUtensorMap* map, CUtensorMapDataType dt, const void* ptr, uint64_t d0, uint64_t d1, uint64_t pitch_bytes,
               uint32_t b0, uint32_t b1, CUtensorMapSwizzle swz, CUtensorMapL2promotion promo) {
  const MapKey key{ptr, d0, d1, pitch_bytes, b0, b1, (uint32_t)dt, (uint32_t)swz, (uint32_t)promo};
  {
    std::lock_guard<std::mutex> lock(g_map_mutex);
    auto it = g_map_cache.find(key);
    if (it != g_map_cache.end()) { *map = it->second; return true; }
  }
  cuuint64_t dims[2] = {d0, d1};
  cuuint64_t strides[1] = {pitch_bytes};
  cuuint32_t box[2] = {b0, b1};
  cuuint32_t estr[2] = {1, 1};
  const CUresult r = g_encode(map, dt, 2, const_cast<void*>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swz, promo,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return false;
  std::lock_guard<std::mutex> lock(g_map_mutex);
  if (g_map_cache.size() >= kMapCacheMax) g_map_cache.clear();
  g_map_cache.emplace(key, *map);
  return true;
}

// Tensor map of a convolution's NHWC code tensor for im2col loads of `chunk_bytes` of channels and 128 output
// pixels (kept in the same table as the tiled ones).  False: the driver does not take this geometry.
bool make_im2col_map(CUtensorMap* map, const GemmArgs& g, int64_t images, int chunk_bytes) {
  const int esz = g.is_bf16 ? 2 : 1;
  const CUtensorMapDataType dt = g.is_bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8;
  const CUtensorMapSwizzle swz = chunk_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B;
  const int lower = -g.conv_pad, upper_w = g.conv_pad - (g.conv_kw - 1), upper_h = g.conv_pad - (g.conv_kh - 1);
  if (!g_encode_im2col || g.conv_kh != g.conv_kw || lower < -128 || upper_w < -128 || upper_h < -128 || g.conv_pad > 127 || g.conv_stride > 8 || g.conv_kw > 128 ||
      g.conv_kh > 128 || images > 0x7fffffff || g.conv_h >= 0x10000 || g.conv_w >= 0x10000)
    return false;
  const MapKey key{g.a, (uint64_t)g.conv_c | ((uint64_t)g.conv_w << 32), (uint64_t)g.conv_h | ((uint64_t)images << 32),
                   (uint64_t)g.conv_kh | ((uint64_t)g.conv_kw << 16) | ((uint64_t)g.conv_stride << 32) | ((uint64_t)g.conv_pad << 48),
                   (uint32_t)chunk_bytes, (uint32_t)BM, (uint32_t)dt, 0x100u | (uint32_t)swz, 0u};
  {
    std::lock_guard<std::mutex> lock(g_map_mutex);
    auto it = g_map_cache.find(key);
    if (it != g_map_cache.end()) { *map = it->second; return true; }
  }
  cuuint64_t dims[4] = {(cuuint64_t)g.conv_c, (cuuint64_t)g.conv_w, (cuuint64_t)g.conv_h, (cuuint64_t)images};
  const cuuint64_t px = (cuuint64_t)g.conv_c * esz;
  cuuint64_t strides[3] = {px, px * g.conv_w, px * g.conv_w * g.conv_h};
  int lo[2] = {lower, lower}, up[2] = {upper_w, upper_h};
  cuuint32_t estr[4] = {1, (cuuint32_t)g.conv_stride, (cuuint32_t)g.conv_stride, 1};
  const CUresult r = g_encode_im2col(map, dt, 4, const_cast<void*>(g.a), dims, strides, lo, up, (cuuint32_t)(chunk_bytes / esz), (cuuint32_t)BM,
                                     estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return false;
  std::lock_guard<std::mutex> lock(g_map_mutex);
  if (g_map_cache.size() >= kMapCacheMax) g_map_cache.clear();
  g_map_cache.emplace(key, *map);
  return true;
}

// How a stride-1 convolution is cut into slab tiles: the cut with the fewest tiles, of those the one that loads least.
// False: some limit of the load (256 pixels or rows per box dimension) is in the way of every cut.
bool slab_plan(const GemmArgs& g, int64_t images, int OH, int OW, SlabDesc* best) {
  int64_t best_tiles = 0, best_px = 0;
  for (int tw = 1; tw <= OW && tw <= BM; ++tw) {
    SlabDesc d{};
    d.tw = tw;
    d.pitch = tw + 2 - (tw < OW ? 0 : g.conv_pad < 2 ? g.conv_pad : 2);
    d.rows = (BM - tw) / d.pitch + 1;
    if (d.rows > OH) d.rows = OH;
    d.tiles_w = (OW + tw - 1) / tw;
    d.tiles_h = (OH + d.rows - 1) / d.rows;
    d.img_pitch = (d.rows + 2) * d.pitch;
    d.imgs = 1;
    if (tw == OW && d.rows == OH) d.imgs = (BM - ((OH - 1) * d.pitch + tw)) / d.img_pitch + 1;
    if (d.imgs > images) d.imgs = (int32_t)images;
    if (d.pitch > 256 || d.rows + 2 > 256 || d.imgs > 256) continue;
    const int64_t tiles = (int64_t)d.tiles_w * d.tiles_h * ((images + d.imgs - 1) / d.imgs), px = (int64_t)d.img_pitch * d.imgs;
    if (best_tiles == 0 || tiles < best_tiles || (tiles == best_tiles && px < best_px)) {
      best_tiles = tiles; best_px = px; *best = d;
    }
  }
  if (best_tiles == 0 || best_tiles > 0x3fffffff) return false;
  best->images = (int32_t)images;
  best->chunk = g.conv_c % 128 ? 64 : 128;
  best->chunks = g.conv_c / best->chunk;
  best->tx_bytes = (int32_t)(best_px * best->chunk);
  const int64_t reach = (int64_t)2 * best->pitch + 2 + BM;      // pixels the last tap's operand ends at
  best->bytes = (int32_t)(((reach > best_px ? reach : best_px) * best->chunk + 1023) / 1024 * 1024);
  return true;
}

// Tensor map of a convolution's NHWC code tensor for slab loads.
bool make_slab_map(CUtensorMap* map, const GemmArgs& g, int64_t images, const SlabDesc& d) {
  const MapKey key{g.a, (uint64_t)g.conv_c | ((uint64_t)g.conv_w << 32), (uint64_t)g.conv_h | ((uint64_t)images << 32),
                   (uint64_t)d.pitch | ((uint64_t)(d.rows + 2) << 16) | ((uint64_t)d.imgs << 32), (uint32_t)d.chunk, 0u, 0u, 0x200u, 0u};
  {
    std::lock_guard<std::mutex> lock(g_map_mutex);
    auto it = g_map_cache.find(key);
    if (it != g_map_cache.end()) { *map = it->second; return true; }
  }
  const cuuint64_t px = (cuuint64_t)g.conv_c;
  cuuint64_t dims[4] = {px, (cuuint64_t)g.conv_w, (cuuint64_t)g.conv_h, (cuuint64_t)images};
  cuuint64_t strides[3] = {px, px * g.conv_w, px * g.conv_w * g.conv_h};
  cuuint32_t box[4] = {(cuuint32_t)d.chunk, (cuuint32_t)d.pitch, (cuuint32_t)(d.rows + 2), (cuuint32_t)d.imgs}, estr[4] = {1, 1, 1, 1};
  const CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void*>(g.a), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                              d.chunk == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return false;
  std::lock_guard<std::mutex> lock(g_map_mutex);
  if (g_map_cache.size() >= kMapCacheMax) g_map_cache.clear();
  g_map_cache.emplace(key, *map);
  return true;
}

// chunk_bytes: bytes of the reduction per row of a box, and its swizzle span
int make_map(Ctx* ctx, CUtensorMap* map, const void* ptr, int is_bf16, int64_t k, int64_t rows, int64_t ld, int box_rows, int chunk_bytes = kStageKBytes) {
  const int esz = is_bf16 ? 2 : 1;
  if (!encode_2d(map, is_bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8, ptr, (uint64_t)k, (uint64_t)rows,
                 (uint64_t)(ld * esz), (uint32_t)(chunk_bytes / esz), (uint32_t)box_rows,
                 chunk_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                 CU_TENSOR_MAP_L2_PROMOTION_L2_256B))
    return set_error(ctx, QCFG_ECUDA, "cuTensorMapEncodeTiled failed");
  return QCFG_OK;
}

// Tensor map of an output matrix [m x n] for stores of 32-row pieces (32 columns, or 16 for 4-byte elements).  Returns false
// (direct stores are used instead) when the pointer or the row pitch is not 16-byte aligned.
bool make_out_map(CUtensorMap* map, const OutDesc& o, int64_t m, int64_t n) {
  int esz; CUtensorMapDataType dt;
  switch (o.kind) {
    case 1: esz = 1; dt = CU_TENSOR_MAP_DATA_TYPE_UINT8; break;
    case 2: esz = 2; dt = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16; break;
    case 3: esz = 4; dt = CU_TENSOR_MAP_DATA_TYPE_FLOAT32; break;
    default: esz = 4; dt = CU_TENSOR_MAP_DATA_TYPE_INT32; break;
  }
  if (((uintptr_t)o.ptr & 15) || ((o.ld * esz) & 15)) return false;
  return encode_2d(map, dt, o.ptr, (uint64_t)n, (uint64_t)m, (uint64_t)(o.ld * esz), esz == 4 ? 16u : 32u, 32u,
                   esz == 4 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE);
}

// Tensor map of the output a fast epilogue body writes: 32-row boxes of 64 int8 columns (64B
// swizzle), of 64 bf16 or of 32 fp32 columns (128B swizzle).
bool make_fast_map(CUtensorMap* map, const OutDesc& o, int64_t m, int64_t n) {
  const bool codes = o.kind == 1, half = o.kind == 2;
  const int esz = codes ? 1 : half ? 2 : 4;
  if (((uintptr_t)o.ptr & 15) || ((o.ld * esz) & 15)) return false;
  return encode_2d(map, codes ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : half ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32,
                   o.ptr, (uint64_t)n, (uint64_t)m, (uint64_t)(o.ld * esz), codes || half ? 64u : 32u, 32u, codes ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                   CU_TENSOR_MAP_L2_PROMOTION_NONE);
}

// Self-test of the bounded waits: the kernel waits on a barrier nothing ever arrives on and on
// counters (global and shared) nothing ever advances, each with a caller-chosen limit.  Every wait
// has to give up; only then does the last one set the time-out bit of the error word.  The kernel
// ends normally either way.
__global__ void wait_timeout_kernel(uint64_t limit_ns, unsigned* err, const unsigned* zero_word) {
  __shared__ uint64_t bar;
  __shared__ int abort_flag;
  __shared__ unsigned local_err;
  __shared__ uint32_t counters[kEpiWarps + 1];
  if (threadIdx.x == 0) {
    abort_flag = 0;
    local_err = 0;
    for (int i = 0; i <= kEpiWarps; ++i) counters[i] = 0;
    mbar_init(smem_u32(&bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  const int lane = threadIdx.x & 31;
  // whole-warp wait on the per-warp report counters
  const bool gave_up_rep = !reported_wait(smem_u32(&counters[0]), 1u, lane, &abort_flag, &local_err, limit_ns);
  bool all = gave_up_rep;
  if (threadIdx.x == 0) {
    abort_flag = 0;
    all = all && !cleared_wait(smem_u32(&counters[kEpiWarps]), 1u, &abort_flag, &local_err, limit_ns);
    abort_flag = 0;
    all = all && !flag_wait(zero_word, 1u, &abort_flag, &local_err, limit_ns);
    abort_flag = 0;
    if (all) (void)mbar_wait(smem_u32(&bar), 0, &abort_flag, err, limit_ns);
  }
}

}  // namespace

int launch_wait_timeout(Ctx* ctx, uint64_t limit_ns, cudaStream_t st) {
  ChainState* cs = static_cast<ChainState*>(chain_slot(ctx));
  if (!cs) return set_error(ctx, QCFG_ESTATE, "wait self-test: context not initialised");
  wait_timeout_kernel<<<1, 32, 0, st>>>(limit_ns, err_word(ctx), cs->zero);
  count_launch(ctx);
  return check_cuda(ctx, cudaGetLastError(), "wait self-test launch");
}

int gemm_init(Ctx* ctx) {
  if (!g_encode) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres);
    if (e != cudaSuccess || qres != cudaDriverEntryPointSuccess || !fn)
      return set_error(ctx, QCFG_ECUDA, "cuTensorMapEncodeTiled entry point not found");
    void* fi = nullptr;
    e = cudaGetDriverEntryPoint("cuTensorMapEncodeIm2col", &fi, cudaEnableDefault, &qres);
    if (e == cudaSuccess && qres == cudaDriverEntryPointSuccess) g_encode_im2col = reinterpret_cast<EncodeIm2colFn>(fi);
    else (void)cudaGetLastError();        // convolutions then keep the gather warps
    g_encode = reinterpret_cast<EncodeTiledFn>(fn);
  }
  ChainState* cs = new (std::nothrow) ChainState();
  if (!cs) return set_error(ctx, QCFG_ENOMEM, "gemm: host allocation failed");
  cudaError_t e = cudaMalloc(&cs->ring, kFlagRingBytes);
  if (e == cudaSuccess) e = cudaMemset(cs->ring, 0, kFlagRingBytes);
  if (e == cudaSuccess) e = cudaMalloc(&cs->zero, sizeof(unsigned));
  if (e == cudaSuccess) e = cudaMemset(cs->zero, 0, sizeof(unsigned));
  if (e != cudaSuccess) {
    if (cs->ring) cudaFree(cs->ring);
    if (cs->zero) cudaFree(cs->zero);
    delete cs;
    return check_cuda(ctx, e, "gemm chain counters");
  }
  chain_slot(ctx) = cs;
  return QCFG_OK;
}

void gemm_destroy(Ctx* ctx) {
  ChainState* cs = static_cast<ChainState*>(chain_slot(ctx));
  if (!cs) return;
  if (cs->ring) cudaFree(cs->ring);
  if (cs->zero) cudaFree(cs->zero);
  delete cs;
  chain_slot(ctx) = nullptr;
}

// ----- chains: consecutive GEMM launches of a forward pass folded into one cooperative launch

void gemm_chain_open(Ctx* ctx) {
  ChainState* cs = static_cast<ChainState*>(chain_slot(ctx));
  if (cs && ctx_chain_enabled(ctx)) cs->open = true;
}

int gemm_chain_flush(Ctx* ctx) {
  ChainState* cs = static_cast<ChainState*>(chain_slot(ctx));
  if (!cs || cs->args.n == 0) return QCFG_OK;
  const int n = cs->args.n;
  cs->args.n = 0;
  LaunchArgs<true>& A = cs->args;
  if (n == 1) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)cs->solo_grid);
    cfg.blockDim = dim3(kGemmThreads);
    cfg.dynamicSmemBytes = cs->solo_smem;
    cfg.stream = cs->st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 2; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    cs->solo.rec[0].p.stamp = prof_stamp(ctx, cs->bf16 ? 1 : 0, cs->ops);
    cs->ops = 0.0;
    const auto kern = cs->bf16 ? cs->solo_grouped ? gemm_kernel<true, true, true, false> : gemm_kernel<true, true, false, false>
                               : cs->solo_grouped ? gemm_kernel<false, true, true, false> : gemm_kernel<false, true, false, false>;
    cudaError_t le = make_ready(cs, (const void*)kern);
    if (le == cudaSuccess) le = cudaLaunchKernelEx(&cfg, kern, cs->solo);
    if (le != cudaSuccess) return check_cuda(ctx, le, "gemm launch");
    count_launch(ctx);
    return check_cuda(ctx, cudaGetLastError(), "gemm launch");
  }
  // counters: two per row tile and record, from a region nobody has used since it was cleared
  const int stride = 2 * A.rec[0].p.tiles_m;
  const size_t need = (size_t)n * stride * sizeof(unsigned);
  if (cs->ring_used + need > kFlagRingBytes) {
    // used up (once in a few thousand launches): wait for every launch that may still read it
    cudaError_t me = cudaDeviceSynchronize();
    if (me == cudaSuccess) me = cudaMemsetAsync(cs->ring, 0, kFlagRingBytes, cs->st);
    if (me != cudaSuccess) return check_cuda(ctx, me, "gemm chain counters");
    cs->ring_used = 0;
  }
  A.flags = cs->ring + cs->ring_used / sizeof(unsigned);
  cs->ring_used += need;
  A.flag_stride = stride;
  A.n = n;
  int total = 0;
  for (int i = 0; i < n; ++i) {
    GemmParams& rp = A.rec[i].p;
    total += rp.tiles_m * rp.tiles_n;
    rp.need = 0;
    for (int gi = 0; gi < kMaxGroups; ++gi)
      if (rp.grp[gi].tn_begin != 0x7fffffff && rp.grp[gi].signal) rp.need += rp.grp[gi].gtiles_n;
  }
  A.total_tiles = total;
  A.rec[0].p.stamp = prof_stamp(ctx, cs->bf16 ? 1 : 0, cs->ops);
  cs->ops = 0.0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)cs->grid);
  cfg.blockDim = dim3(kGemmThreads + 64);      // two more warps: one publishes finished tiles, one clears tiles whose inputs are complete
  cfg.dynamicSmemBytes = cs->smem;
  cfg.stream = cs->st;
  cudaLaunchAttribute attr[3];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 2; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  attr[2].id = cudaLaunchAttributeCooperative;      // CTAs wait for tiles of other CTAs
  attr[2].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 3;
  const auto kern = cs->bf16 ? gemm_kernel<true, true, true, true> : gemm_kernel<false, true, true, true>;
  cudaError_t le = make_ready(cs, (const void*)kern);
  if (le == cudaSuccess) le = cudaLaunchKernelEx(&cfg, kern, A);
  A.n = 0;
  if (le == cudaErrorCooperativeLaunchTooLarge || le == cudaErrorNotSupported) {
    // The device cannot keep the whole grid resident right now (or does not take cooperative
    // launches): nothing ran.  The records go out one by one through the ordinary flavour, in
    // their order, and this context stops chaining.
    (void)cudaGetLastError();
    ctx_disable_chains(ctx);
    cudaLaunchConfig_t one = cfg;
    one.blockDim = dim3(kGemmThreads);
    one.numAttrs = 2;
    for (int i = 0; i < n; ++i) {
      memset(&cs->solo, 0, sizeof(cs->solo));
      memcpy(cs->solo.rec[0].m, A.rec[i].m, sizeof(A.rec[i].m));     // pool indices stay valid in the larger pool
      cs->solo.rec[0].p = A.rec[i].p;
      for (int d = 0; d < kMaxDeps; ++d) cs->solo.rec[0].p.deps[d] = -1;
      cs->solo.n = 1;
      cs->solo.total_tiles = A.rec[i].p.tiles_m * A.rec[i].p.tiles_n;
      const auto apart = cs->bf16 ? gemm_kernel<true, true, true, false> : gemm_kernel<false, true, true, false>;
      cudaError_t se = make_ready(cs, (const void*)apart);
      if (se == cudaSuccess) se = cudaLaunchKernelEx(&one, apart, cs->solo);
      if (se != cudaSuccess) return check_cuda(ctx, se, "gemm launch");
      count_launch(ctx);
    }
    return check_cuda(ctx, cudaGetLastError(), "gemm launch");
  }
  if (le != cudaSuccess) return check_cuda(ctx, le, "gemm chain launch");
  count_launch(ctx);
  return check_cuda(ctx, cudaGetLastError(), "gemm chain launch");
}

int gemm_chain_close(Ctx* ctx) {
  ChainState* cs = static_cast<ChainState*>(chain_slot(ctx));
  if (!cs) return QCFG_OK;
  cs->open = false;
  return gemm_chain_flush(ctx);
}

// After a device-side wait gave up, counters of unfinished launches may be left behind.
int gemm_chain_reset(Ctx* ctx) {
  ChainState* cs = static_cast<ChainState*>(chain_slot(ctx));
  if (!cs) return QCFG_OK;
  cs->args.n = 0;
  cs->ops = 0.0;
  cs->ring_used = 0;
  return check_cuda(ctx, cudaMemset(cs->ring, 0, kFlagRingBytes), "gemm chain counters reset");
}

// Tile width a GEMM of n columns gets.
static int tile_n_of(int64_t n) { return n <= 32 ? 32 : n <= 64 ? 64 : n <= 128 ? 128 : 256; }

bool gemm_groupable(const GemmArgs& a, const GemmArgs& b) {
  if (a.conv_kh > 0 || b.conv_kh > 0) return false;
  return a.m == b.m && a.k == b.k && a.is_bf16 == b.is_bf16 && tile_n_of(a.n) == tile_n_of(b.n);
}

// The body for shortcut layers leaves room for a ring of two stages, stages twice the operand bytes of a 256-column pair
// tile and joins no chain, so it pays while the reduction is short against the blocks it moves.  us for such a
// layer between three small ones, this body / the general one:
//   12288 x 768    k = 768 39.3 / 48.6    1024 43.1 / 53.3    1280 48.1 / 55.6    1536 53.4 / 57.3    2048 66.4 / 64.2
//   25088 x 1024   k = 768 95.7 / 107.7   1024 110.3 / 111.0  1280 124.1 / 116.5
//   50176 x 512    k = 768 113.5 / 119.3  1024 128.2 / 125.5
//   6144 x 1024    k = 1280 36.7 / 44.3   1536 40.0 / 47.6    2048 45.4 / 48.9
//   3072 x 768     k = 1536 25.2 / 31.0   2048 26.9 / 32.2    3072 31.1 / 35.5     (one tile per CTA: no ring to keep full)
// Alone it would also pay at 1536 in few rounds of tiles and at 3072 with one tile per CTA.  In a stack it does not, where the
// general body's launches overlap their neighbours or join a chain: four transformer blocks with shortcuts, hidden / ffn,
// 768 / 1536 at 12288 rows 441 / 404, 1024 / 1536 at 6144 rows 337 / 305, 768 / 3072 at 3072 rows 242 / 236, 1024 / 4096 at 1500 rows
// 249 / 224; 768 / 1024 at 12288 rows 395 / 379 and at 6144 rows 254 / 288.
static bool shortcut_body_pays(const GemmArgs& g, int bn, int sms) {
  const int64_t width = bn > 128 ? 128 : bn;
  if (g.k <= 768) return true;
  if (g.k <= 2048 && ((g.m + BM - 1) / BM) * ((g.n + width - 1) / width) <= sms) return true;
  return g.k <= 1280 && g.m * g.k <= (g.k <= 1024 ? (int64_t)32 << 20 : (int64_t)16 << 20);
}

// The body that writes fp32 rows line by line turns whole 128-column halves of a tile and has its warps meet twice per half; the
// general one works in 32-column chunks, with a shuffle per element at int8, and leaves more sectors half written, which costs
// most once the output no longer fits in L2.  us per launch, general / line by line:
//   int8    38001 x 131, k = 64: 14.2 / 16.0    75719 x 150: 20.9 / 22.5    75719 x 177: 22.5 / 22.2    38001 x 201: 16.5 / 16.5    38001 x 255: 18.4 / 16.2
//           12000 x 513: 14.4 / 12.4    12000 x 2049: 34.5 / 30.2    12000 x 4001: 89.2 / 51.8
//   16 bit  38001 x 131, k = 500: 15.1 / 17.5    38001 x 201: 17.2 / 17.8    38001 x 255: 18.8 / 18.4
//           6000 x 3999 (96 MB), k = 64: 24.9 / 26.5    256: 29.6 / 31.4    500: 41.0 / 39.5    1024: 63.1 / 59.5
//           12000 x 2049 (98 MB), k = 64: 25.2 / 26.6    256: 30.9 / 31.7    500: 45.0 / 40.8    1024: 68.4 / 60.0
//           8231 x 3999 (132 MB), k = 64: 54.7 / 42.3    12000 x 4001 (192 MB), k = 64: 89.4 / 47.1    500: 91.7 / 74.7
static bool rows_body_pays(const GemmArgs& g) {
  if (g.n <= (g.is_bf16 ? 208 : 176)) return false;      // few columns of the second half
  return !g.is_bf16 || g.k >= 500 || 4 * g.m * g.n > (int64_t)96 << 20;
}

// Whether a convolution goes by slabs (and how it is cut).  Integer widths only: the reduction runs chunk by chunk, tap by
// tap inside, and only integer sums do not depend on the order.
// By slabs / by im2col loads, us of a launch between two small ones, channels x channels, side, images:
//   weights resident   64 56 128: 128 / 163   128 28 128: 52 / 61   64 8 128: 10.5 / 11.3   128 8 128: 12.9 / 14.0   128 28 8: 13.9 / 12.5 (56 tiles)
//   weights streamed   256 14 128: 28.4 / 31.2   512 7 128: 25 / 27.7   512 6 128: 24.2 / 25.4 (64 tiles, 36 runs)   256 9 128: 21.3 / 21.7
//                      256 8 128: 19.0 / 18.3 (128 tiles, 64 runs)   256 12 128: 26.2 / 21.7 (two rounds of CTA pairs in place of one)   256 14 8: 16.0 / 14.4
//   ... of 128 columns or fewer (three slabs of the cut leave the weights no room): 128 40 32: 38.5 / 35.2   128 40 128: 110.0 / 104.6   128 -> 96 40 64: 67.6 / 65.9
//   so such a convolution goes by slabs only with its weights resident.  Streamed without CTA pairs: 256 14 128: 39.1 / 38.7   256 40 16: 40.6 / 40.4   512 7 128: 31.6 / 30.9
static bool slab_pays(const GemmArgs& g, int sms, SlabDesc* sd) {
  if (g.conv_kh != 3 || g.conv_kw != 3 || g.conv_stride != 1 || g.is_bf16 || g.conv_c % 64 || g.n % 32 || g.residual || g.amax || g.acc || g.y ||
      g.slots[0].kind != 1 || g.slots[1].kind || g.slots[2].kind || ((uintptr_t)g.slots[0].ptr & 15) || g.slots[0].ld % 16)
    return false;
  const int OH = g.conv_h + 2 * g.conv_pad - 2, OW = g.conv_w + 2 * g.conv_pad - 2;
  if (OH < 1 || OW < 1 || g.m % ((int64_t)OH * OW) || g.conv_pad > 127 || g.m > 0x7fffffff) return false;
  if (!slab_plan(g, g.m / ((int64_t)OH * OW), OH, OW, sd)) return false;
  const int64_t tiles = (int64_t)sd->tiles_w * sd->tiles_h * ((sd->images + sd->imgs - 1) / sd->imgs), runs = (g.m + BM - 1) / BM;
  if (sd->bytes > 40 * 1024) return false;
  sd->count = 3;
  sd->resident = sd->chunks == 1 && g.n <= 128;
  if (sd->resident) {      // one column tile of the width tile_n_of gives: 2 * tiles > sms leaves it as it is
    const int weights = 9 * tile_n_of(g.n) * sd->chunk;
    if (3 * sd->bytes + weights > kSlabRoom) return false;
    if (4 * sd->bytes + weights <= kSlabRoom) sd->count = kMaxSlabs;
    return 2 * tiles > sms && tiles <= 2 * runs;
  }
  const int64_t cols = (g.n + 255) / 256;
  auto rounds = [&](int64_t t) { return ((t + 1) / 2 * cols + sms / 2 - 1) / (sms / 2); };
  return g.n > 128 && sms > 1 && tiles * ((g.n + 127) / 128) > sms && rounds(tiles) <= rounds(runs) && 5 * tiles <= 9 * runs;
}

int launch_gemm_group(Ctx* ctx, const GemmArgs* gs_in, int count, cudaStream_t st) {
  if (count < 1 || count > kMaxGroups) return set_error(ctx, QCFG_EINVAL, "gemm: %d groups", count);
  // While launches are being chained a record's tiles run group after group.  Of three groups,
  // those that write operand codes for later layers go in the middle: the group before them gives
  // the previous record time to complete the rows they read, the group after them gives their own
  // rows time to complete before the next record asks for them.  Of two, they go first.
  GemmArgs ordered[kMaxGroups];
  {
    ChainState* st_ = static_cast<ChainState*>(chain_slot(ctx));
    if (st_ && st_->open && count > 1) {
      int feed[kMaxGroups], n_feed = 0, rest[kMaxGroups], n_rest = 0;
      for (int i = 0; i < count; ++i) {
        bool feeds = false;
        for (int s = 0; s < kMaxSlots; ++s) feeds = feeds || gs_in[i].slots[s].kind != 0;
        if (feeds) feed[n_feed++] = i; else rest[n_rest++] = i;
      }
      int k = 0;
      const int before = count == 3 ? (n_rest + 1) / 2 : 0;   // two groups: the feeder first, the other one is the buffer
      for (int i = 0; i < before; ++i) ordered[k++] = gs_in[rest[i]];
      for (int i = 0; i < n_feed; ++i) ordered[k++] = gs_in[feed[i]];
      for (int i = before; i < n_rest; ++i) ordered[k++] = gs_in[rest[i]];
    } else {
      for (int i = 0; i < count; ++i) ordered[i] = gs_in[i];
    }
  }
  const GemmArgs* gs = ordered;
  const GemmArgs& g0 = gs[0];
  const int esz = g0.is_bf16 ? 2 : 1;
  for (int i = 0; i < count; ++i) {
    const GemmArgs& g = gs[i];
    if (g.m <= 0 || g.n <= 0 || g.k <= 0) return set_error(ctx, QCFG_ESHAPE, "gemm: m, n, k must be positive");
    if (((uintptr_t)g.a & 15) || ((uintptr_t)g.b & 15) || (g.lda * esz) % 16 || (g.ldb * esz) % 16)
      return set_error(ctx, QCFG_EALIGN, "gemm: operands need 16-byte aligned pointers and row strides");
    if (g.conv_kh > 0) {
      if (count > 1) return set_error(ctx, QCFG_EINVAL, "gemm: convolutions are launched alone");
      if ((g.conv_c * esz) % 16 || g.lda != g.conv_c || g.k != (int64_t)g.conv_kh * g.conv_kw * g.conv_c || g.conv_stride < 1)
        return set_error(ctx, QCFG_ESHAPE, "gemm: convolution needs channels in whole 16-byte chunks and k = kh*kw*c");
      if (g.ldb < g.k) return set_error(ctx, QCFG_ESHAPE, "gemm: leading dimension below k");
    } else if (g.lda < g.k || g.ldb < g.k) return set_error(ctx, QCFG_ESHAPE, "gemm: leading dimension below k");
    if (g.m > 0x7fffffff || g.n > 0x7fffffff) return set_error(ctx, QCFG_ESHAPE, "gemm: dimension too large");
    if (i && !gemm_groupable(g0, g)) return set_error(ctx, QCFG_EINVAL, "gemm: grouped launches need equal m, k, type and tile width");
  }

  // Tile width: by the output's width, then halved while every CTA of the launch still has one tile at
  // most: a launch that fills half of the SMs or fewer is as long as one tile, and half a tile is
  // shorter (a mixed 4/8/16-bit block of 768 x 3072 at 3072 tokens: 76.6 -> 74.1 us; the results do not
  // depend on the tile width).
  int bn = tile_n_of(g0.n);
  // Slab tiles of a convolution in place of runs of 128 output pixels
  SlabDesc sd{};
  CUtensorMap slab_map;
  const bool slab = count == 1 && slab_pays(g0, sm_count(ctx), &sd) && make_slab_map(&slab_map, g0, sd.images, sd);
  const int64_t row_tiles = slab ? (int64_t)sd.tiles_w * sd.tiles_h * ((sd.images + sd.imgs - 1) / sd.imgs) : (g0.m + BM - 1) / BM;
  {
    const int sms = sm_count(ctx);
    auto ctas = [&](int width) {
      int64_t cols = 0;
      for (int i = 0; i < count; ++i) cols += (gs[i].n + width - 1) / width;
      return cols * row_tiles;
    };
    while (bn > 32 && ctas(bn / 2) <= sms) bn /= 2;
  }
  // Shortcut layers at integer widths whose matrices TMA can reach: a body of its own, which keeps two fp32
  // blocks per epilogue warp in shared memory and therefore works on 128 columns at most.
  bool shortcut = false;
  if (count == 1 && !g0.is_bf16 && g0.residual && shortcut_body_pays(g0, bn, sm_count(ctx)) && (g0.y || g0.slots[0].kind) && !g0.acc && !g0.amax && g0.conv_kh == 0 && !g0.slots[2].kind) {
    auto aligned = [](const void* q, int64_t ld_bytes) { return ((uintptr_t)q & 15) == 0 && (ld_bytes & 15) == 0; };
    shortcut = aligned(g0.residual, g0.ldr * 4) && (!g0.y || aligned(g0.y, g0.ldy * 4));
    for (int i = 0; i < 2; ++i)
      if (g0.slots[i].kind) shortcut = shortcut && g0.slots[i].kind == 1 && aligned(g0.slots[i].ptr, g0.slots[i].ld);
    if (shortcut && bn > 128) bn = 128;
  }
  GemmParams p{};
  p.m = (int32_t)g0.m;
  const int64_t kbytes = g0.k * esz;
  p.k_blocks = (int32_t)((kbytes + kStageKBytes - 1) / kStageKBytes);
  p.bn = bn;
  // pair flavour (two CTAs per 256-row tile, cta_group::2) for wide outputs with at least two
  // row tiles: it halves the B bytes each SM stages per k-block
  bool pair = ctx_pair_enabled(ctx) && bn == 256 && (slab ? row_tiles > 1 && sd.chunk == 128 : g0.m > BM) && sm_count(ctx) >= 2;
  // ... and for wide outputs whose tiles were narrowed to 128 columns, while the pairs still have one tile each: a
  // stage is 24 KB instead of 32 and the ring one or two stages deeper (noise table of the block above:
  // 360 -> 345 us; its evaluation 66.5 -> 66.2).  A lone int8 code matrix stays with one CTA per tile, where its own body
  // is.  Four SMs are left out of the count: some may have no partner.
  if (ctx_pair_enabled(ctx) && bn == 128 && tile_n_of(g0.n) == 256 && !shortcut && g0.conv_kh == 0 && g0.m > BM) {
    int64_t cols = 0;
    for (int i = 0; i < count; ++i) cols += (gs[i].n + bn - 1) / bn;
    const bool codes = count == 1 && !g0.residual && !g0.amax && !g0.acc && !g0.y && g0.slots[0].kind == 1 && !g0.slots[1].kind && !g0.slots[2].kind;
    pair = !codes && 2 * cols * ((g0.m + 2 * BM - 1) / (2 * BM)) <= sm_count(ctx) - 4;
  }
  const int tile_rows = pair ? 2 * BM : BM;
  p.tiles_m = slab ? (int32_t)(pair ? (row_tiles + 1) / 2 : row_tiles) : (int32_t)((g0.m + tile_rows - 1) / tile_rows);
  const int stage_bytes = slab ? (pair ? bn / 2 : bn) * sd.chunk : (BM + (pair ? bn / 2 : bn)) * kStageKBytes;
  p.is_bf16 = g0.is_bf16;
  // instruction descriptor: D format (F32 = 1, S32 = 2) at bit 4, A/B format (BF16 = 1, S8 = 1)
  // at bits 7 and 10, both operands K-major, N/8 at bit 17, M/16 at bit 24
  p.idesc = ((g0.is_bf16 ? 1u : 2u) << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(bn >> 3) << 17) | ((uint32_t)(tile_rows >> 4) << 24);
  p.err = err_word(ctx);

  CUtensorMap maps[kPoolAll];      // group i's maps at i * kMapsPerGroup + MAP_*
  memset(maps, 0, sizeof(maps));
  for (int i = 0; i < kMaxGroups; ++i)
    for (int j = 0; j < kMapsPerGroup; ++j) p.mi[i][j] = (uint8_t)(i * kMapsPerGroup + j);
  bool wide = false;
  int32_t tn_total = 0;
  double ops = 0.0;
  for (int i = 0; i < kMaxGroups; ++i) { p.grp[i].tn_begin = 0x7fffffff; p.grp[i].tile_first = 0x7fffffff; p.grp[i].gtiles_n = 1; }
  for (int i = 0; i < count; ++i) {
    const GemmArgs& g = gs[i];
    GroupDesc& G = p.grp[i];
    G.n = (int32_t)g.n;
    G.tn_begin = tn_total;
    G.gtiles_n = (int32_t)((g.n + bn - 1) / bn);
    G.tile_first = p.tiles_m * tn_total;
    tn_total += (int32_t)((g.n + bn - 1) / bn);
    G.scale_x = g.scale_x; G.scale_w = g.scale_w; G.act = g.act;
    G.residual = g.residual; G.ldr = g.ldr;
    G.amax = reinterpret_cast<unsigned*>(g.amax);
    if (g.acc && !g.is_bf16) { G.outs[0].kind = 4; G.outs[0].ptr = g.acc; G.outs[0].ld = g.n; }
    if (g.y) { G.outs[1].kind = 3; G.outs[1].ptr = g.y; G.outs[1].ld = g.ldy; }
    G.need_y = g.y != nullptr || g.amax != nullptr;
    for (int s = 0; s < kMaxSlots; ++s) {
      if (!g.slots[s].kind) continue;
      OutDesc& o = G.outs[2 + s];
      o.kind = g.slots[s].kind; o.ptr = g.slots[s].ptr; o.ld = g.slots[s].ld;
      o.inv_scale = g.slots[s].inv_scale; o.qmax = g.slots[s].qmax;
      G.need_y = 1;
    }
    if (!G.need_y && !G.outs[0].kind) return set_error(ctx, QCFG_EINVAL, "gemm: no output requested");
    if (G.need_y && !g.is_bf16 && !g.scale_w) return set_error(ctx, QCFG_EINVAL, "gemm: scale_w is null");
    for (int j = 0; j < kNumOuts; ++j)
      if (G.outs[j].kind) G.outs[j].tma = make_out_map(&maps[i * kMapsPerGroup + MAP_OUT + j], G.outs[j], g.m, g.n) ? 1 : 0;
    // staging per epilogue warp: two slots of 1 KB when only int8 codes are written, else of 2 KB
    for (int j = 0; j < kNumOuts; ++j) if (G.outs[j].kind >= 3 || (G.outs[j].kind == 2 && G.outs[j].tma)) wide = true;
    G.mode = EPI_GENERAL;
    if (bn < 256 && !pair && count == 1 && !G.residual && !G.amax && !G.outs[0].kind && !G.outs[1].kind && G.outs[2].kind == 1 && G.outs[2].tma &&
        !G.outs[3].kind && !G.outs[4].kind)
      G.mode = EPI_CODES32;
    if (bn == 256 && !G.residual && !G.outs[0].kind && !G.outs[1].kind && G.outs[2].kind == 2 && !G.outs[3].kind && !G.outs[4].kind &&
        make_fast_map(&maps[i * kMapsPerGroup + MAP_FAST], G.outs[2], g.m, g.n))
      G.mode = EPI_BF16;
    if (bn == 256 && !G.residual && !G.amax && !G.outs[0].kind && !G.outs[3].kind && !G.outs[4].kind) {
      if (!G.outs[1].kind && G.outs[2].kind == 1 && make_fast_map(&maps[i * kMapsPerGroup + MAP_FAST], G.outs[2], g.m, g.n)) G.mode = EPI_CODES1;
      else if (G.outs[1].kind && !G.outs[2].kind && make_fast_map(&maps[i * kMapsPerGroup + MAP_FAST], G.outs[1], g.m, g.n)) { G.mode = EPI_Y; wide = true; }
    }
    if (bn < 256 && (!pair || count > 1) && !shortcut && !g.is_bf16 && g.conv_kh == 0 && !G.residual && !G.amax && !G.outs[0].kind && G.outs[1].kind && !G.outs[2].kind && !G.outs[3].kind &&
        !G.outs[4].kind && make_fast_map(&maps[i * kMapsPerGroup + MAP_FAST], G.outs[1], g.m, g.n))
      G.mode = EPI_Y32;
    if (shortcut) {      // MAP_OUT, the raw accumulators' place, holds the shortcut's map
      OutDesc in{};
      in.kind = 3; in.ptr = const_cast<float*>(g.residual); in.ld = g.ldr;
      if ((g.y && !make_fast_map(&maps[MAP_FAST], G.outs[1], g.m, g.n)) || !make_fast_map(&maps[MAP_OUT], in, g.m, g.n))
        return set_error(ctx, QCFG_ECUDA, "cuTensorMapEncodeTiled failed");
      for (int j = 2; j < 4; ++j)
        if (G.outs[j].kind && !G.outs[j].tma) return set_error(ctx, QCFG_ECUDA, "cuTensorMapEncodeTiled failed");
      G.mode = EPI_SHORTCUT;
    }
    int rc = g.conv_kh > 0 ? QCFG_OK : make_map(ctx, &maps[i * kMapsPerGroup + MAP_A], g.a, g.is_bf16, g.k, g.m, g.lda, BM);
    if (rc == QCFG_OK) rc = make_map(ctx, &maps[i * kMapsPerGroup + MAP_B], g.b, g.is_bf16, g.k, g.n, g.ldb, pair ? bn / 2 : bn, slab ? sd.chunk : kStageKBytes);
    if (rc != QCFG_OK) return rc;
    ops += 2.0 * (double)g.m * (double)g.n * (double)g.k;
  }
  p.tiles_n = tn_total;
  // an fp32 matrix that TMA cannot write, in whole 256-column tiles, and nothing else (narrower tiles keep the general body)
  const bool rows_out = count == 1 && bn == 256 && rows_body_pays(g0) && g0.conv_kh == 0 && !g0.residual && !g0.amax && !p.grp[0].outs[0].kind && p.grp[0].outs[1].kind &&
                        !p.grp[0].outs[1].tma && !p.grp[0].outs[2].kind && !p.grp[0].outs[3].kind && !p.grp[0].outs[4].kind;
  const bool conv = g0.conv_kh > 0;
  if (conv) {
    ConvDesc& cv = p.conv;
    cv.on = CONV_GATHER; cv.H = g0.conv_h; cv.W = g0.conv_w; cv.C = g0.conv_c; cv.kh = g0.conv_kh; cv.kw = g0.conv_kw;
    cv.stride = g0.conv_stride; cv.pad = g0.conv_pad; cv.esz = esz; cv.K = (int32_t)g0.k;
    cv.OH = (cv.H + 2 * cv.pad - cv.kh) / cv.stride + 1;
    cv.OW = (cv.W + 2 * cv.pad - cv.kw) / cv.stride + 1;
    cv.img_bytes = (int64_t)cv.H * cv.W * cv.C * esz;
    cv.src = reinterpret_cast<const uint8_t*>(g0.a);
    if (cv.OH < 1 || cv.OW < 1 || g0.m % ((int64_t)cv.OH * cv.OW))
      return set_error(ctx, QCFG_ESHAPE, "gemm: convolution rows are not a whole number of images");
    // TMA in its im2col mode where the channels come in whole 64-byte chunks, gather warps otherwise
    const int64_t images = g0.m / ((int64_t)cv.OH * cv.OW), cbytes = (int64_t)cv.C * esz;
    if (slab) {
      maps[MAP_A] = slab_map;
      cv.on = CONV_SLAB;
    } else if (cbytes % 128 == 0 && make_im2col_map(&maps[MAP_A], g0, images, 128)) cv.on = CONV_TMA128;
    else if (cbytes % 64 == 0 && make_im2col_map(&maps[MAP_A], g0, images, 64)) cv.on = CONV_TMA64;
  }
  // Launches that may join a chain all take the larger staging size, so any sequence of them
  // shares one shared-memory layout.
  ChainState* cs = static_cast<ChainState*>(chain_slot(ctx));
  if (!cs) return set_error(ctx, QCFG_ESTATE, "gemm: context not initialised");
  // (a GEMM with fewer tiles than CTA pairs has nothing to overlap with: the wait for its
  // producer's rows would cost more than the launch boundary it saves)
  const bool chainable = cs->open && ctx_chain_enabled(ctx) && pair && !conv && !rows_out && bn == 256 && prof_mode(ctx) != 1 && p.tiles_m <= kChainMaxTilesM &&
                         2 * p.tiles_m * p.tiles_n >= sm_count(ctx);
  p.alternate = !pair && bn == 64 && (slab || p.grp[0].mode == EPI_CODES32);
  p.epi_bytes = slab ? 0 : shortcut ? kShortcutBytes : (wide || chainable) ? 4096 : 2048;
  if (slab) {
    if (sd.resident && (pair || p.tiles_n != 1)) return set_error(ctx, QCFG_ESHAPE, "gemm: resident weights need one column tile");
    p.slab = sd;
    p.k_blocks = 9 * sd.chunks;
  }
  int stages = (kSmemMax - kSmemHeader - kCsBytes - 1024 - kEpiWarps * p.epi_bytes - (slab ? sd.count * sd.bytes : 0)) / stage_bytes;
  if (stages > kMaxStages) stages = kMaxStages;
  if (slab && sd.resident) stages = p.k_blocks;
  if (stages <= (shortcut ? 1 : kGatherDepth)) return set_error(ctx, QCFG_ESHAPE, "gemm: too few pipeline stages");
  p.stages = stages;

  const int num_tiles = p.tiles_m * p.tiles_n;
  int grid = sm_count(ctx);
  if (pair) {
    int* cached = pair_cluster_cache(ctx) + (g0.is_bf16 ? 1 : 0);
    if (*cached == 0) {     // how many CTA pairs the device keeps resident at once
      cudaLaunchConfig_t q = {};
      q.gridDim = dim3((unsigned)(grid & ~1));
      q.blockDim = dim3(kGemmThreads);
      q.dynamicSmemBytes = kSmemMax;
      cudaLaunchAttribute qa[1];
      qa[0].id = cudaLaunchAttributeClusterDimension;
      qa[0].val.clusterDim.x = 2; qa[0].val.clusterDim.y = 1; qa[0].val.clusterDim.z = 1;
      q.attrs = qa; q.numAttrs = 1;
      int n = 0;
      const auto probe = g0.is_bf16 ? gemm_kernel<true, true, true, true> : gemm_kernel<false, true, true, true>;
      cudaError_t oe = make_ready(cs, (const void*)probe);
      if (oe == cudaSuccess) oe = cudaOccupancyMaxActiveClusters(&n, probe, &q);
      if (oe != cudaSuccess || n < 1) { (void)cudaGetLastError(); n = grid / 2; }
      if (n > grid / 2) n = grid / 2;
      *cached = n;
    }
    grid = 2 * (*cached);
    if (grid > 2 * num_tiles && !chainable) grid = 2 * num_tiles;
  } else if (grid > num_tiles) grid = num_tiles;
  const size_t smem = (size_t)kSmemHeader + kCsBytes + 1024 + (size_t)kEpiWarps * p.epi_bytes + (size_t)stages * stage_bytes +
                      (slab ? (size_t)sd.count * sd.bytes : 0);
  // a chain record carries only the distinct maps it uses; one that needs more runs on its own
  CUtensorMap pool[kPoolChain];
  bool fits = true;
  if (chainable) {
    memset(pool, 0, sizeof(pool));
    int used = 0;
    auto place = [&](int i, int j) {
      const CUtensorMap& mm = maps[i * kMapsPerGroup + j];
      int at = -1;
      for (int u = 0; u < used && at < 0; ++u) if (memcmp(&pool[u], &mm, sizeof(CUtensorMap)) == 0) at = u;
      if (at < 0) {
        if (used == kPoolChain) { fits = false; return; }
        pool[used] = mm; at = used++;
      }
      p.mi[i][j] = (uint8_t)at;
    };
    for (int i = 0; i < kMaxGroups; ++i)
      for (int j = 0; j < kMapsPerGroup; ++j) p.mi[i][j] = 0;
    for (int i = 0; i < count && fits; ++i) {
      place(i, MAP_A);
      place(i, MAP_B);
      if (p.grp[i].mode != EPI_GENERAL) {       // a fast body writes through this one map only
        place(i, MAP_FAST);
        continue;
      }
      for (int j = 0; j < kNumOuts && fits; ++j)
        if (p.grp[i].outs[j].kind && p.grp[i].outs[j].tma) place(i, MAP_OUT + j);
    }
    if (!fits)
      for (int i = 0; i < kMaxGroups; ++i)
        for (int j = 0; j < kMapsPerGroup; ++j) p.mi[i][j] = (uint8_t)(i * kMapsPerGroup + j);
  }
  const bool chained = chainable && fits;
  if (cs->args.n > 0 &&
      (!chained || cs->args.n == kChainMax || cs->st != st || cs->bf16 != (g0.is_bf16 != 0) || cs->grid != grid ||
       cs->smem != smem || cs->m != g0.m)) {
    const int rc = gemm_chain_flush(ctx);
    if (rc != QCFG_OK) return rc;
  }
  if (chained) {
    // What the record reads and writes, as byte ranges.  Reading rows an earlier record of the
    // chain writes is a dependency the kernel waits for; any other overlap ends the chain first.
    ChainRecInfo info{};
    bool b_clash = false;
    auto overlap = [](const Span& x, const Span& y) { return x.lo < y.hi && y.lo < x.hi; };
    auto span_of = [&](const void* ptr, int64_t ld, int64_t cols, int esz_) {
      const uint8_t* lo = static_cast<const uint8_t*>(ptr);
      return Span{lo, lo + ((g0.m - 1) * ld + cols) * esz_};
    };
    for (int i = 0; i < count; ++i) {
      const GemmArgs& g = gs[i];
      info.in[info.n_in++] = span_of(g.a, g.lda, g.k, esz);
      if (g.residual) info.in[info.n_in++] = span_of(g.residual, g.ldr, g.n, 4);
      for (int j = 0; j < kNumOuts; ++j) {
        const OutDesc& o = p.grp[i].outs[j];
        if (o.kind) { info.out_grp[info.n_out] = i; info.out[info.n_out++] = span_of(o.ptr, o.ld, g.n, o.kind == 1 ? 1 : o.kind == 2 ? 2 : 4); }
      }
      // weights and their scales are never chain outputs in a forward pass; if they were, run apart
      const uint8_t* blo = static_cast<const uint8_t*>(g.b);
      const Span bs{blo, blo + ((g.n - 1) * g.ldb + g.k) * esz};
      for (int r = 0; r < cs->args.n; ++r)
        for (int o = 0; o < cs->info[r].n_out; ++o) b_clash = b_clash || overlap(bs, cs->info[r].out[o]);
    }
    int deps[kMaxDeps], n_deps = 0;
    bool read_grp[kChainMax][kMaxGroups] = {};
    bool clash = b_clash;
    for (int r = 0; r < cs->args.n && !clash; ++r) {
      const ChainRecInfo& E = cs->info[r];
      for (int o = 0; o < info.n_out && !clash; ++o) {
        for (int x = 0; x < E.n_in; ++x) clash = clash || overlap(info.out[o], E.in[x]);
        for (int x = 0; x < E.n_out; ++x) clash = clash || overlap(info.out[o], E.out[x]);
      }
      bool reads = false;
      for (int x = 0; x < info.n_in; ++x)
        for (int o = 0; o < E.n_out; ++o)
          if (overlap(info.in[x], E.out[o])) { reads = true; read_grp[r][E.out_grp[o]] = true; }
      if (reads) {
        if (n_deps == kMaxDeps) clash = true;
        else deps[n_deps++] = r;
      }
    }
    if (clash) {
      const int rc = gemm_chain_flush(ctx);
      if (rc != QCFG_OK) return rc;
      n_deps = 0;
    }
    for (int d = 0; d < kMaxDeps; ++d) p.deps[d] = d < n_deps ? deps[d] : -1;
    for (int d = 0; d < n_deps; ++d)
      for (int i = 0; i < kMaxGroups; ++i)
        if (read_grp[deps[d]][i]) cs->args.rec[deps[d]].p.grp[i].signal = 1;
    for (int i = 0; i < kMaxGroups; ++i) p.grp[i].signal = 0;
    p.need = 0;
    p.stamp = nullptr;
    const int slot = cs->args.n++;
    if (slot == 0) {
      GemmParams ps = p;
      for (int i = 0; i < kMaxGroups; ++i)
        for (int j = 0; j < kMapsPerGroup; ++j) ps.mi[i][j] = (uint8_t)(i * kMapsPerGroup + j);
      ps.epi_bytes = wide ? 4096 : 2048;
      int st_solo = (kSmemMax - kSmemHeader - kCsBytes - 1024 - kEpiWarps * ps.epi_bytes) / stage_bytes;
      if (st_solo > kMaxStages) st_solo = kMaxStages;
      ps.stages = st_solo;
      memcpy(cs->solo.rec[0].m, maps, sizeof(maps));
      cs->solo.rec[0].p = ps;
      cs->solo.n = 1; cs->solo.total_tiles = num_tiles; cs->solo.flag_stride = 0; cs->solo.flags = nullptr;
      cs->solo_grid = grid > 2 * num_tiles ? 2 * num_tiles : grid;
      cs->solo_grouped = count > 1 ? 1 : 0;
      cs->solo_smem = (size_t)kSmemHeader + kCsBytes + 1024 + (size_t)kEpiWarps * ps.epi_bytes + (size_t)st_solo * stage_bytes;
    }
    memcpy(cs->args.rec[slot].m, pool, sizeof(pool));
    cs->args.rec[slot].p = p;
    cs->info[slot] = info;
    cs->ops += ops;
    cs->st = st; cs->bf16 = g0.is_bf16 != 0; cs->grid = grid; cs->smem = smem; cs->m = g0.m;
    return QCFG_OK;
  }
  for (int d = 0; d < kMaxDeps; ++d) p.deps[d] = -1;
  // Programmatic dependent launch: the kernel's prologue (barrier set-up, TMEM allocation) may
  // start while the previous kernel in the stream drains; it waits (griddepcontrol.wait) before
  // touching global memory.
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(p.conv.on == CONV_GATHER ? kGemmThreadsConv : kGemmThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 2; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pair ? 2 : 1;
  using Kern = void (*)(const LaunchArgs<false>);
  static const Kern kernels[8] = {
      gemm_kernel<false, false, false, false>, gemm_kernel<false, false, true, false>, gemm_kernel<false, true, false, false>,
      gemm_kernel<false, true, true, false>,   gemm_kernel<true, false, false, false>,  gemm_kernel<true, false, true, false>,
      gemm_kernel<true, true, false, false>,   gemm_kernel<true, true, true, false>};
  static const Kern conv_kernels[4] = {
      gemm_kernel<false, false, false, false, FL_CONV>, gemm_kernel<false, true, false, false, FL_CONV>,
      gemm_kernel<true, false, false, false, FL_CONV>,  gemm_kernel<true, true, false, false, FL_CONV>};
  static const Kern slab_kernels[3] = {gemm_kernel<false, false, false, false, FL_SLAB64>, gemm_kernel<false, false, false, false, FL_SLAB>,
                                       gemm_kernel<false, true, false, false, FL_SLAB>};
  static const Kern rows_kernels[4] = {gemm_kernel<false, false, false, false, FL_ROWS>, gemm_kernel<false, true, false, false, FL_ROWS>,
                                       gemm_kernel<true, false, false, false, FL_ROWS>, gemm_kernel<true, true, false, false, FL_ROWS>};
  const Kern kern = rows_out ? rows_kernels[(g0.is_bf16 ? 2 : 0) + (pair ? 1 : 0)] : slab ? slab_kernels[sd.chunk == 64 ? 0 : pair ? 2 : 1] : shortcut ? gemm_kernel<false, false, false, false, FL_SHORTCUT>
                    : conv   ? conv_kernels[(g0.is_bf16 ? 2 : 0) + (pair ? 1 : 0)]
                             : kernels[(g0.is_bf16 ? 4 : 0) + (pair ? 2 : 0) + (count > 1 ? 1 : 0)];
  if (conv) count_form(ctx, p.conv.on == CONV_GATHER ? QCFG_FORM_CONV_GATHER : !slab ? QCFG_FORM_CONV_IM2COL : sd.resident ? QCFG_FORM_CONV_SLAB : QCFG_FORM_CONV_STREAMED);
  if (shortcut) count_form(ctx, QCFG_FORM_SHORTCUT);
  if (rows_out) count_form(ctx, QCFG_FORM_ROWS);
  for (int i = 0; i < count; ++i) if (p.grp[i].mode == EPI_Y32) count_form(ctx, QCFG_FORM_NARROW_FP32);
  p.stamp = prof_stamp(ctx, g0.is_bf16 ? 1 : 0, ops);
  static thread_local LaunchArgs<false> one;
  memcpy(one.rec[0].m, maps, sizeof(maps));
  one.rec[0].p = p;
  one.n = 1; one.total_tiles = num_tiles; one.flag_stride = 0; one.flags = nullptr;
  prof_begin(ctx, g0.is_bf16 ? 1 : 0, st);
  cudaError_t le = make_ready(cs, (const void*)kern);
  if (le == cudaSuccess) le = cudaLaunchKernelEx(&cfg, kern, one);
  prof_end(ctx, g0.is_bf16 ? 1 : 0, ops, st);
  if (le != cudaSuccess) return check_cuda(ctx, le, "gemm launch");
  count_launch(ctx);
  return check_cuda(ctx, cudaGetLastError(), "gemm launch");
}

int launch_gemm(Ctx* ctx, const GemmArgs& g, cudaStream_t st) { return launch_gemm_group(ctx, &g, 1, st); }

}  // namespace qcfg
