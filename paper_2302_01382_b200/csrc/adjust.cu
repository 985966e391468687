// Kernels of the scale-adjustment step (Section 3.1, second step of the scale estimation: the
// quantization scales are adapted by backpropagation while the model's parameters stay fixed).
// The two backward GEMMs of a layer run on the tensor-core kernel of gemm.cu with bf16 operands;
// what is here is the element-wise and reduction work around them: activation forward and
// derivative, the loss gradient, the straight-through derivative of the quantizer (1 inside the
// clip range, 0 outside), the reductions that give the gradient of each scale, and the update.
#include "common.cuh"

namespace qcfg {

namespace {

__device__ __forceinline__ float act_forward(float y, int act) {
  if (act == QCFG_ACT_RELU) return fmaxf(y, 0.0f);
  if (act == QCFG_ACT_GELU_TANH) return gelu_tanh(y);
  return y;
}
// derivative of the activation at y
__device__ __forceinline__ float act_derivative(float y, int act) {
  if (act == QCFG_ACT_RELU) return y > 0.0f ? 1.0f : 0.0f;
  if (act == QCFG_ACT_GELU_TANH) {
    const float c = 0.7978845608028654f, a = 0.044715f;
    const float u = c * (y + a * y * y * y);
    const float sig = 1.0f / (1.0f + __expf(-2.0f * u));
    return sig + y * sig * (1.0f - sig) * 2.0f * c * (1.0f + 3.0f * a * y * y);
  }
  return 1.0f;
}

// Four consecutive elements per thread; VEC: whole aligned groups of four in every row.
template <bool VEC>
__global__ void __launch_bounds__(256) act_apply_kernel(const float* __restrict__ ylin, const float* __restrict__ res,
                                                        int64_t ldr, int act, float* __restrict__ y, int64_t rows, int64_t n) {
  pdl_entry();
  const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 4;
  if (i >= rows * n) return;
  if (VEC) {
    float4 v = __ldg(reinterpret_cast<const float4*>(ylin + i));
    if (res) {
      const int64_t r = i / n;
      const float4 a = __ldg(reinterpret_cast<const float4*>(res + r * ldr + (i - r * n)));
      v.x = __fadd_rn(v.x, a.x); v.y = __fadd_rn(v.y, a.y); v.z = __fadd_rn(v.z, a.z); v.w = __fadd_rn(v.w, a.w);
    }
    *reinterpret_cast<float4*>(y + i) = make_float4(act_forward(v.x, act), act_forward(v.y, act), act_forward(v.z, act), act_forward(v.w, act));
  } else {
    for (int64_t e = i; e < i + 4 && e < rows * n; ++e) {
      float v = ylin[e];
      if (res) { const int64_t r = e / n; v = __fadd_rn(v, res[r * ldr + (e - r * n)]); }
      y[e] = act_forward(v, act);
    }
  }
}

// Everything a layer's backward products need from dL/d(output), in one pass over it: the gradient behind
// the activation g = gout * act'(ylin + res) (or, for the last layer, gout = coef * (y - yref) formed
// here), its column-scaled bf16 operand gs = bf16(g * s_w[c]), its transposed bf16 operand
// gt = bf16(g)^T, and the column sums of g * ylin.  As five kernels (loss or activation gradient,
// column reduction, operand, transpose) the same took 130 us for 3072 x 3072, four reads and three
// writes of the matrix; one read of two matrices and two bf16 writes take 23 us.
// One block per 64 columns and a strip of 64-row tiles; a thread owns 4 columns x every 16th row, so its
// column sums stay in registers until the end of the strip; the tile is turned in shared memory.
// Reads of gout and ylin, coefficients and sums are those of the separate steps, bit for bit.
constexpr int kTile = 64;
__device__ __forceinline__ uint4 turned8(const uint32_t* p) { return make_uint4(p[0], p[1], p[2], p[3]); }
template <bool VEC>
__global__ void __launch_bounds__(256) backward_operands_kernel(
    float* __restrict__ gout, const float* __restrict__ y, const float* __restrict__ yref, const float* __restrict__ coef_dev,
    const float* __restrict__ ylin, const float* __restrict__ res, int64_t ldr, int act, const float* __restrict__ s_w, int64_t rows, int64_t n, int keep_g,
    __nv_bfloat16* __restrict__ gs, int64_t ld_gs, __nv_bfloat16* __restrict__ gt, int64_t ld_gt, double* __restrict__ colsum,
    int tiles_per_block) {
  pdl_entry();
  __shared__ uint32_t turn[kTile][kTile / 2 + 1];          // [column][row], bf16 pairs; the odd pitch keeps both directions off each other's banks
  __shared__ double csum[16][kTile + 1];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int64_t c0 = (int64_t)blockIdx.x * kTile + 4 * tx;
  double part[4] = {0.0, 0.0, 0.0, 0.0};
  const float coef = yref ? *coef_dev : 0.0f;
  float sw[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) sw[j] = s_w && c0 + j < n ? s_w[c0 + j] : 1.0f;
  for (int t = 0; t < tiles_per_block; ++t) {
    const int64_t r0 = ((int64_t)blockIdx.y * tiles_per_block + t) * kTile;
    if (r0 >= (gt ? ld_gt : rows)) break;                 // uniform over the block
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const int rl = ty + 16 * p;
      const int64_t r = r0 + rl;
      float g[4] = {0.0f, 0.0f, 0.0f, 0.0f}, yl[4] = {0.0f, 0.0f, 0.0f, 0.0f}, pre[4];
      if (r < rows && c0 < n) {
        const int64_t at = r * n + c0;
        if (VEC) {
          const float4 v = *reinterpret_cast<const float4*>(ylin + at);
          yl[0] = v.x; yl[1] = v.y; yl[2] = v.z; yl[3] = v.w;
          if (yref) {
            const float4 a = *reinterpret_cast<const float4*>(y + at), b = *reinterpret_cast<const float4*>(yref + at);
            g[0] = coef * (a.x - b.x); g[1] = coef * (a.y - b.y); g[2] = coef * (a.z - b.z); g[3] = coef * (a.w - b.w);
          } else {
            const float4 a = *reinterpret_cast<const float4*>(gout + at);
            g[0] = a.x; g[1] = a.y; g[2] = a.z; g[3] = a.w;
          }
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (c0 + j < n) { yl[j] = ylin[at + j]; g[j] = yref ? coef * (y[at + j] - yref[at + j]) : gout[at + j]; }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          pre[j] = yl[j];
          if (res && c0 + j < n) pre[j] = __fadd_rn(pre[j], res[r * ldr + c0 + j]);
          g[j] *= act_derivative(pre[j], act);
          part[j] += (double)g[j] * (double)yl[j];
          if (keep_g && c0 + j < n) gout[at + j] = g[j];
        }
      }
      if (gs && r < rows && c0 < ld_gs) {                 // ld_gs is a multiple of 8: whole groups of four
        __nv_bfloat162 lo = __floats2bfloat162_rn(s_w ? g[0] * sw[0] : g[0], s_w ? g[1] * sw[1] : g[1]);
        __nv_bfloat162 hi = __floats2bfloat162_rn(s_w ? g[2] * sw[2] : g[2], s_w ? g[3] * sw[3] : g[3]);
        *reinterpret_cast<uint2*>(gs + r * ld_gs + c0) = make_uint2(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi));
      }
      if (gt) {
#pragma unroll
        for (int j = 0; j < 4; ++j) reinterpret_cast<__nv_bfloat16*>(turn[4 * tx + j])[rl] = __float2bfloat16_rn(g[j]);
      }
    }
    if (gt) {
      __syncthreads();
      const int c = threadIdx.x >> 2, q = (threadIdx.x & 3) * 16;      // one column, 16 rows
      const int64_t col = (int64_t)blockIdx.x * kTile + c;
      if (col < n) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
          if (r0 + q + 8 * h < ld_gt)                     // ld_gt is a multiple of 8; columns rows..ld_gt-1 get zeros
            *reinterpret_cast<uint4*>(gt + col * ld_gt + r0 + q + 8 * h) = turned8(turn[c] + (q + 8 * h) / 2);
      }
      __syncthreads();
    }
  }
  if (colsum) {
#pragma unroll
    for (int j = 0; j < 4; ++j) csum[ty][4 * tx + j] = part[j];
    __syncthreads();
    if (threadIdx.x < kTile && (int64_t)blockIdx.x * kTile + threadIdx.x < n) {
      double v = csum[0][threadIdx.x];
#pragma unroll
      for (int k = 1; k < 16; ++k) v += csum[k][threadIdx.x];
      atomicAdd(colsum + (int64_t)blockIdx.x * kTile + threadIdx.x, v);
    }
  }
}

// *coef = 2 / sum of the reference's squares, from the per-block partial sums {difference, reference} of the
// loss; 0 for an all-zero reference (the call then ends with an error)
__global__ void __launch_bounds__(256) loss_coef_kernel(const double* __restrict__ partial, int blocks, float* __restrict__ coef) {
  pdl_entry();
  double v = 0.0;
  for (int i = threadIdx.x; i < blocks; i += 256) v += partial[2 * i + 1];
  v = warp_sum(v);
  __shared__ double sm[8];
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) v += sm[w];
    *coef = v > 0.0 ? (float)(2.0 / v) : 0.0f;
  }
}

__global__ void __launch_bounds__(256) gamma_finish_kernel(const double* __restrict__ colsum, const float* __restrict__ s_w,
                                                           float s_x, int64_t n, double* __restrict__ d_sw, double* __restrict__ d_sx) {
  pdl_entry();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  double v = 0.0;
  if (i < n) {
    d_sw[i] = colsum[i] / (double)s_w[i];
    v = colsum[i] / (double)s_x;
  }
  v = warp_sum(v);
  if ((threadIdx.x & 31) == 0 && v != 0.0) atomicAdd(d_sx, v);
}

// dst[c][r] = bf16(src[r][c]): 64 x 64 tiles turned in shared memory, 16-byte reads and writes; dst columns
// beyond `rows` get zero.  src rows start on 16 bytes (ld_src * sizeof(T) is a multiple of 16).
template <typename T>
__global__ void __launch_bounds__(256) transpose_bf16_kernel(const T* __restrict__ src, int64_t rows, int64_t cols, int64_t ld_src,
                                                             __nv_bfloat16* __restrict__ dst, int64_t ld_dst) {
  pdl_entry();
  __shared__ uint32_t turn[kTile][kTile / 2 + 1];
  const int64_t r0 = (int64_t)blockIdx.x * kTile, c0 = (int64_t)blockIdx.y * kTile;
  {
    const int rl = threadIdx.x >> 2, q = (threadIdx.x & 3) * 16;       // one row, 16 columns
    const int64_t r = r0 + rl, c = c0 + q;
    __nv_bfloat16 v[16];
    constexpr int kPer = 16 / (int)sizeof(T);                          // elements per 16-byte load
#pragma unroll
    for (int h = 0; h < 16 / kPer; ++h) {
      uint4 raw = make_uint4(0, 0, 0, 0);
      if (r < rows && c + h * kPer < ld_src) raw = __ldg(reinterpret_cast<const uint4*>(src + r * ld_src + c) + h);
      const T* e = reinterpret_cast<const T*>(&raw);
#pragma unroll
      for (int k = 0; k < kPer; ++k) {
        if (sizeof(T) == 1) v[h * kPer + k] = __float2bfloat16_rn((float)e[k]);
        else v[h * kPer + k] = *reinterpret_cast<const __nv_bfloat16*>(&e[k]);
      }
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) reinterpret_cast<__nv_bfloat16*>(turn[q + k])[rl] = v[k];
  }
  __syncthreads();
  const int cl = threadIdx.x >> 2, q = (threadIdx.x & 3) * 16;
  if (c0 + cl >= cols) return;
#pragma unroll
  for (int h = 0; h < 2; ++h)
    if (r0 + q + 8 * h < ld_dst)
      *reinterpret_cast<uint4*>(dst + (c0 + cl) * ld_dst + r0 + q + 8 * h) = turned8(turn[cl] + (q + 8 * h) / 2);
}

// One warp per run of 128 columns of a row, rows strided over the grid: no division per element.
// assign: gprod has no earlier contribution yet.
template <bool VEC>
__global__ void __launch_bounds__(256) input_backward_kernel(const float* __restrict__ dxq, const float* __restrict__ x, int64_t ldx,
                                                             float s_x, float inv_x, float qmax, int64_t rows, int64_t k,
                                                             float* __restrict__ gprod, int64_t ldg, int assign, double* __restrict__ d_ix) {
  pdl_entry();
  double part = 0.0;
  const float pass = __fmul_rn(s_x, inv_x);
  const int lane = threadIdx.x & 31;
  const int64_t c = ((int64_t)blockIdx.x * 32 + lane) * 4;
  for (int64_t r = (int64_t)blockIdx.y * 8 + (threadIdx.x >> 5); r < rows; r += (int64_t)gridDim.y * 8) {
    if (c >= k) break;
    float d[4] = {0.0f, 0.0f, 0.0f, 0.0f}, xv[4] = {0.0f, 0.0f, 0.0f, 0.0f}, o[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    float* gp = gprod ? gprod + r * ldg + c : nullptr;
    if (VEC) {
      const float4 a = __ldg(reinterpret_cast<const float4*>(dxq + r * k + c));
      d[0] = a.x; d[1] = a.y; d[2] = a.z; d[3] = a.w;
      if (qmax != 0.0f) {
        const float4 b = __ldg(reinterpret_cast<const float4*>(x + r * ldx + c));
        xv[0] = b.x; xv[1] = b.y; xv[2] = b.z; xv[3] = b.w;
      }
      if (gp && !assign) { const float4 b = *reinterpret_cast<const float4*>(gp); o[0] = b.x; o[1] = b.y; o[2] = b.z; o[3] = b.w; }
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (c + j < k) {
          d[j] = __ldg(dxq + r * k + c + j);
          if (qmax != 0.0f) xv[j] = __ldg(x + r * ldx + c + j);
          if (gp && !assign) o[j] = gp[j];
        }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (qmax == 0.0f) { o[j] += d[j]; continue; }               // 16-bit layer: rounding passed through
      if (fabsf(__fmul_rn(xv[j], inv_x)) <= qmax) {               // derivative of the clip
        part += (double)d[j] * (double)xv[j];
        o[j] += d[j] * pass;
      }
    }
    if (gp) {
      if (VEC) *reinterpret_cast<float4*>(gp) = make_float4(o[0], o[1], o[2], o[3]);
      else {
#pragma unroll
        for (int j = 0; j < 4; ++j) if (c + j < k) gp[j] = o[j];
      }
    }
  }
  if (!d_ix) return;
  part = warp_sum(part);
  __shared__ double sm[8];
  if (lane == 0) sm[threadIdx.x >> 5] = part;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int w = 0; w < 8; ++w) v += sm[w];
    if (v != 0.0) atomicAdd(d_ix, v * (double)s_x);
  }
}

// One block per weight row.  The gradient of the codes comes as PARTS partial sums (a reduction cut into
// equal pieces, one after the other in memory), added here in double.  Four columns per load and all parts'
// loads issued together: a warp per row with single loads took 40 us for 768 x 3072, this 9 us.
template <bool VEC, int PARTS>
__global__ void __launch_bounds__(256) weight_alpha_kernel(const float* __restrict__ dwq, const float* __restrict__ w,
                                                           const float* __restrict__ s_w, const float* __restrict__ inv_w, float s_x,
                                                           float qmax, int64_t n, int64_t k, double* __restrict__ d_iw) {
  pdl_entry();
  const int64_t row = blockIdx.x;
  const float iw = inv_w[row];
  const float* wr = w + row * k;
  const float* dr = dwq + row * k;
  double v = 0.0;
  auto term = [&](float wv, const float (&d)[PARTS]) {
    if (fabsf(__fmul_rn(wv, iw)) <= qmax) {
      double s = (double)d[0];
#pragma unroll
      for (int p = 1; p < PARTS; ++p) s += (double)d[p];
      v += s * (double)wv;
    }
  };
  if (VEC) {
#pragma unroll 2
    for (int64_t c = threadIdx.x; c < (k >> 2); c += 256) {
      const float4 wv = __ldg(reinterpret_cast<const float4*>(wr) + c);
      float4 q[PARTS];
#pragma unroll
      for (int p = 0; p < PARTS; ++p) q[p] = __ldg(reinterpret_cast<const float4*>(dr + p * n * k) + c);
      float d[4][PARTS];
#pragma unroll
      for (int p = 0; p < PARTS; ++p) { d[0][p] = q[p].x; d[1][p] = q[p].y; d[2][p] = q[p].z; d[3][p] = q[p].w; }
      term(wv.x, d[0]); term(wv.y, d[1]); term(wv.z, d[2]); term(wv.w, d[3]);
    }
  } else {
    for (int64_t c = threadIdx.x; c < k; c += 256) {
      float d[PARTS];
#pragma unroll
      for (int p = 0; p < PARTS; ++p) d[p] = __ldg(dr + p * n * k + c);
      term(__ldg(wr + c), d);
    }
  }
  v = warp_sum(v);
  __shared__ double sm[8];
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < 8; ++i) v += sm[i];
    d_iw[row] = v * (double)s_x * (double)s_w[row];
  }
}

__global__ void __launch_bounds__(256) sgd_kernel(float* __restrict__ s, const double* __restrict__ g, double lr, int64_t n) {
  pdl_entry();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) s[i] = (float)__dsub_rn((double)s[i], __dmul_rn(lr, g[i]));     // two roundings, as written
}

inline unsigned blocks_for(int64_t count) { return (unsigned)((count + 255) / 256); }

}  // namespace

static inline bool vec4(const void* p, int64_t n, int64_t ld) { return !p || ((uintptr_t)p % 16 == 0 && n % 4 == 0 && ld % 4 == 0); }

int launch_act_apply(Ctx* ctx, const float* ylin, const float* res, int64_t ldr, int act, float* y, int64_t rows, int64_t n, cudaStream_t st) {
  if (rows * n == 0) return QCFG_OK;
  const unsigned blocks = blocks_for((rows * n + 3) / 4);
  if (vec4(ylin, n, n) && vec4(res, n, ldr) && vec4(y, n, n)) launch_pdl(act_apply_kernel<true>, dim3(blocks), dim3(256), 0, st, ylin, res, ldr, act, y, rows, n);
  else launch_pdl(act_apply_kernel<false>, dim3(blocks), dim3(256), 0, st, ylin, res, ldr, act, y, rows, n);
  count_launch(ctx);
  return check_cuda(ctx, cudaGetLastError(), "activation launch");
}
int launch_backward_operands(Ctx* ctx, float* gout, const float* y, const float* yref, const float* coef, const float* ylin,
                             const float* res, int64_t ldr, int act, const float* s_w, int64_t rows, int64_t n, bool keep_g, void* gs, int64_t ld_gs,
                             void* gt, int64_t ld_gt, double* colsum, cudaStream_t st) {
  if (rows * n == 0) return QCFG_OK;
  const int64_t bx = ((gs && ld_gs > n ? ld_gs : n) + kTile - 1) / kTile;
  const int64_t tiles = ((gt ? ld_gt : rows) + kTile - 1) / kTile;
  // four blocks per SM, or one tile each; a strip ends with one atomic add per column
  int64_t per = (tiles * bx + (int64_t)sm_count(ctx) * 4 - 1) / ((int64_t)sm_count(ctx) * 4);
  if (per < 1) per = 1;
  if (per < (tiles + 65534) / 65535) per = (tiles + 65534) / 65535;
  const dim3 grid((unsigned)bx, (unsigned)((tiles + per - 1) / per));
  __nv_bfloat16* s16 = reinterpret_cast<__nv_bfloat16*>(gs);
  __nv_bfloat16* t16 = reinterpret_cast<__nv_bfloat16*>(gt);
  if (vec4(gout, n, n) && vec4(y, n, n) && vec4(yref, n, n) && vec4(ylin, n, n))
    launch_pdl(backward_operands_kernel<true>, dim3(grid), dim3(256), 0, st, gout, y, yref, coef, ylin, res, ldr, act, s_w, rows, n, keep_g, s16, ld_gs, t16, ld_gt, colsum, (int)per);
  else
    launch_pdl(backward_operands_kernel<false>, dim3(grid), dim3(256), 0, st, gout, y, yref, coef, ylin, res, ldr, act, s_w, rows, n, keep_g, s16, ld_gs, t16, ld_gt, colsum, (int)per);
  count_launch(ctx);
  return check_cuda(ctx, cudaGetLastError(), "backward operand launch");
}
int launch_loss_coef(Ctx* ctx, const double* partial, int blocks, float* coef, cudaStream_t st) {
  launch_pdl(loss_coef_kernel, dim3(1), dim3(256), 0, st, partial, blocks, coef);
  count_launch(ctx);
  return check_cuda(ctx, cudaGetLastError(), "loss coefficient launch");
}
int launch_gamma_finish(Ctx* ctx, const double* colsum, const float* s_w, float s_x, int64_t n, double* d_sw, double* d_sx, cudaStream_t st) {
  if (n == 0) return QCFG_OK;
  launch_pdl(gamma_finish_kernel, dim3(blocks_for(n)), dim3(256), 0, st, colsum, s_w, s_x, n, d_sw, d_sx);
  count_launch(ctx);
  return check_cuda(ctx, cudaGetLastError(), "scale gradient launch");
}
int launch_transpose_bf16(Ctx* ctx, const void* src, int kind, int64_t rows, int64_t cols, int64_t ld_src, void* dst, int64_t ld_dst, cudaStream_t st) {
  if (cols == 0 || ld_dst == 0) return QCFG_OK;
  const dim3 grid((unsigned)((ld_dst + kTile - 1) / kTile), (unsigned)((cols + kTile - 1) / kTile));
  __nv_bfloat16* d = reinterpret_cast<__nv_bfloat16*>(dst);
  if (kind == 1) launch_pdl(transpose_bf16_kernel<int8_t>, dim3(grid), dim3(256), 0, st, reinterpret_cast<const int8_t*>(src), rows, cols, ld_src, d, ld_dst);
  else launch_pdl(transpose_bf16_kernel<__nv_bfloat16>, dim3(grid), dim3(256), 0, st, reinterpret_cast<const __nv_bfloat16*>(src), rows, cols, ld_src, d, ld_dst);
  count_launch(ctx);
  return check_cuda(ctx, cudaGetLastError(), "transpose launch");
}
int launch_input_backward(Ctx* ctx, const float* dxq, const float* x, int64_t ldx, float s_x, float inv_x, float qmax,
                          int64_t rows, int64_t k, float* gprod, int64_t ldg, bool assign, double* d_ix, cudaStream_t st) {
  if (rows * k == 0) return QCFG_OK;
  const int64_t bx = (k + 127) / 128;
  int64_t by = ((int64_t)sm_count(ctx) * 8 + bx - 1) / bx;
  if (by > (rows + 7) / 8) by = (rows + 7) / 8;
  const dim3 grid((unsigned)bx, (unsigned)by);
  if (vec4(dxq, k, k) && vec4(x, k, ldx) && vec4(gprod, k, ldg))
    launch_pdl(input_backward_kernel<true>, dim3(grid), dim3(256), 0, st, dxq, x, ldx, s_x, inv_x, qmax, rows, k, gprod, ldg, assign, d_ix);
  else
    launch_pdl(input_backward_kernel<false>, dim3(grid), dim3(256), 0, st, dxq, x, ldx, s_x, inv_x, qmax, rows, k, gprod, ldg, assign, d_ix);
  count_launch(ctx);
  return check_cuda(ctx, cudaGetLastError(), "input backward launch");
}
int launch_weight_alpha(Ctx* ctx, const float* dwq, int parts, const float* w, const float* s_w, const float* inv_w, float s_x, float qmax,
                        int64_t n, int64_t k, double* d_iw, cudaStream_t st) {
  if (n == 0) return QCFG_OK;
  const bool v4 = vec4(dwq, k, k) && vec4(w, k, k);
  using Kern = void (*)(const float*, const float*, const float*, const float*, float, float, int64_t, int64_t, double*);
  const Kern kern = parts == 1 ? (v4 ? weight_alpha_kernel<true, 1> : weight_alpha_kernel<false, 1>)
                               : (v4 ? weight_alpha_kernel<true, 3> : weight_alpha_kernel<false, 3>);
  launch_pdl(kern, dim3((unsigned)n), dim3(256), 0, st, dwq, w, s_w, inv_w, s_x, qmax, n, k, d_iw);
  count_launch(ctx);
  return check_cuda(ctx, cudaGetLastError(), "weight scale gradient launch");
}
int launch_sgd(Ctx* ctx, float* s, const double* g, double lr, int64_t n, cudaStream_t st) {
  if (n == 0) return QCFG_OK;
  launch_pdl(sgd_kernel, dim3(blocks_for(n)), dim3(256), 0, st, s, g, lr, n);
  count_launch(ctx);
  return check_cuda(ctx, cudaGetLastError(), "scale update launch");
}

}  // namespace qcfg
