// Implicit neural decoder g(X; xhat) (Section 3.1, Eq. kinematicRestriction;
// Section 4, Table 1) with its Jacobians (Eq. defGrad: dg/dX; Eq. timederOne:
// dg/dxhat) on sm_103a tensor cores.
//
// Network: h0 = act(W0 [Xn, xhat] + b0), h_l = act(W_l h_{l-1} + b_l) for the
// square hidden layers, y = Wout h + bout, g = out_scale * y + out_shift,
// Xn = (X - X_min) / X_range (min-max input scaling and output
// standardisation of Appendix B), act = ELU.
//
// Derivatives are propagated forward as extra rows of the same GEMMs: every
// point contributes R rows to a 128-row tile (kind-major: rows kind*Pt + q),
//   kind 0          primal              h = act(z)
//   tangent kinds   dg along an input direction   t = act'(z) . (W t_prev)
//   secant kind     g(xhat + delta) - g(xhat)     s = act(z + W s_prev) - act(z)
//   mixed kinds     d/d(input b) of the JVP row   m = act''(z) (W u)(W t) + act'(z) (W m_prev)
// where z is the primal pre-activation of the same point and, for a mixed row,
// W u and W t are the pre-activations of the JVP row and of the input-b tangent
// row of the same point; the pre-activations of a 32-column chunk are
// exchanged between the rows of a tile through shared memory.  The secant rows give differences of decoder outputs without
// the BF16 rounding of the two absolute evaluations (the Gauss-Newton
// residual needs differences far below BF16 resolution).
//
// This describes decoder_tc, the general kernel (mixed rows, r > 28, split BF16);
// decoder_bf16 and decoder_tc3 take the other BF16 and FP32 calls with rows in
// (point, kind) order, decoder_f32 the FP32 calls left (see each kernel).
//
// Per tile: layer 0 (K = d + r <= 35) and the output layer (N = d) run in
// FP32 on the CUDA cores; each square 128 x 128 layer is one M=128, N=128,
// K=128 tcgen05.mma chain (BF16 operands from shared memory in the 128-byte
// swizzled K-major layout, FP32 accumulator in tensor memory), read back with
// tcgen05.ld for the bias/activation/tangent epilogue, which writes the next
// layer's BF16 operand tile in place.  All square-layer weights stay resident
// in shared memory (loaded once per CTA with bulk async copies); the kernel
// is persistent over tiles.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <string>
#include <vector>

#include "common.cuh"
#include "tc.cuh"

#include "decoder_common.cuh"
#include "pipe.cuh"

namespace mpmrom {

// --------------------------------------------------------------------------
// Decoders without square layers (linear, or a single hidden layer): SIMT.
// --------------------------------------------------------------------------
__global__ void decoder_simt(DecArgs a) {
  const int64_t n = dec_count(a);
  const int64_t rows = n * a.R;
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < rows; g += (int64_t)gridDim.x * blockDim.x) {
    const int k = (int)(g / n);
    RowInfo ri;
    ri.p = g % n;
    ri.q = 0;
    ri.kind = a.kinds[k];
    ri.cls = kind_class(ri.kind);
    float in[40], dir[40];
    row_inputs(a, ri, in, dir);
    const int K = a.d + a.r;
    float y[3] = {0.f, 0.f, 0.f};
    if (a.linear) {
      // an affine map has no mixed second derivative
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        if (i >= a.d) break;
        float z = 0.f;
        if (ri.cls != 3)
          for (int c = 0; c < K; ++c) z = fmaf(a.W0[i * K + c], ri.cls == 0 ? in[c] : dir[c], z);
        y[i] = z + (ri.cls == 0 ? a.b0[i] : 0.f);
      }
    } else {
      for (int c = 0; c < kW; ++c) {
        float z = a.b0[c], zd = 0.f;
        for (int i = 0; i < K; ++i) {
          z = fmaf(a.W0[c * K + i], in[i], z);
          zd = fmaf(a.W0[c * K + i], dir[i], zd);
        }
        float h;
        if (ri.cls == 0) h = act_f(a.act, z);
        else if (ri.cls == 1) h = act_d1(a.act, z) * zd;
        else if (ri.cls == 2) h = act_sec(a.act, z, zd);
        else h = act_d2(a.act, z) * zd * mixed_t0(a, a.W0 + c * K, ri.kind);
#pragma unroll
        for (int i = 0; i < 3; ++i)
          if (i < a.d) y[i] = fmaf(a.Wout[i * kW + c], h, y[i]);
      }
      if (ri.cls == 0)
#pragma unroll
        for (int i = 0; i < 3; ++i)
          if (i < a.d) y[i] += a.bout[i];
    }
    float* o = a.out + ((int64_t)k * a.n + ri.p) * a.d;   // kind stride = capacity a.n
#pragma unroll
    for (int i = 0; i < 3; ++i)
      if (i < a.d) o[i] = y[i] * a.norm[3 * a.d + i] + (ri.cls == 0 ? a.norm[2 * a.d + i] : 0.f);
  }
}

// --------------------------------------------------------------------------
// Tensor-core decoder kernel: 256 threads.  Warps w and w + 4 read the same
// tensor-memory lane group (lanes 32 (w % 4) ..): thread t owns tile row
// rw = 32 (w % 4) + lane and the column half h = w / 4 (columns 64 h .. 64 h + 63)
// of every layer, so each row's epilogue is split over two warps.
// --------------------------------------------------------------------------
constexpr int kDecThreads = 256;
constexpr int kXbStride = 33;                            // padded row stride of the exchange
constexpr int kW0Stride = 40;                            // first-layer row stride (d + r <= 40)

__device__ __forceinline__ float elu_bf16_input(float z) {
  // ELU whose result feeds a BF16 operand (or the FP32 output layer): exp(z) - 1
  // with the fast exponential; its absolute error (~1e-7) is far below BF16
  // resolution of the activations
  return z > 0.f ? z : __expf(z) - 1.0f;
}

// The operand tile of the next square layer: BF16, or (split) the BF16 pair hi = bf16(v),
// lo = bf16(v - hi) in two tiles kLayerBytes apart.
template <bool SPLIT>
__device__ __forceinline__ void store_operand(uint8_t* tile, int row, int col, const float* v) {
  if (!SPLIT) {
    store_bf16x8(tile, row, col, v);
  } else {
    float hi[8], lo[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      hi[i] = __bfloat162float(__float2bfloat16_rn(v[i]));
      lo[i] = v[i] - hi[i];   // exact in FP32
    }
    store_bf16x8(tile, row, col, hi);
    store_bf16x8(tile + kLayerBytes, row, col, lo);
  }
}

// SPLIT = false: BF16 operands, all square layers resident in shared memory.
// SPLIT = true: FP32-accurate square layers from split BF16 operands (hi + lo for the
// activations and the weights), three MMAs per K step into the same FP32 accumulator,
//   A W ~ A_hi W_hi + A_hi W_lo + A_lo W_hi,
// the dropped A_lo W_lo term and the residuals of the splits being about 2^-16 of each product;
// the two weight images of one layer at a time are streamed into shared memory while the
// previous layer's epilogue runs, and the activations take the accurate exponential.
// TRAIN (not with SPLIT): the activations of every layer and the primal rows' slopes are stored.  A variant
// of its own: with the stores behind a runtime test the evaluations were 5 to 8 % slower (20,000 points x 12
// rows with secants, r = 32: 1.14 -> 1.05 ms; split BF16, r = 16: 1.35 -> 1.28).
template <bool SPLIT, bool TRAIN>
__global__ void __launch_bounds__(kDecThreads, 1) decoder_tc(DecArgs a) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  // 1024-byte alignment for the swizzled operand tiles
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* wsm = smem;                                   // n_tc x 32 KB (split: the current layer, hi and lo)
  uint8_t* atile = smem + (SPLIT ? 2 : kMaxTC) * kLayerBytes;  // 32 KB (split: hi and lo, 64 KB)
  // first layer: FP32 [128][kW0Stride], zero-padded (CUDA cores), or its 16 KB split BF16 image
  uint8_t* w0s = atile + (SPLIT ? 2 : 1) * kLayerBytes;
  float* sW0 = (float*)w0s;
  float* xb = sW0 + kW * kW0Stride;                      // [2 halves][128 rows][33]: one chunk per half
  float* ypart = xb + 2 * 128 * kXbStride;               // [128 rows][3]: output partial of half 1
  float* sb0 = ypart + 128 * 3;                          // [128]
  float* sbh = sb0 + kW;                                 // [kMaxTC][128] square-layer biases
  float* sWout = sbh + kMaxTC * kW;                      // [3][128] output layer
  DecSmemTail* tail = (DecSmemTail*)(sWout + 3 * kW);
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int rw = (warp & 3) * 32 + lane;                 // tile row / tensor-memory lane
  const int h = warp >> 2;                               // column half

  if (t == 0) {
    tc::mbar_init(&tail->bar_w, 1);
    tc::mbar_init(&tail->bar_mma, 1);
    tail->abort = 0;
    tc::fence_mbar_init();
  }
  if (warp == 0) tc::tmem_alloc<kW>(&tail->tmem);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = tail->tmem;

  // The first layer runs on the tensor cores when its inputs fit 32 entries of the padded layout:
  // z = W0 [in] from split BF16 pairs, in_hi W0_hi + in_hi W0_lo + in_lo W0_hi (FP32 accumulate),
  // the dropped products and the residuals of the splits about 2^-16 of each product.
  const int K0 = kTcLat + a.r;                           // first-layer inputs in the padded layout
  const bool l0_tc = !SPLIT && a.w0img != nullptr && K0 <= 32;

  // FP32 first layer (CUDA-core form), biases and output layer staged in shared memory (read by
  // every row of every tile)
  {
    const int K0s = a.d + a.r;
    // the tensor-core input layout (row_inputs_tc): coordinates at 0 .. 3, latents from kTcLat
    for (int e = t; e < (l0_tc ? 0 : kW * kW0Stride); e += kDecThreads) {
      const int c = e / kW0Stride, ii = e % kW0Stride;
      const int i = ii < kTcLat ? (ii < a.d ? ii : -1) : (ii - kTcLat < a.r ? a.d + ii - kTcLat : -1);
      sW0[e] = i >= 0 ? a.W0[c * K0s + i] : 0.f;
    }
    for (int e = t; e < kW; e += kDecThreads) sb0[e] = a.b0[e];
    for (int e = t; e < a.n_tc * kW; e += kDecThreads) sbh[e] = a.bh[e];
    for (int e = t; e < a.d * kW; e += kDecThreads) sWout[e] = a.Wout[e];
  }
  // resident weights of the square layers; split: the first layer's two images (thread 0 waits
  // for them before its first MMA)
  uint32_t w_phase = 0;
  bool w_pending = false;   // thread 0: a weight copy is in flight
  if (!SPLIT) {
    if (t == 0) {
      tc::mbar_expect_tx(&tail->bar_w, (uint32_t)(a.n_tc * kLayerBytes + (l0_tc ? kLayerBytes / 2 : 0)));
      for (int l = 0; l < a.n_tc; ++l)
        tc::bulk_g2s(wsm + l * kLayerBytes, a.wimg + (size_t)l * kLayerBytes, kLayerBytes, &tail->bar_w);
      if (l0_tc) tc::bulk_g2s(w0s, a.w0img, kLayerBytes / 2, &tail->bar_w);
    }
    if (!tc::mbar_wait(&tail->bar_w, 0)) {
      raise_status(a.status, STATUS_TIMEOUT);
      atomicExch(&tail->abort, 1);
    }
  } else if (t == 0) {
    tc::mbar_expect_tx(&tail->bar_w, (uint32_t)(2 * kLayerBytes));
    tc::bulk_g2s(wsm, a.wimg, kLayerBytes, &tail->bar_w);
    tc::bulk_g2s(wsm + kLayerBytes, a.wimg_lo, kLayerBytes, &tail->bar_w);
    w_pending = true;
  }
  __syncthreads();

  constexpr uint32_t idesc = tc::idesc_bf16_f32(128, kW);
  uint32_t mma_phase = 0;
  const int64_t n_pts = dec_count(a);
  const int64_t n_tiles = (n_pts + a.Pt - 1) / a.Pt;
  float* xh = xb + h * 128 * kXbStride;                  // this half's exchange buffer

  for (int64_t tile = blockIdx.x; tile < n_tiles && !tail->abort; tile += gridDim.x) {
    const int64_t first = tile * a.Pt;
    const RowInfo ri = row_info(a, rw, first, n_pts);
    float in[40], dir[40];
    if (ri.cls >= 0) row_inputs_tc(a, ri, in, dir);

    if (l0_tc) {
      // ---- the first layer's operand row: the primal rows' input, the tangent and secant rows'
      // direction (their pre-activation tangent or increment), zero for the mixed rows (the first
      // layer is linear: their second-order part starts at zero) and the unused rows; half 0
      // stores the high parts at columns 0 .. 31, half 1 the low parts at 32 .. 63
#pragma unroll
      for (int c0 = 0; c0 < 32; c0 += 8) {
        float p[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const float v = ri.cls == 0 ? in[c0 + j] : (ri.cls == 1 || ri.cls == 2) ? dir[c0 + j] : 0.f;
          const float hi = __bfloat162float(__float2bfloat16_rn(v));
          p[j] = h == 0 ? hi : v - hi;
        }
        store_bf16x8(atile, rw, 32 * h + c0, p);
      }
    } else
    // ---- layer 0 on the CUDA cores (FP32), this thread's 64 columns, 8 at a time
    for (int c0 = 64 * h; c0 < 64 * h + 64; c0 += 8) {
      // the 8 columns' sums advance together over the inputs (16 independent chains), so that
      // their FMAs and the broadcast weight loads overlap instead of running column by column
      float z[8], zd[8], hv[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        z[j] = sb0[c0 + j];
        zd[j] = 0.f;
      }
      if (ri.cls == 0) {   // primal rows: no directional part
#pragma unroll
        for (int i4 = 0; i4 < kW0Stride / 4; ++i4) {
          if (4 * i4 < K0) {   // padded weights are zero, as are in[] and dir[] beyond K0
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const float4 w = *reinterpret_cast<const float4*>(sW0 + (c0 + j) * kW0Stride + 4 * i4);
              z[j] = fmaf(w.x, in[4 * i4 + 0], z[j]);
              z[j] = fmaf(w.y, in[4 * i4 + 1], z[j]);
              z[j] = fmaf(w.z, in[4 * i4 + 2], z[j]);
              z[j] = fmaf(w.w, in[4 * i4 + 3], z[j]);
            }
          }
        }
      } else if (ri.cls > 0) {
#pragma unroll
        for (int i4 = 0; i4 < kW0Stride / 4; ++i4) {
          if (4 * i4 < K0) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const float4 w = *reinterpret_cast<const float4*>(sW0 + (c0 + j) * kW0Stride + 4 * i4);
              z[j] = fmaf(w.x, in[4 * i4 + 0], z[j]);
              z[j] = fmaf(w.y, in[4 * i4 + 1], z[j]);
              z[j] = fmaf(w.z, in[4 * i4 + 2], z[j]);
              z[j] = fmaf(w.w, in[4 * i4 + 3], z[j]);
              zd[j] = fmaf(w.x, dir[4 * i4 + 0], zd[j]);
              zd[j] = fmaf(w.y, dir[4 * i4 + 1], zd[j]);
              zd[j] = fmaf(w.z, dir[4 * i4 + 2], zd[j]);
              zd[j] = fmaf(w.w, dir[4 * i4 + 3], zd[j]);
            }
          }
        }
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int c = c0 + j;
        if (ri.cls < 0) hv[j] = 0.f;
        else if (ri.cls == 0) hv[j] = a.act == 0 ? (SPLIT ? elu(z[j]) : elu_bf16_input(z[j])) : z[j];
        else if (ri.cls == 1) hv[j] = act_d1(a.act, z[j]) * zd[j];
        else if (ri.cls == 2) hv[j] = act_sec(a.act, z[j], zd[j]);
        else {
          const int b = ri.kind - KIND_MIXED - 1;   // input of the mixed derivative, padded layout below
          const float t0 = b < a.d ? sW0[c * kW0Stride + b] / a.norm[a.d + b] : sW0[c * kW0Stride + kTcLat + b - a.d];
          hv[j] = act_d2(a.act, z[j]) * zd[j] * t0;
        }
        if (TRAIN && ri.cls == 0)
          a.dstore[(int64_t)c * a.rows_total + tile * 128 + rw] = __float2bfloat16_rn(act_slope_record(a.act, z[j]));
      }
      store_operand<SPLIT>(atile, rw, c0, hv);
    }

    float y[3] = {0.f, 0.f, 0.f};
    // layer -1 is the first layer when it runs on the tensor cores
    for (int l = l0_tc ? -1 : 0; l < a.n_tc; ++l) {
      // make the generic-proxy writes of the operand tile visible to the tensor core
      tc::fence_async_smem();
      tc::tc_fence_before();
      __syncthreads();
      if (t == 0) {
        tc::tc_fence_after();
        bool w_ok = true;
        if (SPLIT && w_pending) {
          w_ok = tc::mbar_wait(&tail->bar_w, w_phase);
          w_phase ^= 1u;
          w_pending = false;
          if (!w_ok) {
            raise_status(a.status, STATUS_TIMEOUT);
            atomicExch(&tail->abort, 1);
          }
        }
        if (w_ok && l < 0) {
          // two K steps of 16 over the 32 padded inputs; hi at byte 0 of a row, lo at byte 64
          const uint32_t a_base = tc::smem_addr(atile), b_base = tc::smem_addr(w0s);
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const uint32_t hi = (uint32_t)(k * 32), lo = (uint32_t)(64 + k * 32);
            tc::mma_bf16(tmem, tc::smem_desc_sw128(a_base + hi), tc::smem_desc_sw128(b_base + hi), idesc,
                         k > 0 ? 1u : 0u);
            tc::mma_bf16(tmem, tc::smem_desc_sw128(a_base + hi), tc::smem_desc_sw128(b_base + lo), idesc, 1u);
            tc::mma_bf16(tmem, tc::smem_desc_sw128(a_base + lo), tc::smem_desc_sw128(b_base + hi), idesc, 1u);
          }
        } else if (w_ok) {
          const uint32_t a_base = tc::smem_addr(atile);
          const uint32_t b_base = tc::smem_addr(wsm + (SPLIT ? 0 : l * kLayerBytes));
#pragma unroll
          for (int k = 0; k < kW / 16; ++k) {
            const uint32_t koff = (uint32_t)((k >> 2) * (kW * 128) + (k & 3) * 32);
            tc::mma_bf16(tmem, tc::smem_desc_sw128(a_base + koff), tc::smem_desc_sw128(b_base + koff), idesc,
                         k > 0 ? 1u : 0u);
            if (SPLIT) {
              tc::mma_bf16(tmem, tc::smem_desc_sw128(a_base + koff),
                           tc::smem_desc_sw128(b_base + kLayerBytes + koff), idesc, 1u);
              tc::mma_bf16(tmem, tc::smem_desc_sw128(a_base + kLayerBytes + koff),
                           tc::smem_desc_sw128(b_base + koff), idesc, 1u);
            }
          }
        }
        tc::mma_commit(&tail->bar_mma);
      }
      // training: the previous layer's activations leave the operand tile while the tensor core
      // reads it (both are reads; the barrier after the wait orders them before the next writes)
      if (TRAIN && l >= 0)
        copy_out_tile(a.astore + (int64_t)l * kW * a.rows_total, a.rows_total, atile, tile, t);
      if (!tc::mbar_wait(&tail->bar_mma, mma_phase)) {
        raise_status(a.status, STATUS_TIMEOUT);
        atomicExch(&tail->abort, 1);
      }
      mma_phase ^= 1u;
      if (SPLIT && t == 0 && a.n_tc > 1 && !tail->abort) {
        // the MMAs have read the buffer: stream the next layer's images (this tile's next layer, or
        // the first layer of the CTA's next tile) while the epilogue runs
        const int nl = (l + 1) % a.n_tc;
        if (l + 1 < a.n_tc || tile + gridDim.x < n_tiles) {
          tc::mbar_expect_tx(&tail->bar_w, (uint32_t)(2 * kLayerBytes));
          tc::bulk_g2s(wsm, a.wimg + (size_t)nl * kLayerBytes, kLayerBytes, &tail->bar_w);
          tc::bulk_g2s(wsm + kLayerBytes, a.wimg_lo + (size_t)nl * kLayerBytes, kLayerBytes, &tail->bar_w);
          w_pending = true;
        }
      }
      tc::tc_fence_after();
      __syncthreads();
      if (tail->abort) break;
      const bool last = (l == a.n_tc - 1);
      const float* bl = l < 0 ? sb0 : sbh + l * kW;
      for (int i2 = 0; i2 < 2; ++i2) {
        const int ch = 2 * h + i2;
        float acc[32];
        tc::tmem_ld32(tmem + ((uint32_t)((warp & 3) * 32) << 16) + ch * 32, acc);
        if (ri.cls == 0) {
#pragma unroll
          for (int i = 0; i < 32; ++i) acc[i] += bl[ch * 32 + i];
        }
        if (a.R > 1) {
          // publish this row's pre-activations of the chunk (stride 33: conflict-free)
#pragma unroll
          for (int i = 0; i < 32; ++i) xh[rw * kXbStride + i] = acc[i];
          __syncthreads();
          // training: the primal rows' activation slopes (the backward's act' and act'' terms), from
          // the published pre-activations, spread over the half's four warps: feature = lane, 8 rows
          // per thread, one 16-byte store of 8 rows of one feature (the training calls have R > 1)
          if (TRAIN) {
            for (int k = warp & 3; 8 * k < a.Pt; k += 4) {
              float v[8];
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                // in place: the primal rows' slopes replace their pre-activations in the exchange
                float* e = xh + (8 * k + j) * kXbStride + lane;
                v[j] = act_slope_record(a.act, *e);
                *e = v[j];
              }
              __nv_bfloat162 p0 = __floats2bfloat162_rn(v[0], v[1]), p1 = __floats2bfloat162_rn(v[2], v[3]);
              __nv_bfloat162 p2 = __floats2bfloat162_rn(v[4], v[5]), p3 = __floats2bfloat162_rn(v[6], v[7]);
              uint4 u;
              u.x = *reinterpret_cast<uint32_t*>(&p0);
              u.y = *reinterpret_cast<uint32_t*>(&p1);
              u.z = *reinterpret_cast<uint32_t*>(&p2);
              u.w = *reinterpret_cast<uint32_t*>(&p3);
              *reinterpret_cast<uint4*>(a.dstore + ((int64_t)(l + 1) * kW + ch * 32 + lane) * a.rows_total +
                                        tile * 128 + 8 * k) = u;
            }
            __syncthreads();
          }
        }
        // the primal row of point q is tile row q (kind index 0)
        const float* zq = xh + ri.q * kXbStride;
        if (TRAIN) {
          // training (primal and tangent rows only): the slope s of the primal row, e^z where z < 0
          // and -1 elsewhere, gives both activations without another exponential: ELU(z) = s - 1
          // (z where s < 0), act'(z) = s (1 where s < 0); the same values as below
          if (ri.cls == 0) {
#pragma unroll
            for (int i = 0; i < 32; ++i) acc[i] = zq[i] < 0.f ? acc[i] : zq[i] - 1.0f;
          } else if (ri.cls == 1) {
#pragma unroll
            for (int i = 0; i < 32; ++i) acc[i] *= zq[i] < 0.f ? 1.0f : zq[i];
          } else {
#pragma unroll
            for (int i = 0; i < 32; ++i) acc[i] = 0.f;
          }
        } else if (ri.cls == 0) {
          if (a.act == 0) {
#pragma unroll
            for (int i = 0; i < 32; ++i) acc[i] = SPLIT ? elu(acc[i]) : elu_bf16_input(acc[i]);
          }
        } else if (ri.cls == 1) {
#pragma unroll
          for (int i = 0; i < 32; ++i) acc[i] *= act_d1(a.act, zq[i]);
        } else if (ri.cls == 2) {
#pragma unroll
          for (int i = 0; i < 32; ++i) acc[i] = act_sec(a.act, zq[i], acc[i]);
        } else if (ri.cls == 3) {
          const float* uq = xh + (ri.ja * a.Pt + ri.q) * kXbStride;
          const float* tq = xh + (ri.jb * a.Pt + ri.q) * kXbStride;
#pragma unroll
          for (int i = 0; i < 32; ++i) acc[i] = act_d2(a.act, zq[i]) * uq[i] * tq[i] + act_d1(a.act, zq[i]) * acc[i];
        } else {
#pragma unroll
          for (int i = 0; i < 32; ++i) acc[i] = 0.f;
        }
        if (last) {
          // output layer fused into the last epilogue (FP32), partial over this half's columns
#pragma unroll
          for (int o = 0; o < 3; ++o) {   // compile-time bound: y stays in registers
            if (o >= a.d) break;
            float sacc = 0.f;
#pragma unroll
            for (int i = 0; i < 32; ++i) sacc = fmaf(sWout[o * kW + ch * 32 + i], acc[i], sacc);
            y[o] += sacc;
          }
        }
        // the next layer's operand tile; in training also the last layer's, for the copy-out
        if (!last || TRAIN) {
#pragma unroll
          for (int j = 0; j < 32; j += 8) store_operand<SPLIT>(atile, rw, ch * 32 + j, acc + j);
        }
        if (a.R > 1) __syncthreads();
      }
      tc::tc_fence_before();
    }
    if (tail->abort) break;
    // combine the two column halves of the output layer
    if (h == 1) {
#pragma unroll
      for (int o = 0; o < 3; ++o)
        if (o < a.d) ypart[rw * 3 + o] = y[o];
    }
    __syncthreads();
    // training: the last layer's activations (the barrier at the end of the tile orders these
    // reads before the next tile's first operand writes)
    if (TRAIN) copy_out_tile(a.astore + (int64_t)a.n_tc * kW * a.rows_total, a.rows_total, atile, tile, t);
    if (h == 0 && ri.cls >= 0) {
      const int kidx = rw / a.Pt;  // position of this row's kind in `kinds`
      float* o = a.out + ((int64_t)kidx * a.n + ri.p) * a.d;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        if (i >= a.d) break;
        float v = y[i] + ypart[rw * 3 + i] + (ri.cls == 0 ? __ldg(&a.bout[i]) : 0.f);
        o[i] = v * a.norm[3 * a.d + i] + (ri.cls == 0 ? a.norm[2 * a.d + i] : 0.f);
      }
    }
    __syncthreads();
  }
  // a weight copy still in flight (an aborted tile loop) lands before the CTA exits
  if (SPLIT && t == 0 && w_pending) (void)tc::mbar_wait(&tail->bar_w, w_phase);
  __syncthreads();
  tc::tc_fence_after();
  if (warp == 0) tc::tmem_free<kW>(tmem);
}

// --------------------------------------------------------------------------
// FP32 decoder on the CUDA cores, for calls whose rows are too few to keep the
// tensor cores busy and whose results need FP32 accuracy (the reduced step's
// positions and gradients).  Same row kinds as decoder_tc; one persistent CTA
// of 512 threads (16 warps) per SM; tiles of TR = 32 or 64 row slots.
// Rows reach the tiles in one of two ways:
//   aligned  (mixed rows present) slot k Pt + q = kind k of point q, Pt = TR / R
//            points per tile, as in decoder_tc;
//   packed   the call's rows in (point, kind) order, U <= TR - 1 per tile,
//            chosen so that the tiles spread over all SMs; slot 0 recomputes
//            the primal row of the tile's first point (its derivative rows may
//            start mid-point) and is not written out.
// Per tile:
//   layer 0       512 / TR threads per row, each 128 TR / 512 columns; inputs
//                 staged in shared memory first
//   square layer  128 x TR x 128 FP32 GEMM from shared memory: TR / 4 warps,
//                 warp w features (512 / TR) w .. + 512 / TR - 1 of every slot,
//                 lane = (slot group of 4, feature group of 4): per k one float4
//                 of activations and one of weights (two or three shared-memory
//                 wavefronts per warp for 16 FMAs per lane); weights
//                 double-buffered from a transposed copy by asynchronous copies;
//                 activations by warps w < TR / 4, slots 4 w .. 4 w + 3
//   exchange      pre-activations to a second buffer (row-major, float4 quads
//                 permuted per row group); derivative rows read the primal
//                 (and, for mixed rows, JVP and tangent) rows' values as float4
//                 of the thread's own 4 features
//   output layer  512 / TR threads per row, interleaved k, shuffle reduction
// Activations (the GEMM's input) are stored feature-major, [f][TR slots], the
// slots in float4 groups permuted per feature (group g of feature f at
// g ^ (f mod TR / 4)) so that the feature-strided stores of a warp spread over
// the banks.  Two barriers per square layer.
// --------------------------------------------------------------------------
constexpr int kF32Threads = 512;
constexpr int kF32Rows = 64;              // largest tile (row slots)
constexpr int kF32In = 41;                // staged input row stride (d + r <= 40)

// ELU for the FP32 path: exp(z) - 1 with the fast exponential (absolute error at the FP32 ulp of
// values near 1, far below the parity tolerance)
__device__ __forceinline__ float act_f32path(int act, float z) {
  return act == 0 ? (z > 0.f ? z : __expf(z) - 1.0f) : z;
}

// Offset of (feature f, slot) in an activation buffer of TR slots.
template <int TR>
__device__ __forceinline__ int f32_slot(int f, int slot) {
  return f * TR + 4 * ((slot >> 2) ^ (f & (TR / 4 - 1))) + (slot & 3);
}

// Offset of the float4 of features f .. f + 3 (f a multiple of 4) of a slot in the row-major
// pre-activation buffer.
__device__ __forceinline__ int f32_zslot(int slot, int f) { return slot * kW + 4 * ((f >> 2) ^ ((slot >> 2) & 7)); }

// Activation of a derivative row from its own pre-activation zo, the primal row's zq and, for a
// mixed row, the JVP row's za and the tangent row's zb (same point, same feature).
__device__ __forceinline__ float f32_deriv_act(int act, int cls, float zo, float zq, float za, float zb) {
  if (cls == 1) return act_d1(act, zq) * zo;
  if (cls == 2) return act_sec(act, zq, zo);
  return act_d2(act, zq) * za * zb + act_d1(act, zq) * zo;
}

// One slot of an FP32-path tile: the row (kind, class, point), the slots of its partner rows and
// the output block it is written to (-1: not written).
struct F32Row {
  RowInfo ri;
  int qs, as, bs;
  int kidx;
};

__device__ __forceinline__ F32Row f32_row(const DecArgs& a, int slot, int64_t tile, int64_t n_pts) {
  F32Row fr;
  if (a.f32_U == 0) {
    fr.ri = row_info(a, slot, tile * a.Pt, n_pts);
    fr.qs = fr.ri.q;
    fr.as = fr.ri.ja * a.Pt + fr.ri.q;
    fr.bs = fr.ri.jb * a.Pt + fr.ri.q;
    fr.kidx = fr.ri.cls >= 0 ? slot / a.Pt : -1;
    return fr;
  }
  const int U = a.f32_U;
  const int64_t g0 = tile * U;
  const int64_t g = slot == 0 ? (g0 / a.R) * a.R : g0 + slot - 1;
  fr.ri.q = fr.ri.ja = fr.ri.jb = 0;
  fr.qs = fr.as = fr.bs = 0;
  if (slot > U || g >= n_pts * a.R) {
    fr.ri.cls = -1;
    fr.ri.kind = -1;
    fr.ri.p = 0;
    fr.kidx = -1;
    return fr;
  }
  const int64_t p = g / a.R;
  const int k = (int)(g - p * a.R);
  fr.ri.p = p;
  fr.ri.kind = a.kinds[k];
  fr.ri.cls = kind_class(fr.ri.kind);
  const int64_t gp = p * a.R;   // the point's primal row: in this tile, or recomputed in slot 0
  fr.qs = gp >= g0 ? (int)(gp - g0 + 1) : 0;
  fr.kidx = slot == 0 ? -1 : k;
  return fr;
}

template <int TR>
__global__ void __launch_bounds__(kF32Threads, 1) decoder_f32(DecArgs a) {
  constexpr int G = TR / 4;                   // 4-slot groups = GEMM warps = activation warps
  constexpr int TPR = kF32Threads / TR;       // threads per row in layer 0 and the output layer
  constexpr int CPT = kW / TPR;               // layer-0 columns per thread
  extern __shared__ __align__(16) float fsm[];
  float* A0 = fsm;                            // [128 f][TR slots] activations (GEMM input)
  float* A1 = A0 + kW * kF32Rows;             // [TR slots][128 f] pre-activations; staged inputs at layer 0
  float* Wt0 = A1 + kW * kF32Rows;            // two [128 in][128 out] weight buffers, transposed
  float* W0T = Wt0 + 2 * kW * kW;             // [40 in][128 out] first layer, transposed
  float* sb0 = W0T + kW0Stride * kW;          // [128]
  float* sbh = sb0 + kW;                      // [kMaxTC][128]
  float* sWout = sbh + kMaxTC * kW;           // [3][128]
  F32Row* srow = reinterpret_cast<F32Row*>(sWout + 3 * kW);        // [TR] the tile's rows
  int64_t* sxrow = reinterpret_cast<int64_t*>(srow + kF32Rows);    // [TR] their X rows
  int* sli = reinterpret_cast<int*>(sxrow + kF32Rows);             // [TR] their latent rows
  float* IN = A1;                             // [TR][kF32In] normalised inputs (layer 0 only)
  float* DIR = A1 + kF32Rows * kF32In;        // [TR][kF32In] input directions
  const int t = threadIdx.x;
  const int K0 = a.d + a.r;
  // constant operands: all loads issued before any is used
#pragma unroll
  for (int j = 0; j < (kW0Stride * kW) / kF32Threads; ++j) {
    const int e = t + j * kF32Threads;   // e = i * 128 + c
    const int i = e >> 7, c = e & (kW - 1);
    if (i < K0) W0T[e] = a.W0[c * K0 + i];
  }
  if (t < kW) sb0[t] = a.b0[t];
  if (t < a.n_tc * kW) sbh[t] = a.bh[t];
  if (t < a.d * kW) sWout[t] = a.Wout[t];
  // weights of square layer l into buffer l % 2 (asynchronous copy, waited before its GEMM)
  auto prefetch = [&](int l) {
    const float* src = a.wsqT + (size_t)l * kW * kW;
    float* dst = Wt0 + (l & 1) * kW * kW;
#pragma unroll
    for (int j = 0; j < kW * kW / 4 / kF32Threads; ++j) {
      const int e = t + j * kF32Threads;
      cp_async16(dst + 4 * e, src + 4 * e);
    }
    cp_async_commit();
  };

  const int64_t n_pts = dec_count(a);
  const int64_t n_tiles = a.f32_U ? (n_pts * a.R + a.f32_U - 1) / a.f32_U : (n_pts + a.Pt - 1) / a.Pt;
  const int warp = t >> 5, lane = t & 31;
  const int f0 = 4 * lane;                    // activations: features f0 .. f0 + 3 of slots 4 warp .. 4 warp + 3
  const int rw = t % TR, cg = t / TR;         // layer 0: slot rw, columns CPT cg .. CPT cg + CPT - 1
  for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    if (a.n_tc > 0) prefetch(0);
    // ---- the tile's rows (integer divisions once per slot) and their inputs
    if (t < TR) {
      const F32Row fr = f32_row(a, t, tile, n_pts);
      srow[t] = fr;
      int64_t xrow = 0;
      int li = 0;
      if (fr.ri.cls >= 0) row_source(a, fr.ri, xrow, li);
      sxrow[t] = xrow;
      sli[t] = li;
    }
    __syncthreads();
    for (int e = t; e < TR * K0; e += kF32Threads) {
      const int slot = e / K0, i = e - slot * K0;
      const F32Row& fr = srow[slot];
      float vin = 0.f, vdir = 0.f;
      if (fr.ri.cls >= 0) row_input_from(a, fr.ri, sxrow[slot], sli[slot], i, vin, vdir);
      IN[slot * kF32In + i] = vin;
      DIR[slot * kF32In + i] = vdir;
    }
    __syncthreads();
    // ---- layer 0 (FP32)
    {
      const RowInfo ri = srow[rw].ri;
      float z[CPT], zd[CPT];
#pragma unroll
      for (int c = 0; c < CPT; ++c) {
        z[c] = sb0[CPT * cg + c];
        zd[c] = 0.f;
      }
      for (int i = 0; i < K0; ++i) {
        const float vin = IN[rw * kF32In + i], vdir = DIR[rw * kF32In + i];
        const float4* w4 = reinterpret_cast<const float4*>(W0T + i * kW + CPT * cg);
#pragma unroll
        for (int q = 0; q < CPT / 4; ++q) {
          const float4 w = w4[q];
          z[4 * q + 0] = fmaf(w.x, vin, z[4 * q + 0]);
          z[4 * q + 1] = fmaf(w.y, vin, z[4 * q + 1]);
          z[4 * q + 2] = fmaf(w.z, vin, z[4 * q + 2]);
          z[4 * q + 3] = fmaf(w.w, vin, z[4 * q + 3]);
          zd[4 * q + 0] = fmaf(w.x, vdir, zd[4 * q + 0]);
          zd[4 * q + 1] = fmaf(w.y, vdir, zd[4 * q + 1]);
          zd[4 * q + 2] = fmaf(w.z, vdir, zd[4 * q + 2]);
          zd[4 * q + 3] = fmaf(w.w, vdir, zd[4 * q + 3]);
        }
      }
#pragma unroll
      for (int c = 0; c < CPT; ++c) {
        const int col = CPT * cg + c;
        float hv = 0.f;
        if (ri.cls == 0) hv = act_f32path(a.act, z[c]);
        else if (ri.cls == 1) hv = act_d1(a.act, z[c]) * zd[c];
        else if (ri.cls == 2) hv = act_sec(a.act, z[c], zd[c]);
        else if (ri.cls == 3) {
          const int b = ri.kind - KIND_MIXED - 1;
          const float t0 = b < a.d ? W0T[b * kW + col] / a.norm[a.d + b] : W0T[b * kW + col];
          hv = act_d2(a.act, z[c]) * zd[c] * t0;
        }
        A0[f32_slot<TR>(col, rw)] = hv;
      }
    }
    for (int l = 0; l < a.n_tc; ++l) {
      cp_async_wait_all();
      __syncthreads();                                  // A0 complete, weights of layer l landed, A1 free
      if (l + 1 < a.n_tc) prefetch(l + 1);              // overlaps the GEMM below
      if (warp < G) {
        // GEMM: lane (sg, fg) of warp w computes slots 4 sg .. 4 sg + 3 and features
        // fbase .. fbase + 3 (fbase = (512 / TR) w + 4 fg): per k one float4 of activations (eight
        // or sixteen distinct in the warp) and one of weights (four or two distinct)
        constexpr int FG = 128 / TR;                  // feature groups per warp
        const int sg = lane / FG, fg = lane % FG;
        const int fbase = (512 / TR) * warp + 4 * fg;
        const float* Wt = Wt0 + (l & 1) * kW * kW;
        float acc[4][4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int i = 0; i < 4; ++i) acc[j][i] = 0.f;
#pragma unroll 8
        for (int k = 0; k < kW; ++k) {
          const float4 av = *reinterpret_cast<const float4*>(A0 + k * TR + 4 * (sg ^ (k & (G - 1))));
          const float4 wv = *reinterpret_cast<const float4*>(Wt + k * kW + fbase);
          const float ar[4] = {av.x, av.y, av.z, av.w};
          const float wr[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
          for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[j][i] = fmaf(ar[j], wr[i], acc[j][i]);
        }
        // pre-activations (bias on primal rows) to A1
        const float4 b4 = *reinterpret_cast<const float4*>(sbh + l * kW + fbase);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (srow[4 * sg + j].ri.cls == 0) {
            acc[j][0] += b4.x;
            acc[j][1] += b4.y;
            acc[j][2] += b4.z;
            acc[j][3] += b4.w;
          }
          *reinterpret_cast<float4*>(A1 + f32_zslot(4 * sg + j, fbase)) =
              make_float4(acc[j][0], acc[j][1], acc[j][2], acc[j][3]);
        }
      }
      __syncthreads();                                  // A1 complete, every GEMM has read A0
      {
        // activations of the next layer into A0: every warp takes SPW = TR / 16 slots (warp w:
        // slots SPW w ..), so that the short dependent chains of the activations run on all
        // sixteen warps; derivative rows read their partners' pre-activations
        constexpr int SPW = TR / 16;
        float h[SPW][4];
#pragma unroll
        for (int j = 0; j < SPW; ++j) {
          const F32Row& fr = srow[SPW * warp + j];
          const float4 z4 = *reinterpret_cast<const float4*>(A1 + f32_zslot(SPW * warp + j, f0));
          const float zr[4] = {z4.x, z4.y, z4.z, z4.w};
          if (fr.ri.cls == 0) {
#pragma unroll
            for (int i = 0; i < 4; ++i) h[j][i] = act_f32path(a.act, zr[i]);
          } else if (fr.ri.cls < 0) {
#pragma unroll
            for (int i = 0; i < 4; ++i) h[j][i] = 0.f;
          } else {
            const float4 q4 = *reinterpret_cast<const float4*>(A1 + f32_zslot(fr.qs, f0));
            float4 a4 = q4, c4 = q4;
            if (fr.ri.cls == 3) {
              a4 = *reinterpret_cast<const float4*>(A1 + f32_zslot(fr.as, f0));
              c4 = *reinterpret_cast<const float4*>(A1 + f32_zslot(fr.bs, f0));
            }
            h[j][0] = f32_deriv_act(a.act, fr.ri.cls, zr[0], q4.x, a4.x, c4.x);
            h[j][1] = f32_deriv_act(a.act, fr.ri.cls, zr[1], q4.y, a4.y, c4.y);
            h[j][2] = f32_deriv_act(a.act, fr.ri.cls, zr[2], q4.z, a4.z, c4.z);
            h[j][3] = f32_deriv_act(a.act, fr.ri.cls, zr[3], q4.w, a4.w, c4.w);
          }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (SPW == 4) {
            *reinterpret_cast<float4*>(A0 + f32_slot<TR>(f0 + i, 4 * warp)) =
                make_float4(h[0][i], h[1][i], h[2 % SPW][i], h[3 % SPW][i]);
          } else {
            *reinterpret_cast<float2*>(A0 + f32_slot<TR>(f0 + i, SPW * warp)) = make_float2(h[0][i], h[1 % SPW][i]);
          }
        }
      }
    }
    __syncthreads();                                    // A0 complete
    // ---- output layer (FP32): TPR threads per row, k interleaved, combined by shuffles
    {
      const int slot = t / TPR, part = t % TPR;
      const F32Row fr = srow[slot];
      float y[3] = {0.f, 0.f, 0.f};
#pragma unroll 4
      for (int kk = 0; kk < kW / TPR; ++kk) {
        const int k = part + TPR * kk;
        const float h = A0[f32_slot<TR>(k, slot)];
#pragma unroll
        for (int i = 0; i < 3; ++i)
          if (i < a.d) y[i] = fmaf(sWout[i * kW + k], h, y[i]);
      }
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int o = 1; o < TPR; o <<= 1) y[i] += __shfl_xor_sync(0xffffffffu, y[i], o);
      if (part == 0 && fr.kidx >= 0) {
        const RowInfo& ri = fr.ri;
        float* o = a.out + ((int64_t)fr.kidx * a.n + ri.p) * a.d;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          if (i >= a.d) break;
          const float v = y[i] + (ri.cls == 0 ? a.bout[i] : 0.f);
          o[i] = v * a.norm[3 * a.d + i] + (ri.cls == 0 ? a.norm[2 * a.d + i] : 0.f);
        }
      }
    }
    __syncthreads();                                    // A0 / A1 / weight buffer 0 free for the next tile
  }
  cp_async_wait_all();
}

// --------------------------------------------------------------------------
// FP32-accurate decoder on the tensor cores (decoder_tc3).  Every FP32 operand is held as the
// exact sum of three BF16 numbers, v = hi + mid + lo (8 + 8 + 8 significand bits; weights split by
// rounding, activations by truncation), and a layer is the six products of weight 2^-16 and above,
//   A W ~ Ah Wl + Am Wm + Ah Wm + Al Wh + Am Wh + Ah Wh,
// accumulated in FP32 in that order (small terms first, so that the accumulator holds its final
// magnitude for the eight K steps of Ah Wh only); the dropped products are below 2^-23 of each term
// with signs of their own.  All layers but the output layer (N = d, FP32 on the CUDA cores) run
// this way, the first one with its inputs padded (coordinates to 4, all to a multiple of 16).
//
// A tile is 128 rows: four lane groups of 32 rows, each owned by four warps (32 columns apiece).
// Rows are taken in (point, kind) order, so that a derivative row finds its point's primal
// pre-activation in another lane of its warp (one shuffle per feature; no exchange through shared
// memory and no block barrier):
//   pipe_U = 32   32 % R == 0: a lane group holds whole points;
//   pipe_U = 31   any R: 31 consecutive rows, lane 0 recomputing the primal row of the first one's
//                point (not written out).
// NS tile slots per CTA: the sixteen epilogue warps take the slots in turn, so that one slot's
// epilogue overlaps the other's MMAs (NS = 1: calls of at most one tile per SM).  The A operand's
// high and middle images sit in tensor memory (written by the epilogue with tcgen05.st), the low
// image in shared memory; the accumulator takes 128 more columns.  One warp streams the weights
// (atoms of 128 rows x 64 K, 16 KB) through a ring of kRing slots with bulk copies, one warp per
// tile slot issues its MMAs.  A ring slot is refilled once both tile slots' MMAs on it completed.
// What bounds it: per tile and layer the tensor core takes 48 MMAs (about 65 cycles each), the sixteen
// epilogue warps about 3.2k cycles (18 instructions per element, 2.2 of 4 issue slots), the two
// overlapped.  262,144 points x 4 rows, r = 16: 0.63 ms (decoder_f32: 5.07 ms), distance from 64 bits
// 4e-8 .. 7e-8 (6.5e-8); 256 points x 17 rows: 24 us (31 us); 20,000 points x 12 rows with secants:
// 0.34 ms (1.36 ms).
// After a wait that ran out nothing waits on the copies or MMAs any more and no more weights are fetched: the
// pass runs to its end (in bounds, its results void) with the TIMEOUT status raised.
// --------------------------------------------------------------------------
constexpr int kRing = 9;
template <int NS>
constexpr int tc3_threads() { return kEpiThreads + 32 + 32 * NS; }

struct __align__(8) Tc3Tail {
  uint64_t full[kRing];
  uint64_t empty[kRing];
  uint64_t bar_mma[2];
  uint64_t drain;
  uint32_t tmem;
  int abort;      // a wait ran out
};

// hi, mid and lo words (two BF16 values each, first value in the low half) of an FP32 pair: each
// image the truncation of what the previous ones leave, so the three hold the 24 bits exactly
__device__ __forceinline__ void split3(float v0, float v1, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
  constexpr uint32_t top = 0xffff0000u, neg = 0x80000000u;
  uint32_t u0 = __float_as_uint(v0), u1 = __float_as_uint(v1);
  hi = __byte_perm(u0, u1, 0x7632);
  add2(v0, v1, __uint_as_float((u0 & top) ^ neg), __uint_as_float((u1 & top) ^ neg));
  u0 = __float_as_uint(v0);
  u1 = __float_as_uint(v1);
  mid = __byte_perm(u0, u1, 0x7632);
  add2(v0, v1, __uint_as_float((u0 & top) ^ neg), __uint_as_float((u1 & top) ^ neg));
  lo = __byte_perm(__float_as_uint(v0), __float_as_uint(v1), 0x7632);
}

// Activations of 16 columns of a row from their pre-activations (bias included on primal rows):
//   primal   z, or e^z - 1 below zero           tangent  zd, or e^zp zd
//   secant   dz, or e^zp expm1(dz) while both ends are negative and dz is small, else elu_secant
// with zp the primal pre-activation of the row's point (lane psrc).  Below zero all three are
// e^zp m + c: per-lane constants make one expression of the classes of a warp's rows.
template <int MODE>
__device__ __forceinline__ void pipe_activate(float (&z)[16], const PipeRow& rs) {
  if (MODE == PIPE_IDENTITY) return;
  if (MODE == PIPE_PRIMAL) {
#pragma unroll
    for (int i = 0; i < 16; i += 2) {
      float x0 = z[i], x1 = z[i + 1];
      mul2(x0, x1, kLog2e);
      x0 = ex2_ftz(x0);
      x1 = ex2_ftz(x1);
      add2(x0, x1, -1.0f, -1.0f);
      z[i] = z[i] > 0.f ? z[i] : x0;
      z[i + 1] = z[i + 1] > 0.f ? z[i + 1] : x1;
    }
    return;
  }
  const bool primal = rs.cls == 0;
  const float neg_c = primal ? -1.0f : 0.0f;
  const uint32_t keep = primal ? 0u : 0xffffffffu, one = primal ? 0x3f800000u : 0u;
  if (MODE == PIPE_TANGENT) {
#pragma unroll
    for (int i = 0; i < 16; i += 2) {
      const float p0 = __shfl_sync(0xffffffffu, z[i], rs.psrc);
      const float p1 = __shfl_sync(0xffffffffu, z[i + 1], rs.psrc);
      float x0 = p0, x1 = p1;
      mul2(x0, x1, kLog2e);
      x0 = fmaf(ex2_ftz(x0), __uint_as_float((__float_as_uint(z[i]) & keep) | one), neg_c);
      x1 = fmaf(ex2_ftz(x1), __uint_as_float((__float_as_uint(z[i + 1]) & keep) | one), neg_c);
      z[i] = p0 > 0.f ? z[i] : x0;
      z[i + 1] = p1 > 0.f ? z[i + 1] : x1;
    }
    return;
  }
  const bool sec = rs.cls == 2;
  const float secf = sec ? 1.0f : 0.0f;
#pragma unroll
  for (int i0 = 0; i0 < 16; i0 += 8) {
    float zp[8], out[8];
    bool rare = false;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float dz = z[i0 + j];
      zp[j] = __shfl_sync(0xffffffffu, dz, rs.psrc);
      const float z1 = fmaf(dz, secf, zp[j]);
      const bool pos = fminf(zp[j], z1) > 0.f;
      const float poly =
          dz *
          fmaf(0.5f * dz,
               fmaf(dz * (1.f / 3.f), fmaf(0.25f * dz, fmaf(0.2f * dz, fmaf(dz, 1.f / 6.f, 1.f), 1.f), 1.f), 1.f), 1.f);
      const float m = sec ? poly : __uint_as_float((__float_as_uint(dz) & keep) | one);
      rare |= sec && !pos && !(fmaxf(zp[j], z1) <= 0.f && fabsf(dz) < 0.03125f);
      out[j] = pos ? dz : fmaf(ex2_ftz(zp[j] * kLog2e), m, neg_c);
    }
    // ends of opposite sign or a large increment: the general form, for the lanes that need it
    if (__any_sync(0xffffffffu, rare)) {
      if (rare) {
#pragma unroll
        for (int j = 0; j < 8; ++j) out[j] = elu_secant(zp[j], z[i0 + j]);
      }
      __syncwarp();
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) z[i0 + j] = out[j];
  }
}

template <int NS, int MODE>
__global__ void __launch_bounds__(tc3_threads<NS>(), 1) decoder_tc3(DecArgs a) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  // 1024-byte alignment by an offset, so that the pointers stay known as shared memory
  uint8_t* smem = smem_raw + ((1024u - (tc::smem_addr(smem_raw) & 1023u)) & 1023u);
  uint8_t* ring = smem;                                  // kRing x 16 KB weight atoms
  uint8_t* lotile = ring + kRing * kAtomBytes;           // NS x 32 KB low images
  float* ypart = (float*)(lotile + NS * kLayerBytes);    // [3][128][3]
  float* sb0 = ypart + 3 * 128 * 3;                      // [128]
  float* sbh = sb0 + kW;                                 // [kMaxTC][128]
  float* sWout = sbh + kMaxTC * kW;                      // [3][128]
  float* snorm = sWout + 3 * kW;                         // [8] X_min, X_range
  Tc3Tail* tail = (Tc3Tail*)(snorm + 8);
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;

  if (t == 0) {
    for (int i = 0; i < kRing; ++i) {
      tc::mbar_init(&tail->full[i], 1);
      tc::mbar_init(&tail->empty[i], NS);
    }
    tc::mbar_init(&tail->bar_mma[0], 1);
    tc::mbar_init(&tail->bar_mma[1], 1);
    tc::mbar_init(&tail->drain, NS);
    tail->abort = 0;
    tc::fence_mbar_init();
  }
  if (warp == 0) tc::tmem_alloc<256 * NS>(&tail->tmem);
  for (int e = t; e < kW; e += tc3_threads<NS>()) sb0[e] = finite_bias(a.b0[e]);
  for (int e = t; e < a.n_tc * kW; e += tc3_threads<NS>()) sbh[e] = finite_bias(a.bh[e]);
  for (int e = t; e < 3 * kW; e += tc3_threads<NS>()) sWout[e] = e < a.d * kW ? a.Wout[e] : 0.f;
  if (t < 2 * a.d) snorm[t] = a.norm[t];
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();

  const int n_rows = (int)dec_count(a) * a.R;
  const int U = a.pipe_U;
  const int n_tiles = (int)(((int64_t)n_rows + 4 * U - 1) / (4 * U));
  // tiles per pass: one while every tile has a CTA of its own (slot 1 then has none)
  const int NT = n_tiles <= (int)gridDim.x ? 1 : NS;
  const int n_iter = (n_tiles + NT - 1) / NT;
  const int K0 = kTcLat + a.r;                            // first-layer inputs, padded layout
  const int KS0 = (K0 + 15) / 16;                         // their K steps
  const int atoms = 3 + 6 * a.n_tc;

  uint32_t fetched = 0;   // weight copies this thread started
  if (warp == kEpiThreads / 32) {
    // ---- weight stream
    if (lane == 0) {
      const uint32_t passes = (int)blockIdx.x < n_iter ? (uint32_t)(n_iter - 1 - (int)blockIdx.x) / gridDim.x + 1 : 0;
      int j = 0;   // atom of the pass
      fetched = ring_fill<kRing>(
          passes * (uint32_t)atoms,
          [&](uint32_t slot, uint32_t phase) { return pipe_wait(a.status, &tail->abort, &tail->empty[slot], phase); },
          [&](uint32_t slot, uint32_t) {
            tc::mbar_expect_tx(&tail->full[slot], (uint32_t)kAtomBytes);
            tc::bulk_g2s(ring + slot * kAtomBytes, a.wstream + (size_t)j * kAtomBytes, kAtomBytes, &tail->full[slot]);
            j = j + 1 < atoms ? j + 1 : 0;
          });
    }
    __syncwarp();
  } else if (warp > kEpiThreads / 32) {
    // ---- MMA issuer of slot s.  The whole warp runs the loop; one elected lane issues.
    const int s = warp - kEpiThreads / 32 - 1;
    const bool leader = tc::elect_one();
    const uint32_t tD = tail->tmem + (uint32_t)(s * 256), tAh = tD + 128, tAm = tD + 192;
    const uint32_t lo_desc = tc::smem_desc_sw128_lo(tc::smem_addr(lotile + s * kLayerBytes));
    const uint32_t ring_desc = tc::smem_desc_sw128_lo(tc::smem_addr(ring));
    constexpr uint32_t idesc = tc::idesc_bf16_f32(128, kW), kAtomDesc = kAtomBytes >> 4;
    uint32_t atom = 0, mma_phase = 0;
    // waits for the next atom of the stream, returns its ring slot
    auto take = [&]() {
      const uint32_t slot = atom % kRing;
      pipe_wait(a.status, &tail->abort, &tail->full[slot], (atom / kRing) & 1u);
      __syncwarp();
      ++atom;
      return slot;
    };
    for (int it = blockIdx.x; it < n_iter; it += gridDim.x) {
      if (s >= NT || it * NT + s >= n_tiles) {
        // no tile: the slot only releases the pass's atoms
        for (int j = 0; j < atoms; ++j) {
          const uint32_t r = take();
          if (leader) tc::mbar_arrive(&tail->empty[r]);
        }
        continue;
      }
      for (int l = -1; l < a.n_tc; ++l) {
        pipe_sync(1 + s);
        tc::tc_fence_after();
        if (l < 0) {
          // first layer: one atom per image, KS0 K steps
          for (int img = 0; img < 3; ++img) {
            const uint32_t r = take();
            if (leader) {
              const uint32_t bd = ring_desc + r * kAtomDesc;
              auto desc = [](uint32_t lo) { return ((uint64_t)tc::kDescSw128Hi << 32) | lo; };
              if (img == 2)
                for (int k = 0; k < KS0; ++k)
                  tc::mma_bf16(tD, desc(lo_desc + 2 * k), desc(bd + 2 * k), idesc, 1u);
              if (img > 0)
                for (int k = 0; k < KS0; ++k) tc::mma_bf16_ts(tD, tAm + 8 * k, desc(bd + 2 * k), idesc, 1u);
              for (int k = 0; k < KS0; ++k)
                tc::mma_bf16_ts(tD, tAh + 8 * k, desc(bd + 2 * k), idesc, img > 0 || k > 0 ? 1u : 0u);
              tc::mma_commit(&tail->empty[r]);
            }
            __syncwarp();
          }
        } else {
#pragma unroll
          for (int kh = 0; kh < 2; ++kh) {               // low weight image
            const uint32_t r = take();
            if (leader) {
              tc::mma4_bf16_ts(tD, tAh + kh * 32, ring_desc + r * kAtomDesc, idesc, kh);
              tc::mma_commit(&tail->empty[r]);
            }
          }
#pragma unroll
          for (int kh = 0; kh < 2; ++kh) {               // middle
            const uint32_t r = take();
            if (leader) {
              tc::mma4_bf16_ts(tD, tAm + kh * 32, ring_desc + r * kAtomDesc, idesc, 1u);
              tc::mma4_bf16_ts(tD, tAh + kh * 32, ring_desc + r * kAtomDesc, idesc, 1u);
              tc::mma_commit(&tail->empty[r]);
            }
          }
          uint32_t rh[2];
#pragma unroll
          for (int kh = 0; kh < 2; ++kh) {               // high: the small products of both atoms first
            rh[kh] = take();
            if (leader) {
              tc::mma4_bf16_ss(tD, lo_desc + kh * kAtomDesc, ring_desc + rh[kh] * kAtomDesc, idesc, 1u);
              tc::mma4_bf16_ts(tD, tAm + kh * 32, ring_desc + rh[kh] * kAtomDesc, idesc, 1u);
            }
          }
          if (leader) {
#pragma unroll
            for (int kh = 0; kh < 2; ++kh) {
              tc::mma4_bf16_ts(tD, tAh + kh * 32, ring_desc + rh[kh] * kAtomDesc, idesc, 1u);
              tc::mma_commit(&tail->empty[rh[kh]]);
            }
          }
        }
        if (leader) tc::mma_commit(&tail->bar_mma[s]);
        __syncwarp();
        pipe_wait(a.status, &tail->abort, &tail->bar_mma[s], mma_phase);
        mma_phase ^= 1u;
        __syncwarp();
        tc::tc_fence_after();
        tc::tc_fence_before();
        pipe_arrive(3 + s);
      }
    }
    // MMAs of a timed-out pass complete (bounded) before the tensor memory is freed
    if (leader) tc::mma_commit(&tail->drain);
    __syncwarp();
    (void)tc::mbar_wait(&tail->drain, 0);
    __syncwarp();
  } else {
    // ---- epilogue warps: rows 32 (warp % 4) + lane, columns 32 h .. 32 h + 31
    const int h = warp >> 2;
    const bool vec4 = pipe_vec4(a);
    const int rw = (warp & 3) * 32 + lane;                 // tile row / tensor-memory lane
    const uint32_t tbase = tail->tmem + ((uint32_t)((warp & 3) * 32) << 16);
    auto put8 = [&](int s, int c, const float v[8]) {      // inputs 8 c .. 8 c + 7 of the slot's operand row
      uint32_t wh[4], wm[4], wl[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) split3(v[2 * j], v[2 * j + 1], wh[j], wm[j], wl[j]);
      __syncwarp();
      tc::tmem_st4(tbase + s * 256 + 128 + 4 * c, wh);
      tc::tmem_st4(tbase + s * 256 + 192 + 4 * c, wm);
      *reinterpret_cast<uint4*>(lotile + s * kLayerBytes + tc::sw128_offset(rw, 8 * c, kW)) =
          make_uint4(wl[0], wl[1], wl[2], wl[3]);
    };
    // first-layer operand of a slot: inputs 0 .. 31 by the four column parts, 32 .. 47 (K0 > 32) by
    // the first two, which load the last 8 here
    auto put = [&](int s, int tile, PipeIn& in) {
      pipe_finish<MODE>(a.d, snorm, h, in);
      if (h < 2 * KS0) put8(s, h, in.v);
      if (K0 > 32 && h < 2) {
        PipeIn hi;
        (void)pipe_load<MODE>(a, (tile * 4 + (warp & 3)) * U, U, n_rows, lane, 4 + h, vec4, hi);
        pipe_finish<MODE>(a.d, snorm, 4 + h, hi);
        put8(s, 4 + h, hi.v);
      }
    };
    // the slot's operand is complete and its accumulator read: its issuer may go on
    auto ready = [&](int s) {
      tc::tmem_wait_st();
      tc::fence_async_smem();
      tc::tc_fence_before();
      pipe_arrive(1 + s);
    };

    PipeRow rows[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      const int tile = blockIdx.x * NT + s;
      if ((int)blockIdx.x < n_iter && s < NT && tile < n_tiles) {
        PipeIn in;
        rows[s] = pipe_load<MODE>(a, (tile * 4 + (warp & 3)) * U, U, n_rows, lane, h, vec4, in);
        put(s, tile, in);
        ready(s);
      }
    }
    for (int it = blockIdx.x; it < n_iter; it += gridDim.x) {
      for (int l = -1; l < a.n_tc; ++l) {
        const bool last = l == a.n_tc - 1;
        const float* bl = l < 0 ? sb0 : sbh + l * kW;
#pragma unroll 1
        for (int s = 0; s < NS; ++s) {
          if (s >= NT || it * NT + s >= n_tiles) break;
          const PipeRow rs = s == 0 ? rows[0] : rows[NS - 1];
          const bool primal = rs.cls == 0;
          const float one_p = primal ? 1.0f : 0.0f;
          const uint32_t ts = tbase + s * 256;
          uint8_t* lo_t = lotile + s * kLayerBytes;
          float y[3] = {0.f, 0.f, 0.f};
          // the slot's next tile: its inputs load while the last accumulator completes
          PipeIn in;
          const int next = (it + (int)gridDim.x) * NT + s;
          const bool more = last && it + (int)gridDim.x < n_iter && next < n_tiles;
          if (more) {
            const PipeRow nr = pipe_load<MODE>(a, (next * 4 + (warp & 3)) * U, U, n_rows, lane, h, vec4, in);
            if (s == 0) rows[0] = nr;
            else rows[NS - 1] = nr;
          }
          pipe_sync(3 + s);
          tc::tc_fence_after();
#pragma unroll 1
          for (int c0 = 32 * h; c0 < 32 * h + 32; c0 += 16) {
            float z[16];
            tc::tmem_ld16(ts + c0, z);
            // the bias of primal rows (a factor 0 on the others)
#pragma unroll
            for (int i = 0; i < 16; i += 4) {
              const float4 b4 = *reinterpret_cast<const float4*>(bl + c0 + i);
              fma2(z[i], z[i + 1], b4.x, b4.y, one_p);
              fma2(z[i + 2], z[i + 3], b4.z, b4.w, one_p);
            }
            pipe_activate<MODE>(z, rs);
            if (last) {
              // output layer fused into the last epilogue (FP32), partial over this part's columns
#pragma unroll
              for (int o = 0; o < 3; ++o) {
                if (o >= a.d) break;
                float q0 = 0.f, q1 = 0.f, q2 = 0.f, q3 = 0.f;   // short chains, added pairwise
#pragma unroll
                for (int i = 0; i < 16; i += 4) {
                  const float4 w4 = *reinterpret_cast<const float4*>(sWout + o * kW + c0 + i);
                  q0 = fmaf(w4.x, z[i], q0);
                  q1 = fmaf(w4.y, z[i + 1], q1);
                  q2 = fmaf(w4.z, z[i + 2], q2);
                  q3 = fmaf(w4.w, z[i + 3], q3);
                }
                y[o] += (q0 + q1) + (q2 + q3);
              }
            } else {
              uint32_t wh[8], wm[8], wl[8];
#pragma unroll
              for (int j = 0; j < 8; ++j) split3(z[2 * j], z[2 * j + 1], wh[j], wm[j], wl[j]);
              tc::tmem_st8(ts + 128 + c0 / 2, wh);
              tc::tmem_st8(ts + 192 + c0 / 2, wm);
              *reinterpret_cast<uint4*>(lo_t + tc::sw128_offset(rw, c0, kW)) = make_uint4(wl[0], wl[1], wl[2], wl[3]);
              *reinterpret_cast<uint4*>(lo_t + tc::sw128_offset(rw, c0 + 8, kW)) =
                  make_uint4(wl[4], wl[5], wl[6], wl[7]);
            }
          }
          if (!last) {
            ready(s);
            continue;
          }
          if (more) {
            put(s, next, in);
            ready(s);
          }
          if (h < 3) {
#pragma unroll
            for (int o = 0; o < 3; ++o)
              if (o < a.d) ypart[(h * 128 + rw) * 3 + o] = y[o];
          }
          // part 3 (part 0 has the coordinates' divisions in put) waits for the others; they go on
          // (ypart is rewritten after the next accumulator barrier, which part 3 reaches only when it
          // has read it)
          pipe_combine(h);
          if (h == 3 && rs.kidx >= 0) {
            float* o = a.out + ((int64_t)rs.kidx * a.n + rs.p) * a.d;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
              if (i >= a.d) break;
              float v = (ypart[rw * 3 + i] + ypart[(128 + rw) * 3 + i]) + (ypart[(256 + rw) * 3 + i] + y[i]);
              if (primal) v += __ldg(&a.bout[i]);
              o[i] = v * a.norm[3 * a.d + i] + (primal ? a.norm[2 * a.d + i] : 0.f);
            }
          }
        }
      }
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  // after a timeout the last copies land before the CTA exits
  if (fetched > 0 && *(volatile int*)&tail->abort)
    ring_land<kRing>(fetched, [&](uint32_t slot, uint32_t phase) { (void)tc::mbar_wait(&tail->full[slot], phase); });
  if (warp == 0) tc::tmem_free<256 * NS>(tail->tmem);
}

// --------------------------------------------------------------------------
// BF16 decoder for calls without mixed rows (primal, tangent, JVP and secant rows; inputs of at
// most 32 entries in the padded layout), built like decoder_tc3: rows in (point, kind) order, the
// primal pre-activation of a derivative row fetched by a shuffle, sixteen epilogue warps taking the
// NS tile slots in turn, one MMA issuer warp per slot.  All weights are resident (four 32 KB layers
// and the first layer's split image), and the A operand sits in tensor memory alone: 64 columns of
// BF16 activations, or for the first layer 16 + 16 of the inputs' high and low parts.  The
// arithmetic and its order are decoder_tc's (without SPLIT), so the results are the same bits.
//
// TRAIN: whole points only (pipe_U = R floor(32 / R) rows per lane group, the other lanes idle); every
// layer's operand is also stored as the tile image the MMA reads (128 rows x 128 BF16 in the 128-byte
// swizzle, 32 KB): the epilogue writes it to shared memory, from where the MMA reads it and one bulk
// copy stores it (16-byte stores of each thread's row touch 32 lines per instruction: 280 us instead
// of 150 us for 65,536 points x 4 rows); and the primal rows' slope records per point, 16-byte
// chunks permuted per point (stage_chunk).
//
// What bounds it: the epilogue, 1.7k cycles per tile and layer (the special-function unit's 16
// exponentials a clock take 1.0k of them), and about 3k per tile for its inputs and outputs; the
// tensor core is busy 20 % of the time.  1,048,576 primal rows: 0.297 ms (0.493 ms as two groups of
// eight warps with a tile each, whose epilogues ran at the latency of two warps per scheduler);
// 100,003 points x 4 rows 0.173 ms (0.446 ms in decoder_tc, which exchanges the rows'
// pre-activations through shared memory); 5,001 points x 9 rows 35 us (87 us).
// --------------------------------------------------------------------------
template <int NS>
constexpr int bf16_threads() { return kEpiThreads + 32 * NS; }

struct __align__(8) Bf16Tail {
  uint64_t bar_w;
  uint64_t bar_mma[2];
  uint64_t drain;
  uint32_t tmem;
  int abort;      // a wait ran out (as in decoder_tc3)
};

template <int NS, int MODE, bool TRAIN>
__global__ void __launch_bounds__(bf16_threads<NS>(), 1) decoder_bf16(DecArgs a) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (tc::smem_addr(smem_raw) & 1023u)) & 1023u);
  uint8_t* wsm = smem;                                   // kMaxTC x 32 KB square layers
  uint8_t* w0s = smem + kMaxTC * kLayerBytes;            // 16 KB first-layer split image
  uint8_t* images = w0s + kLayerBytes / 2;               // TRAIN: NS x 32 KB operand images
  float* ypart = (float*)(images + (TRAIN ? NS * kLayerBytes : 0));   // [3][128][3]
  float* sb0 = ypart + 3 * 128 * 3;                      // [128]
  float* sbh = sb0 + kW;                                 // [kMaxTC][128]
  float* sWout = sbh + kMaxTC * kW;                      // [3][128]
  float* snorm = sWout + 3 * kW;                         // [8] X_min, X_range
  Bf16Tail* tail = (Bf16Tail*)(snorm + 8);
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;

  if (t == 0) {
    tc::mbar_init(&tail->bar_w, 1);
    tc::mbar_init(&tail->bar_mma[0], 1);
    tc::mbar_init(&tail->bar_mma[1], 1);
    tc::mbar_init(&tail->drain, NS);
    tail->abort = 0;
    tc::fence_mbar_init();
    tc::mbar_expect_tx(&tail->bar_w, (uint32_t)(a.n_tc * kLayerBytes + kLayerBytes / 2));
    tc::bulk_g2s(w0s, a.w0img, kLayerBytes / 2, &tail->bar_w);
    for (int l = 0; l < a.n_tc; ++l)
      tc::bulk_g2s(wsm + l * kLayerBytes, a.wimg + (size_t)l * kLayerBytes, kLayerBytes, &tail->bar_w);
  }
  if (warp == 0) tc::tmem_alloc<256 * NS>(&tail->tmem);
  for (int e = t; e < kW; e += bf16_threads<NS>()) sb0[e] = finite_bias(a.b0[e]);
  for (int e = t; e < a.n_tc * kW; e += bf16_threads<NS>()) sbh[e] = finite_bias(a.bh[e]);
  for (int e = t; e < 3 * kW; e += bf16_threads<NS>()) sWout[e] = e < a.d * kW ? a.Wout[e] : 0.f;
  if (t < 2 * a.d) snorm[t] = a.norm[t];
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();

  const int n_rows = (int)dec_count(a) * a.R;
  const int U = a.pipe_U;
  const int n_tiles = (int)(((int64_t)n_rows + 4 * U - 1) / (4 * U));
  const int NT = n_tiles <= (int)gridDim.x ? 1 : NS;          // tiles per pass, as in decoder_tc3
  const int n_iter = (n_tiles + NT - 1) / NT;

  if (warp >= kEpiThreads / 32) {
    // ---- MMA issuer of slot s
    const int s = warp - kEpiThreads / 32;
    const bool leader = tc::elect_one();
    const uint32_t tD = tail->tmem + (uint32_t)(s * 256), tA = tD + 128, tI = tD + 192;   // tI: inputs hi, lo
    const uint32_t w_desc = tc::smem_desc_sw128_lo(tc::smem_addr(wsm));
    const uint32_t w0_desc = tc::smem_desc_sw128_lo(tc::smem_addr(w0s));
    constexpr uint32_t idesc = tc::idesc_bf16_f32(128, kW);
    uint32_t mma_phase = 0;
    pipe_wait(a.status, &tail->abort, &tail->bar_w, 0);
    __syncwarp();
    uint8_t* image = images + s * kLayerBytes;
    const uint32_t image_desc = tc::smem_desc_sw128_lo(tc::smem_addr(image));
    // TRAIN: the image of activation layer `layer` leaves for the store
    auto store_image = [&](int layer, int tile) {
      tc::bulk_s2g(a.astore + ((int64_t)layer * a.rows_total + (int64_t)tile * 128) * kW, image, kLayerBytes);
    };
    int prev = -1;   // this slot's previous tile, whose last image is not stored yet
    for (int it = blockIdx.x; it < n_iter; it += gridDim.x) {
      if (s >= NT || it * NT + s >= n_tiles) continue;
      for (int l = -1; l < a.n_tc; ++l) {
        pipe_sync(1 + s);
        tc::tc_fence_after();
        if (leader) {
          if (l < 0) {
            auto desc = [](uint32_t lo) { return ((uint64_t)tc::kDescSw128Hi << 32) | lo; };
#pragma unroll
            for (int k = 0; k < 2; ++k) {   // hi at byte 0 of an image row, lo at byte 64
              tc::mma_bf16_ts(tD, tI + 8 * k, desc(w0_desc + 2 * k), idesc, k > 0 ? 1u : 0u);
              tc::mma_bf16_ts(tD, tI + 8 * k, desc(w0_desc + 4 + 2 * k), idesc, 1u);
              tc::mma_bf16_ts(tD, tI + 16 + 8 * k, desc(w0_desc + 2 * k), idesc, 1u);
            }
          } else {
            const uint32_t bd = w_desc + (uint32_t)l * (kLayerBytes >> 4);
            if (TRAIN) {
              tc::mma4_bf16_ss(tD, image_desc, bd, idesc, 0u);
              tc::mma4_bf16_ss(tD, image_desc + (kAtomBytes >> 4), bd + (kAtomBytes >> 4), idesc, 1u);
            } else {
              tc::mma4_bf16_ts(tD, tA, bd, idesc, 0u);
              tc::mma4_bf16_ts(tD, tA + 32, bd + (kAtomBytes >> 4), idesc, 1u);
            }
          }
          tc::mma_commit(&tail->bar_mma[s]);
          if (TRAIN && l >= 0) store_image(l, it * NT + s);
          if (TRAIN && l < 0 && prev >= 0) store_image(a.n_tc, prev);
        }
        __syncwarp();
        pipe_wait(a.status, &tail->abort, &tail->bar_mma[s], mma_phase);
        mma_phase ^= 1u;
        if (TRAIN && leader) tc::bulk_wait_read();   // the image may be rewritten
        __syncwarp();
        tc::tc_fence_after();
        tc::tc_fence_before();
        pipe_arrive(3 + s);
      }
      prev = it * NT + s;
    }
    if (TRAIN && prev >= 0) {
      pipe_sync(1 + s);
      if (leader) {
        store_image(a.n_tc, prev);
        tc::bulk_wait_all();
      }
      __syncwarp();
    }
    // MMAs of a timed-out pass complete (bounded) before the tensor memory is freed; the weights
    // have landed (waited for above, or here after a timeout)
    if (leader) tc::mma_commit(&tail->drain);
    __syncwarp();
    (void)tc::mbar_wait(&tail->drain, 0);
    if (*(volatile int*)&tail->abort) (void)tc::mbar_wait(&tail->bar_w, 0);
    __syncwarp();
  } else {
    // ---- epilogue warps: rows 32 (warp % 4) + lane, columns 32 h .. 32 h + 31
    const int h = warp >> 2;
    const bool vec4 = pipe_vec4(a);
    const int rw = (warp & 3) * 32 + lane;
    const uint32_t tbase = tail->tmem + ((uint32_t)((warp & 3) * 32) << 16);
    auto pack2 = [](float v0, float v1) {
      const __nv_bfloat162 b = __floats2bfloat162_rn(v0, v1);
      return *reinterpret_cast<const uint32_t*>(&b);
    };
    // first-layer operand (inputs in the padded layout: coordinates at 0 .. 3, latents from
    // kTcLat): bf16(v) and bf16(v - bf16(v))
    auto put = [&](int s, PipeIn& in) {
      pipe_finish<MODE>(a.d, snorm, h, in);
      const float* v = in.v;
      uint32_t wh[4], wl[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        wh[j] = pack2(v[2 * j], v[2 * j + 1]);
        wl[j] = pack2(v[2 * j] - __uint_as_float(wh[j] << 16), v[2 * j + 1] - __uint_as_float(wh[j] & 0xffff0000u));
      }
      __syncwarp();
      tc::tmem_st4(tbase + s * 256 + 192 + 4 * h, wh);
      tc::tmem_st4(tbase + s * 256 + 208 + 4 * h, wl);
    };
    auto ready = [&](int s) {
      tc::tmem_wait_st();
      if (TRAIN) tc::fence_async_smem();
      tc::tc_fence_before();
      pipe_arrive(1 + s);
    };

    const int pt = TRAIN ? (warp & 3) * (U / a.R) + lane / a.R : 0;   // the row's point within the tile
    const bool pt_lane = TRAIN && lane < U && lane % a.R == 0;        // a point's (valid or padding) primal row
    PipeRow rows[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      const int tile = blockIdx.x * NT + s;
      if ((int)blockIdx.x < n_iter && s < NT && tile < n_tiles) {
        PipeIn in;
        rows[s] = pipe_load<MODE, TRAIN>(a, (tile * 4 + (warp & 3)) * U, U, n_rows, lane, h, vec4, in);
        put(s, in);
        ready(s);
      }
    }
    for (int it = blockIdx.x; it < n_iter; it += gridDim.x) {
      for (int l = -1; l < a.n_tc; ++l) {
        const bool last = l == a.n_tc - 1;
        const float* bl = l < 0 ? sb0 : sbh + l * kW;
#pragma unroll 1
        for (int s = 0; s < NS; ++s) {
          if (s >= NT || it * NT + s >= n_tiles) break;
          const PipeRow rs = s == 0 ? rows[0] : rows[NS - 1];
          const bool primal = rs.cls == 0;
          const float one_p = primal ? 1.0f : 0.0f;
          const uint32_t ts = tbase + s * 256;
          float y[3] = {0.f, 0.f, 0.f};
          // the slot's next tile: its inputs load while the last accumulator completes
          PipeIn in;
          const int next = (it + (int)gridDim.x) * NT + s;
          const bool more = last && it + (int)gridDim.x < n_iter && next < n_tiles;
          if (more) {
            const PipeRow nr = pipe_load<MODE, TRAIN>(a, (next * 4 + (warp & 3)) * U, U, n_rows, lane, h, vec4, in);
            if (s == 0) rows[0] = nr;
            else rows[NS - 1] = nr;
          }
          pipe_sync(3 + s);
          tc::tc_fence_after();
#pragma unroll 1
          for (int c0 = 32 * h; c0 < 32 * h + 32; c0 += 16) {
            float z[16];
            tc::tmem_ld16(ts + c0, z);
#pragma unroll
            for (int i = 0; i < 16; i += 4) {   // the bias of primal rows (a factor 0 on the others)
              const float4 b4 = *reinterpret_cast<const float4*>(bl + c0 + i);
              fma2(z[i], z[i + 1], b4.x, b4.y, one_p);
              fma2(z[i + 2], z[i + 3], b4.z, b4.w, one_p);
            }
            if (TRAIN) {
              // the primal rows' slope records (act_slope_record), and both activations from them
              uint32_t rec[8];
              const float neg_c = primal ? -1.0f : 0.0f;
              const uint32_t keep = primal ? 0u : 0xffffffffu, one = primal ? 0x3f800000u : 0u;
#pragma unroll
              for (int i = 0; i < 16; i += 2) {
                const float p0 = __shfl_sync(0xffffffffu, z[i], rs.psrc);
                const float p1 = __shfl_sync(0xffffffffu, z[i + 1], rs.psrc);
                float s0 = p0, s1 = p1;
                mul2(s0, s1, kLog2e);
                s0 = ex2_ftz(s0);
                s1 = ex2_ftz(s1);
                const bool lin0 = MODE == PIPE_IDENTITY || !(p0 < 0.f), lin1 = MODE == PIPE_IDENTITY || !(p1 < 0.f);
                rec[i / 2] = pack2(lin0 ? -1.f : s0, lin1 ? -1.f : s1);
                s0 = fmaf(s0, __uint_as_float((__float_as_uint(z[i]) & keep) | one), neg_c);
                s1 = fmaf(s1, __uint_as_float((__float_as_uint(z[i + 1]) & keep) | one), neg_c);
                z[i] = lin0 ? z[i] : s0;
                z[i + 1] = lin1 ? z[i + 1] : s1;
              }
              if (pt_lane) {
                // the point's row of 256 bytes, its chunks permuted by its place in the tile
                uint8_t* o = reinterpret_cast<uint8_t*>(a.dstore + ((int64_t)(l + 1) * a.points_total + rs.p) * kW);
                *reinterpret_cast<uint4*>(o + stage_chunk(pt, c0 / 8) - pt * 256) =
                    make_uint4(rec[0], rec[1], rec[2], rec[3]);
                *reinterpret_cast<uint4*>(o + stage_chunk(pt, c0 / 8 + 1) - pt * 256) =
                    make_uint4(rec[4], rec[5], rec[6], rec[7]);
              }
            } else {
              pipe_activate<MODE>(z, rs);
            }
            if (last) {
              // output layer fused into the last epilogue (FP32): one chain over the part's 32 columns
#pragma unroll
              for (int o = 0; o < 3; ++o) {
                if (o >= a.d) break;
#pragma unroll
                for (int i = 0; i < 16; i += 4) {
                  const float4 w4 = *reinterpret_cast<const float4*>(sWout + o * kW + c0 + i);
                  y[o] = fmaf(w4.x, z[i], y[o]);
                  y[o] = fmaf(w4.y, z[i + 1], y[o]);
                  y[o] = fmaf(w4.z, z[i + 2], y[o]);
                  y[o] = fmaf(w4.w, z[i + 3], y[o]);
                }
              }
            }
            if (!last || TRAIN) {
              uint32_t w[8];
#pragma unroll
              for (int j = 0; j < 8; ++j) w[j] = pack2(z[2 * j], z[2 * j + 1]);
              if (TRAIN) {
                uint8_t* image = images + s * kLayerBytes;
                *reinterpret_cast<uint4*>(image + tc::sw128_offset(rw, c0, kW)) = make_uint4(w[0], w[1], w[2], w[3]);
                *reinterpret_cast<uint4*>(image + tc::sw128_offset(rw, c0 + 8, kW)) = make_uint4(w[4], w[5], w[6], w[7]);
              } else {
                tc::tmem_st8(ts + 128 + c0 / 2, w);
              }
            }
          }
          if (!last) {
            ready(s);
            continue;
          }
          if (more) put(s, in);
          if (more || TRAIN) ready(s);   // TRAIN: the last image, stored by the issuer
          if (h < 3) {
#pragma unroll
            for (int o = 0; o < 3; ++o)
              if (o < a.d) ypart[(h * 128 + rw) * 3 + o] = y[o];
          }
          pipe_combine(h);   // as in decoder_tc3
          if (h == 3 && rs.kidx >= 0) {
            float* o = a.out + ((int64_t)rs.kidx * a.n + rs.p) * a.d;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
              if (i >= a.d) break;
              float vo = (ypart[rw * 3 + i] + ypart[(128 + rw) * 3 + i]) + (ypart[(256 + rw) * 3 + i] + y[i]);
              vo += primal ? __ldg(&a.bout[i]) : 0.f;
              o[i] = vo * a.norm[3 * a.d + i] + (primal ? a.norm[2 * a.d + i] : 0.f);
            }
          }
        }
      }
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  if (warp == 0) tc::tmem_free<256 * NS>(tail->tmem);
}

// Everything the kernels read in another form than the parameter vector's, in one launch (it runs after
// every optimisation step; as eight copies and four kernels a parameter change took 52 us, like this 14.5):
//   bsq      the square layers' biases, contiguous
//   wsqT     the square layers transposed, WT[l][k][f] = W[l][f][k] (decoder_f32)
//   wimg     bf16(w), and wimg_lo bf16(w - bf16(w)), in the 128-byte swizzled K-major layout the MMA reads
//   wstream  decoder_tc3's: per layer the low, middle and high BF16 images (w = hi + mid + lo exactly, each rounded
//            to nearest) as atoms of 128 output rows x 64 K in the same layout: the first layer (padded
//            inputs, at most 42) one atom per image, the square layers two
//   w0img    the first layer for the tensor cores where its padded inputs fit 32: bf16(w) at K 0 .. 31 of a row,
//            bf16(w - bf16(w)) at 32 .. 63 (one 16 KB atom column)
// Padded inputs: coordinates at 0 .. 3, latents from kTcLat, zero where no input sits.
// Blocks of 256 threads: one per 32 x 32 tile of a square layer, then kDeriveW0 for the first layer and the biases.
constexpr int kDeriveThreads = 256, kDeriveW0 = kW * 64 / 1024;
struct DeriveArgs {
  const float* W0;          // (W, d + r)
  const float* sq;          // first square layer, each kW * kW weights and kW biases
  int d, r, n_tc;
  float *bsq, *wsqT;
  uint8_t *wimg, *wimg_lo, *wstream, *w0img;   // w0img may be null
};

__device__ __forceinline__ void put_bf16(uint8_t* img, size_t at, __nv_bfloat16 v) {
  *reinterpret_cast<__nv_bfloat16*>(img + at) = v;
}

__global__ void __launch_bounds__(kDeriveThreads) decoder_derive(DeriveArgs a) {
  __shared__ float tile[32][33];
  const int t = threadIdx.x;
  const int b = (int)blockIdx.x - 16 * a.n_tc;
  const bool square = b < 0;
  const int l = (int)blockIdx.x / 16, f0 = ((int)blockIdx.x / 4 % 4) * 32, k0 = ((int)blockIdx.x % 4) * 32;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    int row, k;             // output feature, input (square layers: of 128; first layer: of 64 padded)
    float w;
    size_t at, step;        // low image's atom, and the distance to the next image's
    if (square) {
      row = f0 + t / 32 + 8 * i;
      k = k0 + t % 32;
      w = a.sq[(size_t)l * (kW * kW + kW) + row * kW + k];
      at = 3 + 6 * (size_t)l + k / 64;
      step = 2;
      tile[t / 32 + 8 * i][t % 32] = w;
    } else {
      const int e = b * 1024 + t + kDeriveThreads * i;
      row = e / 64;
      k = e % 64;
      const int in = k < kTcLat ? (k < a.d ? k : -1) : (k - kTcLat < a.r ? a.d + k - kTcLat : -1);
      w = in >= 0 ? a.W0[row * (a.d + a.r) + in] : 0.f;
      at = 0;
      step = 1;
    }
    const __nv_bfloat16 hi = __float2bfloat16_rn(w);
    const float r1 = w - __bfloat162float(hi);
    const __nv_bfloat16 mid = __float2bfloat16_rn(r1);
    const __nv_bfloat16 lo = __float2bfloat16_rn(r1 - __bfloat162float(mid));
    const size_t o = at * kAtomBytes + tc::sw128_offset(row, k & 63, kW);
    put_bf16(a.wstream, o, lo);
    put_bf16(a.wstream, o + step * kAtomBytes, mid);
    put_bf16(a.wstream, o + 2 * step * kAtomBytes, hi);
    if (square) {
      const size_t q = (size_t)l * kLayerBytes + tc::sw128_offset(row, k, kW);
      put_bf16(a.wimg, q, hi);
      put_bf16(a.wimg_lo, q, mid);
    } else if (a.w0img && k < 32) {
      put_bf16(a.w0img, tc::sw128_offset(row, k, kW), hi);
      put_bf16(a.w0img, tc::sw128_offset(row, 32 + k, kW), mid);
    }
  }
  if (square) {
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i)
      a.wsqT[(size_t)l * kW * kW + (k0 + t / 32 + 8 * i) * kW + f0 + t % 32] = tile[t % 32][t / 32 + 8 * i];
  } else if (b == 0) {
    for (int e = t; e < a.n_tc * kW; e += kDeriveThreads) a.bsq[e] = a.sq[(size_t)(e / kW) * (kW * kW + kW) + kW * kW + e % kW];
  }
}

}  // namespace mpmrom

using namespace mpmrom;



namespace {

size_t dec_smem_bytes(bool split) {
  return 1024 + (split ? 2 : kMaxTC) * kLayerBytes + (split ? 2 : 1) * kLayerBytes +
         (2 * 128 * kXbStride + 128 * 3 + kW * kW0Stride + kW + kMaxTC * kW + 3 * kW) * sizeof(float) +
         sizeof(DecSmemTail);
}

template <int NS>
size_t dec_bf16_smem_bytes(bool train = false) {
  return 1024 + kMaxTC * kLayerBytes + kLayerBytes / 2 + (train ? NS * kLayerBytes : 0) + (3 * 128 * 3 + kW + kMaxTC * kW + 3 * kW + 8) * sizeof(float) +
         sizeof(Bf16Tail);
}

template <int NS>
size_t dec_tc3_smem_bytes() {
  return 1024 + kRing * kAtomBytes + NS * kLayerBytes + (3 * 128 * 3 + kW + kMaxTC * kW + 3 * kW + 8) * sizeof(float) +
         sizeof(Tc3Tail);
}

template <int NS, int MODE>
cudaError_t pipe_limit() {
  const cudaError_t e = cudaFuncSetAttribute(decoder_bf16<NS, MODE, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)dec_bf16_smem_bytes<NS>());
  return e != cudaSuccess ? e
                          : cudaFuncSetAttribute(decoder_tc3<NS, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)dec_tc3_smem_bytes<NS>());
}
template <int NS>
cudaError_t pipe_limit_train() {
  const cudaError_t e = cudaFuncSetAttribute(decoder_bf16<NS, PIPE_TANGENT, true>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)dec_bf16_smem_bytes<NS>(true));
  return e != cudaSuccess ? e
                          : cudaFuncSetAttribute(decoder_bf16<NS, PIPE_IDENTITY, true>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)dec_bf16_smem_bytes<NS>(true));
}
cudaError_t pipe_limits() {
  for (cudaError_t (*f)() : {pipe_limit<1, 0>, pipe_limit<1, 1>, pipe_limit<1, 2>, pipe_limit<1, 3>, pipe_limit<2, 0>,
                             pipe_limit<2, 1>, pipe_limit<2, 2>, pipe_limit<2, 3>, pipe_limit_train<1>, pipe_limit_train<2>})
    if (const cudaError_t e = f(); e != cudaSuccess) return e;
  return cudaSuccess;
}

// decoder_tc3 (fp32) or decoder_bf16 over `tiles` tiles of 128 rows with NS tile slots per CTA.
template <int NS, int MODE>
void pipe_launch(const DecArgs& a, bool fp32, int blocks, cudaStream_t s) {
  if (fp32)
    decoder_tc3<NS, MODE><<<blocks, tc3_threads<NS>(), dec_tc3_smem_bytes<NS>(), s>>>(a);
  else
    decoder_bf16<NS, MODE, false><<<blocks, bf16_threads<NS>(), dec_bf16_smem_bytes<NS>(), s>>>(a);
}
// Rows in (point, kind) order, 32 (whole points) or 31 per lane group, four lane groups per tile; one
// tile per CTA while every tile has an SM of its own (of this caller's share), else two.
void pipe_launch(DecArgs& a, bool fp32, int64_t n_rows, int n_sm, int share, bool secants, cudaStream_t s) {
  a.pipe_U = 32 % a.R == 0 ? 32 : 31;
  const int64_t tiles = (n_rows + 4 * a.pipe_U - 1) / (4 * a.pipe_U);
  const int mode = a.act != 0 ? PIPE_IDENTITY : a.R == 1 ? PIPE_PRIMAL : secants ? PIPE_SECANT : PIPE_TANGENT;
  const bool one = tiles <= share;
  const int blocks = (int)(one ? tiles : std::min<int64_t>((tiles + 1) / 2, n_sm));
  void (*f[2][4])(const DecArgs&, bool, int, cudaStream_t) = {
      {pipe_launch<1, 0>, pipe_launch<1, 1>, pipe_launch<1, 2>, pipe_launch<1, 3>},
      {pipe_launch<2, 0>, pipe_launch<2, 1>, pipe_launch<2, 2>, pipe_launch<2, 3>}};
  f[one ? 0 : 1][mode](a, fp32, blocks, s);
}

size_t dec_f32_smem_bytes() {
  return (size_t)(2 * kW * kF32Rows + 2 * kW * kW + kW0Stride * kW + kW + kMaxTC * kW + 3 * kW) * sizeof(float) +
         kF32Rows * (sizeof(F32Row) + sizeof(int64_t) + sizeof(int));
}

mpm_status refresh_derived_impl(mpm_decoder* dec, cudaStream_t s) {
  if (dec->n_tc == 0) return MPM_OK;
  const DeriveArgs a{dec->params + dec->w_off[0], dec->params + dec->w_off[1], dec->d,       dec->r,
                     dec->n_tc,                   dec->bsq,                    dec->wsqT,    dec->wimg,
                     dec->wimg_lo,                dec->wstream,                dec->w0img};
  decoder_derive<<<16 * dec->n_tc + kDeriveW0, kDeriveThreads, 0, s>>>(a);
  MPM_CUDA_TRY(cudaGetLastError());
  return MPM_OK;
}

}  // namespace

namespace mpmrom {
mpm_status decoder_refresh(mpm_decoder* dec, cudaStream_t s) { return refresh_derived_impl(dec, s); }
// Coordinate and latent widths of a decoder, for code that holds it as an opaque handle.
void decoder_shape(const mpm_decoder* dec, int* d, int* r) {
  *d = dec->d;
  *r = dec->r;
}
// Internal launcher for on-device point sets (used by the reduced-order step).
mpm_status decoder_launch_dev(const mpm_decoder* dec, const float* X, const int32_t* idx, const int32_t* n_dev,
                              int n_rep, int64_t capacity, const float* latents, const float* dirs,
                              const int* kinds, int R, float* out, cudaStream_t s, bool cuda_cores);
}

extern "C" {

mpm_status decoder_create(const decoder_desc* desc, mpm_decoder** out) {
  MPM_CHECK_ARG(desc && out, "null argument");
  *out = nullptr;
  MPM_CHECK_ARG(desc->d == 2 || desc->d == 3, "d must be 2 or 3");
  MPM_CHECK_ARG(desc->r >= 0 && desc->d + desc->r <= 40, "d + r must be <= 40");
  MPM_CHECK_ARG(desc->n_hidden >= 0, "n_hidden >= 0");
  MPM_CHECK_ARG(desc->activation == 0 || desc->activation == 1, "activation: 0 ELU, 1 identity");
  MPM_CHECK_ARG(desc->n_hidden == 0 || desc->width == kW, "hidden width must be 128");
  MPM_CHECK_ARG(desc->n_hidden <= kMaxTC + 1, "at most 5 hidden layers");
  auto* dec = new mpm_decoder();
  dec->d = desc->d;
  dec->r = desc->r;
  dec->width = desc->width;
  dec->n_hidden = desc->n_hidden;
  dec->act = desc->activation;
  dec->n_tc = std::max(0, desc->n_hidden - 1);
  std::vector<int> dims;
  dims.push_back(dec->d + dec->r);
  for (int l = 0; l < dec->n_hidden; ++l) dims.push_back(kW);
  dims.push_back(dec->d);
  int64_t off = 0;
  for (size_t l = 0; l + 1 < dims.size(); ++l) {
    dec->w_off.push_back(off);
    off += (int64_t)dims[l] * dims[l + 1];
    dec->b_off.push_back(off);
    off += dims[l + 1];
  }
  dec->n_params = off;
  int dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&dec->n_sm, cudaDevAttrMultiProcessorCount, dev);
  dec->smem = dec_smem_bytes(false);
  dec->smem_split = dec_smem_bytes(true);
  // one allocation for every buffer of the decoder (each cudaMalloc costs tens of microseconds)
  size_t bytes = 0;
  auto place = [&](size_t n) {
    const size_t at = bytes;
    bytes += (n + 1023) / 1024 * 1024;
    return at;
  };
  const size_t sq = sizeof(float) * dec->n_tc * kW * kW, img = (size_t)dec->n_tc * kLayerBytes;
  const size_t o_params = place(sizeof(float) * dec->n_params), o_norm = place(sizeof(float) * 4 * dec->d);
  const size_t o_status = place(sizeof(uint32_t));
  const size_t o_bsq = place(sizeof(float) * dec->n_tc * kW), o_wsqT = place(sq);
  const size_t o_wimg = place(img), o_wimg_lo = place(img), o_w0img = place(kLayerBytes / 2);
  const size_t o_wstream = place(dec->n_tc > 0 ? (size_t)(3 + 6 * dec->n_tc) * kAtomBytes : 0);
  cudaError_t e = cudaMalloc((void**)&dec->pool, bytes);
  if (e == cudaSuccess) {
    dec->params = (float*)(dec->pool + o_params);
    dec->norm = (float*)(dec->pool + o_norm);
    dec->status = (uint32_t*)(dec->pool + o_status);
    if (dec->n_tc > 0) {
      dec->bsq = (float*)(dec->pool + o_bsq);
      dec->wsqT = (float*)(dec->pool + o_wsqT);
      dec->wimg = dec->pool + o_wimg;
      dec->wimg_lo = dec->pool + o_wimg_lo;
      dec->wstream = dec->pool + o_wstream;
      if (kTcLat + dec->r <= 32) dec->w0img = dec->pool + o_w0img;
    }
  }
  if (e == cudaSuccess) e = cudaMemset(dec->params, 0, sizeof(float) * dec->n_params);
  if (e == cudaSuccess) e = cudaMemset(dec->status, 0, sizeof(uint32_t));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(decoder_tc<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dec->smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(decoder_tc<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dec->smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(decoder_tc<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dec->smem_split);
  if (e == cudaSuccess) e = pipe_limits();
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(decoder_f32<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dec_f32_smem_bytes());
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(decoder_f32<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dec_f32_smem_bytes());
  if (e != cudaSuccess) {
    decoder_destroy(dec);
    return set_error(MPM_ENOMEM, std::string("decoder_create: ") + cudaGetErrorString(e));
  }
  *out = dec;
  return MPM_OK;
}

void decoder_destroy(mpm_decoder* dec) {
  if (!dec) return;
  cudaFree(dec->pool);
  delete dec;
}

int64_t decoder_num_params(const mpm_decoder* dec) { return dec ? dec->n_params : 0; }

mpm_status decoder_set_concurrency(mpm_decoder* dec, int k) {
  MPM_CHECK_ARG(dec, "null decoder");
  MPM_CHECK_ARG(k >= 1, "k >= 1");
  dec->concurrency = k;
  return MPM_OK;
}

mpm_status decoder_set_precision(mpm_decoder* dec, int fp32) {
  MPM_CHECK_ARG(dec, "null decoder");
  MPM_CHECK_ARG(fp32 >= 0 && fp32 <= 2, "precision: 0 BF16, 1 FP32, 2 split BF16");
  dec->fp32 = fp32;
  return MPM_OK;
}

mpm_status decoder_set_params(mpm_decoder* dec, const float* params, const float* norm, void* stream) {
  MPM_CHECK_ARG(dec && params && norm, "null argument");
  cudaStream_t s = (cudaStream_t)stream;
  MPM_CUDA_TRY(cudaMemcpyAsync(dec->params, params, sizeof(float) * dec->n_params, cudaMemcpyDefault, s));
  MPM_CUDA_TRY(cudaMemcpyAsync(dec->norm, norm, sizeof(float) * 4 * dec->d, cudaMemcpyDefault, s));
  return refresh_derived_impl(dec, s);
}

mpm_status decoder_get_params(const mpm_decoder* dec, float* params, float* norm, void* stream) {
  MPM_CHECK_ARG(dec, "null argument");
  cudaStream_t s = (cudaStream_t)stream;
  if (params) MPM_CUDA_TRY(cudaMemcpyAsync(params, dec->params, sizeof(float) * dec->n_params, cudaMemcpyDefault, s));
  if (norm) MPM_CUDA_TRY(cudaMemcpyAsync(norm, dec->norm, sizeof(float) * 4 * dec->d, cudaMemcpyDefault, s));
  return MPM_OK;
}

static mpm_status decoder_launch(const mpm_decoder* dec, const float* X, const int32_t* lat_idx,
                                 const float* latents, const float* dirs, const int32_t* kinds, int R, int64_t n,
                                 float* out, const int32_t* idx, const int32_t* n_dev, int n_rep, cudaStream_t s,
                                 const DecArgs* extra = nullptr, bool cuda_cores = false);

mpm_status decoder_eval(const mpm_decoder* dec, const float* X, const int32_t* lat_idx, const float* latents,
                        const float* dirs, const int32_t* kinds, int R, int64_t n, float* out, void* stream) {
  MPM_CHECK_ARG(dec && kinds, "null argument");
  MPM_CHECK_ARG(n >= 0, "n >= 0");
  if (n == 0) return MPM_OK;
  return decoder_launch(dec, X, lat_idx, latents, dirs, kinds, R, n, out, nullptr, nullptr, 1,
                        (cudaStream_t)stream);
}

static mpm_status decoder_launch(const mpm_decoder* dec, const float* X, const int32_t* lat_idx,
                                 const float* latents, const float* dirs, const int32_t* kinds, int R, int64_t n,
                                 float* out, const int32_t* idx, const int32_t* n_dev, int n_rep, cudaStream_t s,
                                 const DecArgs* extra, bool cuda_cores) {
  MPM_CHECK_ARG(R >= 1 && R <= kMaxR && R <= 128, "R must be in [1, 64]");
  MPM_CHECK_ARG(X && latents && out, "null argument");
  DecArgs a{};
  a.d = dec->d;
  a.r = dec->r;
  a.n_tc = dec->n_tc;
  a.act = dec->act;
  a.linear = dec->n_hidden == 0;
  a.W0 = dec->params + dec->w_off[0];
  a.b0 = dec->params + dec->b_off[0];
  a.bh = dec->bsq;
  const int L = (int)dec->w_off.size();
  a.Wout = dec->params + dec->w_off[L - 1];
  a.bout = dec->params + dec->b_off[L - 1];
  a.norm = dec->norm;
  a.wimg = dec->wimg;
  a.wimg_lo = dec->wimg_lo;
  a.w0img = dec->w0img;
  a.wstream = dec->wstream;
  a.wsqT = dec->wsqT;
  a.X = X;
  a.lat = lat_idx;
  a.latents = latents;
  a.dirs = dirs;
  a.n = n;
  a.R = R;
  a.Pt = 128 / R;
  a.n_dirs = 1;
  bool need_dirs = false, has_mixed = false;
  for (int k = 0; k < R; ++k) {
    const int c = kinds[k];
    const bool mixed = c > KIND_MIXED && c <= KIND_MIXED + dec->d + dec->r;
    const bool secant_dir = c >= KIND_SECANT_DIR && c < KIND_SECANT_DIR + kMaxR;
    MPM_CHECK_ARG(c == KIND_PRIMAL || (c >= 1 && c <= dec->d + dec->r) || c == KIND_JVP || c == KIND_SECANT ||
                      mixed || secant_dir,
                  "unknown row kind");
    need_dirs |= (c == KIND_JVP || c == KIND_SECANT || mixed || secant_dir);
    if (secant_dir) a.n_dirs = std::max(a.n_dirs, c - KIND_SECANT_DIR + 1);
    has_mixed |= mixed;
    a.kinds[k] = c;
    a.mix_jvp[k] = 0;
    a.mix_tan[k] = 0;
    if (mixed) {
      int kj = -1, kt = -1;
      for (int q = 0; q < R; ++q) {
        if (kinds[q] == KIND_JVP && kj < 0) kj = q;
        if (kinds[q] == c - KIND_MIXED && kt < 0) kt = q;
      }
      MPM_CHECK_ARG(kj >= 0 && kt >= 0, "a mixed row needs the JVP row and the tangent row of its input in the call");
      a.mix_jvp[k] = (int8_t)kj;
      a.mix_tan[k] = (int8_t)kt;
    }
  }
  MPM_CHECK_ARG(!need_dirs || dirs, "JVP / secant rows need dirs");
  MPM_CHECK_ARG(kinds[0] == KIND_PRIMAL || dec->n_tc == 0, "the first row kind must be the primal (0)");
  a.out = out;
  a.status = dec->status;
  a.idx = idx;
  a.n_dev = n_dev;
  a.n_rep = n_rep;
  if (extra) {
    a.lat_per_point = extra->lat_per_point;
    a.dstore = extra->dstore;
    a.astore = extra->astore;
    a.rows_total = extra->rows_total;
    a.points_total = extra->points_total;
    MPM_CHECK_ARG(!a.dstore || dec->n_tc > 0, "training stores need square hidden layers");
    MPM_CHECK_ARG(!a.dstore || !has_mixed, "training stores take no mixed rows");
    MPM_CHECK_ARG(!a.dstore || R > 1, "training stores need the tangent rows (R > 1)");
    for (int k = 0; k < R && a.dstore; ++k)
      MPM_CHECK_ARG(a.kinds[k] == KIND_PRIMAL || (a.kinds[k] >= 1 && a.kinds[k] <= dec->d + dec->r) ||
                        a.kinds[k] == KIND_JVP,
                    "training stores take primal, tangent and JVP rows only");
  }
  // the tensor-core kernel's input layout holds r <= 36 latents (decoder_create allows d + r <= 40):
  // larger latents take the FP32 kernel
  const bool f32_path = (dec->fp32 == 1 || dec->r > 40 - kTcLat) && !a.dstore;
  // FP32 calls run on the tensor cores (decoder_tc3) but for mixed rows (their partner rows are not in
  // the row's warp), for callers that keep decoder_f32's rounding, and for calls with secant rows that fit one of
  // decoder_f32's small tiles per SM of the caller's share (256 samples x 12 or 18 rows of a lone caller: 32 us
  // against 40 us; 16 x 12 rows of one of eight callers 33.6 against 41.9, 64 x 12, past it, 55 against 41; without
  // secants, 256 x 17 rows, 31 us against 24 us the other way; 4096 x 4 rows 98 against 25 us)
  const int share = std::max(1, dec->n_sm / std::max(1, dec->concurrency));
  bool secants = false;
  for (int k = 0; k < R; ++k) secants |= kind_class(kinds[k]) == 2;
  const bool pipe = !has_mixed && n * R < ((int64_t)1 << 31) - 4096;   // row numbers and their padding fit 32 bits
  const bool tc3 = f32_path && pipe && !cuda_cores && !(secants && n * R <= 31 * (int64_t)share);
  if (dec->n_tc == 0) {
    int64_t rows = n * R;
    int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((rows + 127) / 128, dec->n_sm * 8));
    decoder_simt<<<blocks, 128, 0, s>>>(a);
  } else if (tc3) {
    pipe_launch(a, true, n * R, dec->n_sm, share, secants, s);
  } else if (f32_path) {
    MPM_CHECK_ARG(R <= kF32Rows, "the FP32 path takes at most 64 row kinds");
    int64_t tiles;
    bool small = false;
    if (has_mixed) {
      // mixed rows read their JVP and tangent partners: point-aligned tiles
      a.f32_U = 0;
      a.Pt = kF32Rows / R;
      tiles = (n + a.Pt - 1) / a.Pt;
    } else {
      // packed tiles: about one per SM (per SM share of the concurrent callers), 32 or 64 slots
      const int64_t rows = n * R;
      const int64_t U = std::max<int64_t>(1, std::min<int64_t>((rows + share - 1) / share, kF32Rows - 1));
      a.f32_U = (int)U;
      a.Pt = 1;
      small = U + 1 <= 32;
      tiles = (rows + U - 1) / U;
    }
    int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(tiles, dec->n_sm));
    if (small)
      decoder_f32<32><<<blocks, kF32Threads, dec_f32_smem_bytes(), s>>>(a);
    else
      decoder_f32<64><<<blocks, kF32Threads, dec_f32_smem_bytes(), s>>>(a);
  } else if (dec->fp32 == 0 && pipe && !a.dstore && dec->w0img) {
    // BF16 rows without partners beyond the primal, first layer on the tensor cores (r <= 28)
    pipe_launch(a, false, n * R, dec->n_sm, dec->n_sm, secants, s);
  } else if (a.dstore && a.points_total > 0) {
    // training on decoder_bf16: whole points per lane group
    a.pipe_U = 32 / R * R;
    const int tiles = (int)(a.rows_total / 128);
    const bool one = tiles <= dec->n_sm;
    const int blocks = one ? tiles : std::min((tiles + 1) / 2, dec->n_sm);
    if (one && a.act == 0)
      decoder_bf16<1, PIPE_TANGENT, true><<<blocks, bf16_threads<1>(), dec_bf16_smem_bytes<1>(true), s>>>(a);
    else if (one)
      decoder_bf16<1, PIPE_IDENTITY, true><<<blocks, bf16_threads<1>(), dec_bf16_smem_bytes<1>(true), s>>>(a);
    else if (a.act == 0)
      decoder_bf16<2, PIPE_TANGENT, true><<<blocks, bf16_threads<2>(), dec_bf16_smem_bytes<2>(true), s>>>(a);
    else
      decoder_bf16<2, PIPE_IDENTITY, true><<<blocks, bf16_threads<2>(), dec_bf16_smem_bytes<2>(true), s>>>(a);
  } else {
    const int64_t tiles = (n + a.Pt - 1) / a.Pt;
    int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(tiles, dec->n_sm));
    if (dec->fp32 == 2 && !a.dstore)
      decoder_tc<true, false><<<blocks, kDecThreads, dec->smem_split, s>>>(a);
    else if (a.dstore)
      decoder_tc<false, true><<<blocks, kDecThreads, dec->smem, s>>>(a);
    else
      decoder_tc<false, false><<<blocks, kDecThreads, dec->smem, s>>>(a);
  }
  MPM_CUDA_TRY(cudaGetLastError());
  return MPM_OK;
}

}  // extern "C"

namespace mpmrom {
// Whether the training forward runs on decoder_bf16 (row-major stores; else decoder_tc's
// feature-major ones).
bool decoder_train_pipe(const mpm_decoder* dec, int64_t rows_total) {
  return dec->n_tc > 0 && dec->w0img != nullptr && rows_total < ((int64_t)1 << 31) - 4096;
}

// Training forward: one latent and one JVP direction per point; stores the
// per-layer activations of every tile row and the primal rows' activation slopes.
mpm_status decoder_launch_train(const mpm_decoder* dec, const float* X, const float* latents, const float* dirs,
                                const int* kinds, int R, int64_t n, float* out, __nv_bfloat16* dstore,
                                __nv_bfloat16* astore, int64_t rows_total, int64_t points_total, cudaStream_t s) {
  DecArgs extra{};
  extra.points_total = points_total;
  extra.lat_per_point = 1;
  extra.dstore = dstore;
  extra.astore = astore;
  extra.rows_total = rows_total;
  return decoder_launch(dec, X, nullptr, latents, dirs, kinds, R, n, out, nullptr, nullptr, 1, s, &extra);
}

mpm_status decoder_launch_dev(const mpm_decoder* dec, const float* X, const int32_t* idx, const int32_t* n_dev,
                              int n_rep, int64_t capacity, const float* latents, const float* dirs,
                              const int* kinds, int R, float* out, cudaStream_t s, bool cuda_cores) {
  if (capacity <= 0) return MPM_OK;
  return decoder_launch(dec, X, nullptr, latents, dirs, kinds, R, capacity, out, idx, n_dev, n_rep, s, nullptr,
                        cuda_cores);
}
}  // namespace mpmrom

extern "C" {

mpm_status decoder_status_word(mpm_decoder* dec, uint32_t* out, int clear, void* stream) {
  MPM_CHECK_ARG(dec && out, "null argument");
  cudaStream_t s = (cudaStream_t)stream;
  uint32_t h = 0;
  MPM_CUDA_TRY(cudaMemcpyAsync(&h, dec->status, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
  if (clear) MPM_CUDA_TRY(cudaMemsetAsync(dec->status, 0, sizeof(uint32_t), s));
  MPM_CUDA_TRY(cudaStreamSynchronize(s));
  *out = h;
  return MPM_OK;
}

}  // extern "C"
