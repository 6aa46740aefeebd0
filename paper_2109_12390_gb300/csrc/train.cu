// Decoder training (Section 4.2 loss, Appendix B optimiser) on sm_103a.
//
// Per minibatch of B (snapshot, particle) pairs, rows per point
// [primal, dg/dX_0 .. dg/dX_{d-1}, JVP along (xhat_{n+1} - xhat_n) / dt_snap]:
//   train_sample     counter-based draw of the pairs (SplitMix64 of
//                    (seed, step, i), uniform over all pairs), gather of X,
//                    latents, JVP directions and targets
//   decoder_bf16     forward (tensor cores), storing every hidden layer's
//                    activations (128-row tiles as MMA images) and the primal
//                    rows' activation slopes (BF16)
//   train_bwd_pipe   loss residuals and output-layer gradients (FP32), then the
//                    reverse sweep: z_bar = act'(z) h_bar + act''(z) sum_j zdot_j t_bar_j
//                    for primal rows, zdot_bar = act'(z) t_bar for tangent rows; for
//                    ELU act''(z) zdot_j = [z < 0] a_j, the tangent row's stored
//                    activation, so the slope record and the activations suffice
//                    (a point's rows sit in one warp: shuffles), next adjoint rows by a
//                    tcgen05 GEMM with the transposed weights resident in shared
//                    memory
//   train_dw_gemm_image  weight gradients of the square layers, dW = Zbar^T A, as
//                    split-K tcgen05 GEMMs over all rows straight from the stored
//                    images, FP32 atomics across splits
//   train_dw0_pipe   first-layer weight gradient (K = d + r) and latent adjoints, FP32
//   (r > 28: decoder_tc, train_bwd_tc, train_dw_gemm and train_dw0_lat, with
//   feature-major activations and adjoints)
//   train_lat_scatter latent-table gradient (snapshot n gets d/dxhat_n of its
//                    own rows and -u_bar / dt; its successor gets +u_bar / dt)
//   train_adam       Adam on the FP32 master parameters and the latent table,
//                    learning rate decaying geometrically lr0 -> lr1
//   + re-pack of the BF16 weight images (forward and transposed)
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "decoder_common.cuh"
#include "encoder.cuh"
#include "pipe.cuh"

namespace mpmrom {
mpm_status decoder_launch_train(const mpm_decoder* dec, const float* X, const float* latents, const float* dirs,
                                const int* kinds, int R, int64_t n, float* out, __nv_bfloat16* dstore,
                                __nv_bfloat16* astore, int64_t rows_total, int64_t points_total, cudaStream_t s);
bool decoder_train_pipe(const mpm_decoder* dec, int64_t rows_total);

__device__ __forceinline__ uint64_t tr_splitmix(uint64_t state, uint64_t k) {
  uint64_t z = state + 0x9E3779B97F4A7C15ull * (k + 1ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}


struct Store {
  int d, r;
  int n_snap;
  const int64_t* snap_base;   // (n_snap + 1) offsets of each snapshot's particle rows
  const int32_t* snap_inst;
  const int32_t* snap_next;
  const int64_t* inst_off;    // particle offsets into X
  const float* X;
  const float* x;
  const float* v;
  const float* F;
};

struct Batch {
  int64_t B;
  float* X;        // (B, d)
  float* xh;       // (B, r)
  float* u;        // (B, r)
  float* tx;       // (B, d)
  float* tv;       // (B, d)
  float* tF;       // (B, d, d)
  float* mask;     // (B)
  int32_t* snap;   // (B)
  int32_t* next;   // (B)
  int32_t* part;   // (B) particle index within its instance
};

// ------------------------------------------------------------- sampler
// A lane draws one point: the pair's position by bisection, then every row it names, all loads before
// the first store (a store might alias the next load, so that interleaved they wait for one another).
// The latent rows are gathered by the warp together, 32 consecutive entries of the batch's rows at a
// time, kGather loads in flight per lane.  Bound by the latency of the bisection; 65,536 points,
// r = 16: 27 us with each point's rows copied entry by entry in its own thread,
// 17 us like this.
constexpr int kGather = 8;

template <int D>
__global__ void __launch_bounds__(128) train_sample(Store st, Batch b, const float* __restrict__ latents,
                                                    float dt_snap, uint64_t seed, const int64_t* step, double* loss,
                                                    int64_t i_offset) {
  const int r = st.r, lane = threadIdx.x & 31;
  const int64_t total = st.snap_base[st.n_snap];
  const uint64_t s0 = tr_splitmix(seed, (uint64_t)*step);
  if (blockIdx.x == 0 && threadIdx.x == 0) *loss = 0.0;
  for (int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x - lane; i0 < b.B;
       i0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = i0 + lane;
    int s = 0, nx = -1;
    if (i < b.B) {
      // draw i_offset + i of the step's minibatch (a data-parallel shard holds a contiguous range)
      const uint64_t h = tr_splitmix(s0, (uint64_t)(i + i_offset));
      const int64_t g = (int64_t)(h % (uint64_t)total);
      // snapshot containing pair g: largest s with snap_base[s] <= g
      int lo = 0, hi = st.n_snap - 1;
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (st.snap_base[mid] <= g) lo = mid;
        else hi = mid - 1;
      }
      s = lo;
      const int64_t local = g - st.snap_base[s];
      const int64_t pidx = st.inst_off[st.snap_inst[s]] + local;
      nx = st.snap_next[s];
      float X[D], x[D], v[D], F[D * D];
#pragma unroll
      for (int a = 0; a < D; ++a) {
        X[a] = st.X[pidx * D + a];
        x[a] = st.x[g * D + a];
        v[a] = st.v[g * D + a];
      }
#pragma unroll
      for (int e = 0; e < D * D; ++e) F[e] = st.F[g * D * D + e];
      b.snap[i] = s;
      b.next[i] = nx;
      b.part[i] = (int32_t)local;
      b.mask[i] = nx >= 0 ? 1.f : 0.f;
#pragma unroll
      for (int a = 0; a < D; ++a) {
        b.X[i * D + a] = X[a];
        b.tx[i * D + a] = x[a];
        b.tv[i * D + a] = v[a];
      }
#pragma unroll
      for (int e = 0; e < D * D; ++e) b.tF[i * D * D + e] = F[e];
    }
    // latents and JVP directions of the warp's points
    const int n = (int)(b.B - i0 < 32 ? b.B - i0 : 32) * r;
    for (int e0 = 0; e0 < n; e0 += 32 * kGather) {
      float xs[kGather], xn[kGather];
      bool next[kGather];
#pragma unroll
      for (int k = 0; k < kGather; ++k) {
        const int e = min(e0 + 32 * k + lane, n - 1), q = e / r, j = e - q * r;
        const int sq = __shfl_sync(0xffffffffu, s, q), nq = __shfl_sync(0xffffffffu, nx, q);
        next[k] = nq >= 0;
        xs[k] = latents[(int64_t)sq * r + j];
        xn[k] = nq >= 0 ? latents[(int64_t)nq * r + j] : 0.f;
      }
#pragma unroll
      for (int k = 0; k < kGather; ++k) {
        const int e = e0 + 32 * k + lane;
        if (e < n) {
          b.xh[i0 * r + e] = xs[k];
          b.u[i0 * r + e] = next[k] ? (xn[k] - xs[k]) / dt_snap : 0.f;
        }
      }
    }
  }
}

// ------------------------------------------------------------- backward
struct BwdArgs {
  float n_norm;   // points of the whole minibatch (over all data-parallel shards)
  int d, r, n_hidden, n_tc, act, R, Pt;
  int64_t n, rows_total, points_total;
  const float* W0;      // (W, d + r)
  const float* Wout;    // (d, W)
  const float* norm;
  const __nv_bfloat16* dstore;   // primal rows' activation slopes (act_slope_record), feature-major
  const __nv_bfloat16* astore;
  const uint8_t* wtimg;
  const float* fwd;     // (R, n, d)
  Batch b;
  float lamF, lamv;
  __nv_bfloat16* zbstore;   // (n_tc, W, rows)
  float* zb0;               // (W, rows)
  float* gparams;
  int64_t gW0_off, gb0_off, gWout_off, gbout_off;
  int64_t gb_off[kMaxTC + 1];   // bias-gradient offsets of hidden layers 0..n_hidden-1
  float* g_lat_pt;          // (n, r)
  float* g_u_pt;            // (n, r)
  double* loss;
  uint32_t* status;
};

constexpr int kExchRows = 104;
constexpr int kBwdMaxR = 5;           // rows per point in training: primal, d <= 3 tangents, JVP
constexpr int kChunkStride = 33;      // padded row stride of one 32-feature chunk: distinct banks

// 256 threads: warps w and w + 4 read the same tensor-memory lane group; thread
// t owns tile row rw = 32 (w % 4) + lane and the feature half h = w / 4
// (features 64 h .. 64 h + 63) of every layer.
constexpr int kBwdThreads = 256;

__global__ void __launch_bounds__(kBwdThreads, 1) train_bwd_tc(BwdArgs a) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* wt = smem;                                 // n_tc x 32 KB (transposed square weights)
  uint8_t* atile = smem + kMaxTC * kLayerBytes;       // 32 KB
  float* exch = (float*)(atile + kLayerBytes);        // [2 halves][kExchRows][33]: tangent-row terms of the chunk
  __nv_bfloat16* sD = (__nv_bfloat16*)(exch + 2 * kExchRows * kChunkStride);  // [64 f][128 rows] slopes
  __nv_bfloat16* sA = sD + 64 * 128;                  // [64 f][128 rows] activations (f: 32 h + feature of chunk)
  float* sy = (float*)(sA + 64 * 128);                // 128 x 3
  float* sbias = sy + 128 * 3;                        // 128
  DecSmemTail* tail = (DecSmemTail*)(sbias + kW);
  __shared__ double s_loss[8];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int rw = (warp & 3) * 32 + lane;              // tile row / tensor-memory lane
  const int h = warp >> 2;                            // feature half
  const int d = a.d, R = a.R, Pt = a.Pt;

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
  if (t == 0 && a.n_tc > 0) {
    tc::mbar_expect_tx(&tail->bar_w, (uint32_t)(a.n_tc * kLayerBytes));
    for (int l = 0; l < a.n_tc; ++l)
      tc::bulk_g2s(wt + l * kLayerBytes, a.wtimg + (size_t)l * kLayerBytes, kLayerBytes, &tail->bar_w);
  }
  if (a.n_tc > 0 && !tc::mbar_wait(&tail->bar_w, 0)) {
    raise_status(a.status, STATUS_TIMEOUT);
    atomicExch(&tail->abort, 1);
  }
  if (t < kW) sbias[t] = 0.f;
  __syncthreads();
  constexpr uint32_t idesc = tc::idesc_bf16_f32(128, kW);
  uint32_t mma_phase = 0;
  const int64_t n_tiles = (a.n + Pt - 1) / Pt;
  const float* scale = a.norm + 3 * d;
  double my_loss = 0.0;

  for (int64_t tile = blockIdx.x; tile < n_tiles && !tail->abort; tile += gridDim.x) {
    const int64_t row0 = tile * 128;
    const int k = rw / Pt, q = rw % Pt;
    const int64_t p = tile * Pt + q;
    const bool valid = (k < R) && (p < a.n);
    const int cls = !valid ? -1 : (k == 0 ? 0 : 1);
    const int64_t gr = row0 + rw;
    // the slopes and activations of step i2z of layer lz (chunk 2 hh + i2z of each half hh),
    // copied asynchronously into the staging buffers in 16-byte pieces (8 rows of one feature) one
    // step ahead of their use, so that the loads overlap the current step: the activations of the
    // tile's 128 rows, the slope records of its first 32 rows only (the primal rows, Pt <= 32)
    auto prefetch_z = [&](int lz, int i2z) {
#pragma unroll
      for (int k2 = 0; k2 < 5; ++k2) {
        const int w = t + kBwdThreads * k2;                    // 64 features x (16 + 4) pieces
        const bool act = w < 64 * 16;
        const int fl = act ? w >> 4 : (w - 64 * 16) >> 2, c8 = act ? w & 15 : w & 3;
        const int fg = (2 * (fl >> 5) + i2z) * 32 + (fl & 31);   // global feature
        const __nv_bfloat16* src = (act ? a.astore : a.dstore) + ((int64_t)lz * kW + fg) * a.rows_total + row0 + 8 * c8;
        cp_async16((act ? sA : sD) + fl * 128 + 8 * c8, src);
      }
      cp_async_commit();
    };
    prefetch_z(a.n_hidden - 1, 0);
    // ---- output layer: residual adjoints ybar (FP32)
    float ybar[3] = {0.f, 0.f, 0.f};
    if (valid) {
      const float* o = a.fwd + ((int64_t)k * a.n + p) * d;
      // loops over the d <= 3 output components have compile-time bounds: with the runtime bound
      // the small register arrays they index (ybar, acc) are placed in local memory
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        if (i >= d) break;
        float e, w;
        if (k == 0) {
          e = o[i] - a.b.tx[p * d + i];
          w = 1.f;
        } else if (k <= d) {
          e = o[i] - a.b.tF[(p * d + i) * d + (k - 1)];
          w = a.lamF;
        } else {
          e = a.b.mask[p] * (o[i] - a.b.tv[p * d + i]);
          w = a.lamv;
        }
        if (h == 0) my_loss += (double)w * e * e;
        ybar[i] = 2.f * w * e * scale[i] / a.n_norm;
      }
    }
    if (h == 0)
      for (int i = 0; i < 3; ++i) sy[rw * 3 + i] = ybar[i];
    __syncthreads();
    {
      // dWout[i][f] = sum_rows ybar_i a_last[f]: thread = feature f = t % 128, rows 64 (t / 128) ..
      const int f = t & 127, rh = t >> 7;
      const __nv_bfloat16* al = a.astore + (int64_t)(a.n_hidden - 1) * kW * a.rows_total + (int64_t)f * a.rows_total +
                                row0 + 64 * rh;
      float acc[3] = {0.f, 0.f, 0.f};
      // unrolled: the eight 16-byte loads of the stored activations are in flight together
#pragma unroll
      for (int c = 0; c < 64; c += 8) {
        const uint4 u = *reinterpret_cast<const uint4*>(al + c);
        const __nv_bfloat16* hv = reinterpret_cast<const __nv_bfloat16*>(&u);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const float av = __bfloat162float(hv[j]);
#pragma unroll
          for (int i = 0; i < 3; ++i)
            if (i < d) acc[i] = fmaf(sy[(64 * rh + c + j) * 3 + i], av, acc[i]);
        }
      }
#pragma unroll
      for (int i = 0; i < 3; ++i)
        if (i < d) atomicAdd(&a.gparams[a.gWout_off + i * kW + f], acc[i]);
      if (t < d) {
        float sb = 0.f;
        for (int q2 = 0; q2 < Pt; ++q2) sb += sy[q2 * 3 + t];
        atomicAdd(&a.gparams[a.gbout_off + t], sb);
      }
    }
    // ---- reverse sweep over the hidden layers
    for (int l = a.n_hidden - 1; l >= 0; --l) {
      const bool from_tmem = (l < a.n_hidden - 1);
      if (from_tmem) {
        if (!tc::mbar_wait(&tail->bar_mma, mma_phase)) {
          raise_status(a.status, STATUS_TIMEOUT);
          atomicExch(&tail->abort, 1);
        }
        mma_phase ^= 1u;
        tc::tc_fence_after();
      }
      cp_async_wait_all();   // this thread's staging copies of the step have landed
      __syncthreads();
      if (tail->abort) break;
      for (int i2 = 0; i2 < 2; ++i2) {
        const int ch = 2 * h + i2;
        float hb[32];
        if (from_tmem) {
          tc::tmem_ld32(tmem + ((uint32_t)((warp & 3) * 32) << 16) + ch * 32, hb);
        } else {
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            float sacc = 0.f;
#pragma unroll
            for (int o = 0; o < 3; ++o)
              if (o < d) sacc = fmaf(__ldg(&a.Wout[o * kW + ch * 32 + i]), ybar[o], sacc);
            hb[i] = sacc;
          }
        }
        float zb[32];
        // the point's primal slope record s (row q): act'(z) = s, or 1 where s < 0; for tangent
        // rows the curvature term act''(z) zdot is the row's own activation where s >= 0 (z < 0)
        float sown[32];
        const __nv_bfloat16* hD = sD + (h * 32) * 128;
        const __nv_bfloat16* hA = sA + (h * 32) * 128;
        if (cls == 0) {   // before the barrier: the staging buffer is refilled after it
#pragma unroll
          for (int i = 0; i < 32; ++i) sown[i] = __bfloat162float(hD[i * 128 + rw]);
        }
        float* hexch = exch + h * kExchRows * kChunkStride;
        if (cls == 1) {
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const float sp = __bfloat162float(hD[i * 128 + q]);
            const float at = __bfloat162float(hA[i * 128 + rw]);
            zb[i] = (sp < 0.f ? 1.f : sp) * hb[i];
            hexch[(rw - Pt) * kChunkStride + i] = (sp >= 0.f ? at : 0.f) * hb[i];
          }
        }
        __syncthreads();
        // every row has read the staged step: stage the next one (this layer's other chunk of
        // each half, or the next layer's first)
        if (i2 == 0) prefetch_z(l, 1);
        else if (l > 0) prefetch_z(l - 1, 0);
        if (cls == 0) {
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            float sacc = (sown[i] < 0.f ? 1.f : sown[i]) * hb[i];
            // compile-time bound (R <= kBwdMaxR): with the runtime bound this loop, inside the
            // unrolled feature loop, ran about 1,000 cycles per feature
#pragma unroll
            for (int kk = 1; kk < kBwdMaxR; ++kk)
              if (kk < R) sacc += hexch[((kk - 1) * Pt + q) * kChunkStride + i];
            zb[i] = sacc;
          }
        } else if (cls < 0) {
#pragma unroll
          for (int i = 0; i < 32; ++i) zb[i] = 0.f;
        }
        // bias gradient: sum of the primal rows' z_bar (primal rows all sit in lane group 0);
        // transpose-reduce the 32 columns across the warp so lane i ends with column i
        if ((warp & 3) == 0) {
          float v[32];
#pragma unroll
          for (int i = 0; i < 32; ++i) v[i] = (cls == 0) ? zb[i] : 0.f;
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            const bool up = (lane & o) != 0;
#pragma unroll
            for (int i = 0; i < o; ++i) {
              // lanes with bit o set keep the upper half of the columns, the others the lower half
              const float send = up ? v[i] : v[i + o];
              const float keep = up ? v[i + o] : v[i];
              v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
          }
          sbias[ch * 32 + lane] += v[0];
        }
        if (l >= 1) {
#pragma unroll
          for (int j = 0; j < 32; j += 8) store_bf16x8(atile, rw, ch * 32 + j, zb + j);
        } else {
          // first-layer adjoints (FP32); the first-layer weight gradient and the latent
          // adjoints are formed from them by train_dw0_lat
          float* zs = a.zb0 + gr;
#pragma unroll
          for (int i = 0; i < 32; ++i) zs[(int64_t)(ch * 32 + i) * a.rows_total] = zb[i];
        }
        if (i2 == 0) cp_async_wait_all();   // the next chunk's staging has landed
        __syncthreads();
      }
      // bias gradient of layer l (sbias was filled before the last barrier)
      if (t < kW) {
        atomicAdd(&a.gparams[a.gb_off[l] + t], sbias[t]);
        sbias[t] = 0.f;
      }
      if (l >= 1) {
        // next adjoint rows: h_bar_{l-1} = z_bar_l W_l  (B operand = W_l^T image)
        tc::fence_async_smem();
        tc::tc_fence_before();
        __syncthreads();
        if (t == 0) {
          tc::tc_fence_after();
          const uint32_t a_base = tc::smem_addr(atile), b_base = tc::smem_addr(wt + (l - 1) * kLayerBytes);
#pragma unroll
          for (int kk = 0; kk < kW / 16; ++kk) {
            const uint32_t koff = (uint32_t)((kk >> 2) * (kW * 128) + (kk & 3) * 32);
            tc::mma_bf16(tmem, tc::smem_desc_sw128(a_base + koff), tc::smem_desc_sw128(b_base + koff), idesc,
                         kk > 0 ? 1u : 0u);
          }
          tc::mma_commit(&tail->bar_mma);
        }
        // the adjoints of layer l (BF16, for the weight-gradient GEMMs) leave the operand tile while
        // the tensor core reads it; the barrier after the next wait orders these reads before the
        // next writes of the tile
        copy_out_tile(a.zbstore + (int64_t)(l - 1) * kW * a.rows_total, a.rows_total, atile, tile, t);
      }
    }
    if (tail->abort) break;
    tc::tc_fence_before();
    __syncthreads();
  }
  // loss (sum over rows of w e^2; the caller divides by n)
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) my_loss += __shfl_down_sync(0xffffffffu, my_loss, o);
  if ((t & 31) == 0) s_loss[warp] = my_loss;
  __syncthreads();
  if (t == 0) {
    double tot = 0.0;
    for (int w = 0; w < kBwdThreads / 32; ++w) tot += s_loss[w];
    atomicAdd(a.loss, tot);
  }
  cp_async_wait_all();   // no staging copy outlives the CTA (an aborted sweep)
  tc::tc_fence_after();
  if (warp == 0) tc::tmem_free<kW>(tmem);
}

// --------------------------------------------------------------------------
// Backward over decoder_bf16's stores (train_bwd_pipe): the reverse sweep of train_bwd_tc with the same
// arithmetic per row, on the alternating-tile pipeline.  A lane group of 32 rows holds whole points (R
// consecutive lanes each), so a point's curvature terms reach its primal row by shuffles, in the order
// of its tangent rows.  Per (tile slot, layer) the slot's 32 KB activation image and its points' slope
// records arrive by bulk copies; a thread takes 32 columns of its row: adjoint from tensor memory (or,
// for the last hidden layer, Wout^T ybar), and writes the new adjoint over the activation it read.
// The image then is the MMA's operand and is stored by one bulk copy for the weight-gradient GEMM.
// Bias gradients: the primal rows' adjoints pass through a small per-warp buffer and are summed per
// column; output-layer gradients likewise per column and warp; both kept on chip over all tiles of
// the CTA.
// --------------------------------------------------------------------------
constexpr int kBwdPipeThreads = kEpiThreads + 64;

struct __align__(8) BwdPipeTail {
  uint64_t bar_w;
  uint64_t full[2];
  uint64_t bar_mma[2];
  uint64_t drain;
  uint32_t tmem;
  int abort;
};

size_t bwd_pipe_smem_bytes() {
  return 1024 + kMaxTC * kLayerBytes + 2 * kLayerBytes + 2 * 32 * 256 +
         (16 * 8 * 8 + 16 * (kMaxTC + 1) * 32 + 3 * kW) * sizeof(float) + sizeof(BwdPipeTail);
}

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

// 16 columns of four neighbouring lanes' rows, transposed by blocks of four: lane j of the four gets columns
// 4 j .. 4 j + 3, row q's at v[4 q ..].
__device__ __forceinline__ void quad_transpose(float (&v)[16], int j) {
#pragma unroll
  for (int x = 1; x < 4; x <<= 1) {
    const bool up = (j & x) != 0;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      if ((i >> 2) & x) continue;
      const float got = __shfl_xor_sync(0xffffffffu, up ? v[i] : v[i + 4 * x], x);
      v[i] = up ? got : v[i];
      v[i + 4 * x] = up ? v[i + 4 * x] : got;
    }
  }
}

template <int D>
__global__ void __launch_bounds__(kBwdPipeThreads, 1) train_bwd_pipe(BwdArgs a) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (tc::smem_addr(smem_raw) & 1023u)) & 1023u);
  uint8_t* wt = smem;                                    // kMaxTC x 32 KB transposed square weights
  uint8_t* images = wt + kMaxTC * kLayerBytes;           // [2 slots] activation, then adjoint images
  uint8_t* slopes = images + 2 * kLayerBytes;            // [2 slots][32 points][256 B] slope records
  float* scratch = (float*)(slopes + 2 * 32 * 256);      // [16 warps][8 primal rows][8 columns]
  float* sbias = scratch + 16 * 8 * 8;                   // [16 warps][hidden layers][32 columns]
  float* sWout = sbias + 16 * (kMaxTC + 1) * 32;         // [3][128]
  BwdPipeTail* tail = (BwdPipeTail*)(sWout + 3 * kW);
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  constexpr int d = D, R = D + 2;
  constexpr int ppg = 32 / R, U = ppg * R;               // points and rows per lane group

  if (t == 0) {
    tc::mbar_init(&tail->bar_w, 1);
    tc::mbar_init(&tail->full[0], 1);
    tc::mbar_init(&tail->full[1], 1);
    tc::mbar_init(&tail->bar_mma[0], 1);
    tc::mbar_init(&tail->bar_mma[1], 1);
    tc::mbar_init(&tail->drain, 2);
    tail->abort = 0;
    tc::fence_mbar_init();
    tc::mbar_expect_tx(&tail->bar_w, (uint32_t)(a.n_tc * kLayerBytes));
    for (int l = a.n_tc - 1; l >= 0; --l)
      tc::bulk_g2s(wt + l * kLayerBytes, a.wtimg + (size_t)l * kLayerBytes, kLayerBytes, &tail->bar_w);
  }
  if (warp == 0) tc::tmem_alloc<512>(&tail->tmem);
  for (int e = t; e < 16 * (kMaxTC + 1) * 32; e += kBwdPipeThreads) sbias[e] = 0.f;
  for (int e = t; e < 3 * kW; e += kBwdPipeThreads) sWout[e] = e < d * kW ? a.Wout[e] : 0.f;
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();

  const int n_tiles = (int)(a.rows_total / 128);
  const int NT = n_tiles <= (int)gridDim.x ? 1 : 2;      // tiles per pass
  const int n_iter = (n_tiles + NT - 1) / NT;

  if (warp >= kEpiThreads / 32) {
    // ---- slot s's copies and MMAs (adjoint of the layer below: z_bar W, B operand the W^T image)
    const int s = warp - kEpiThreads / 32;
    const bool leader = tc::elect_one();
    const uint32_t tD = tail->tmem + (uint32_t)(s * 256);
    uint8_t* image = images + s * kLayerBytes;
    uint8_t* slope = slopes + s * 32 * 256;
    const uint32_t a_desc = tc::smem_desc_sw128_lo(tc::smem_addr(image));
    const uint32_t w_desc = tc::smem_desc_sw128_lo(tc::smem_addr(wt));
    constexpr uint32_t idesc = tc::idesc_bf16_f32(128, kW);
    const uint32_t slope_bytes = (uint32_t)(4 * ppg * 256);
    uint32_t mma_phase = 0;
    Refill fill;                                         // the slot's fetches (the same in every lane)
    // activations and slopes of layer l of a tile into the slot
    auto fetch = [&](int tile, int l) {
      if (!fill.start() || !leader) return;
      tc::mbar_expect_tx(&tail->full[s], (uint32_t)kLayerBytes + slope_bytes);
      tc::bulk_g2s(image, a.astore + ((int64_t)l * a.rows_total + (int64_t)tile * 128) * kW, kLayerBytes,
                   &tail->full[s]);
      tc::bulk_g2s(slope, a.dstore + ((int64_t)l * a.points_total + (int64_t)tile * 4 * ppg) * kW, slope_bytes,
                   &tail->full[s]);
    };
    pipe_wait(a.status, &tail->abort, &tail->bar_w, 0);
    __syncwarp();
    for (int it = blockIdx.x; it < n_iter; it += gridDim.x) {
      const int tile = it * NT + s;
      if (s >= NT || tile >= n_tiles) continue;
      if (fill.n == 0) fetch(tile, a.n_hidden - 1);
      for (int l = a.n_hidden - 1; l >= 0; --l) {
        __syncwarp();
        const bool landed = fill.live && pipe_wait(a.status, &tail->abort, &tail->full[s], fill.last_phase());
        fill.seen(__all_sync(0xffffffffu, landed));
        tc::tc_fence_after();
        tc::tc_fence_before();
        pipe_arrive(3 + s);                              // data and (below the last layer) adjoints are there
        pipe_sync(1 + s);                                // the epilogue has replaced them by the new adjoints
        tc::tc_fence_after();
        if (l >= 1) {
          if (leader) {
            const uint32_t bd = w_desc + (uint32_t)(l - 1) * (kLayerBytes >> 4);
            tc::mma4_bf16_ss(tD, a_desc, bd, idesc, 0u);
            tc::mma4_bf16_ss(tD, a_desc + (kAtomBytes >> 4), bd + (kAtomBytes >> 4), idesc, 1u);
            tc::mma_commit(&tail->bar_mma[s]);
            tc::bulk_s2g(a.zbstore + ((int64_t)(l - 1) * a.rows_total + (int64_t)tile * 128) * kW, image, kLayerBytes);
          }
          __syncwarp();
          pipe_wait(a.status, &tail->abort, &tail->bar_mma[s], mma_phase);
          mma_phase ^= 1u;
          if (leader) tc::bulk_wait_read();
          fetch(tile, l - 1);
        } else {
          const int next = (it + (int)gridDim.x) * NT + s;
          if (it + (int)gridDim.x < n_iter && next < n_tiles) fetch(next, a.n_hidden - 1);
        }
      }
    }
    // nothing is in flight when the memory is freed: the stores, and after a timeout (bounded) the
    // MMAs, the weights and the last fetch
    if (leader) {
      tc::bulk_wait_all();
      tc::mma_commit(&tail->drain);
    }
    __syncwarp();
    (void)tc::mbar_wait(&tail->drain, 0);
    if (*(volatile int*)&tail->abort) (void)tc::mbar_wait(&tail->bar_w, 0);
    if (!fill.live) (void)tc::mbar_wait(&tail->full[s], fill.last_phase());
    __syncwarp();
  } else {
    const int h = warp >> 2, lg = warp & 3;
    const int rw = lg * 32 + lane;                       // tile row / tensor-memory lane
    const uint32_t tbase = tail->tmem + ((uint32_t)(lg * 32) << 16);
    const int q = min(lane / R, ppg - 1), k = lane - (lane / R) * R;   // point within the group, row kind
    const bool prim = lane < U && k == 0;
    float* wscratch = scratch + warp * 64;
    float* wbias = sbias + warp * (kMaxTC + 1) * 32;
    double my_loss = 0.0;
    float gwo[3] = {0.f, 0.f, 0.f}, gbo[3] = {0.f, 0.f, 0.f};
    float yb[2][3];                                      // output adjoints of the two slots' rows
    const float wk = k == 0 ? 1.f : k <= d ? a.lamF : a.lamv;

    // output and target of the thread's row (loads only)
    auto residual_load = [&](int tile, float (&o)[3], float (&g)[3], float& m) {
      const int p = (tile * 4 + lg) * ppg + q;
      const bool live = lane < U && p < a.n;
      m = live ? 1.f : 0.f;
      if (live && k > d) m = a.b.mask[p];
      const float* src = a.fwd + ((int64_t)k * a.n + p) * d;
      const float* tgt = k == 0 ? a.b.tx + (int64_t)p * d : k <= d ? a.b.tF + (int64_t)p * d * d + (k - 1) : a.b.tv + (int64_t)p * d;
      const int step = (k >= 1 && k <= d) ? d : 1;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        o[i] = live && i < d ? src[i] : 0.f;
        g[i] = live && i < d ? tgt[i * step] : 0.f;
      }
    };
    // output adjoints and, once per row, the loss
    auto residual = [&](const float (&o)[3], const float (&g)[3], float m, float (&y)[3]) {
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const float e = k > d ? m * (o[i] - g[i]) : o[i] - g[i];
        if (h == 0 && i < d) my_loss += (double)wk * e * e;
        y[i] = i < d ? 2.f * wk * e * a.norm[3 * d + i] / a.n_norm : 0.f;
      }
    };

#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const int tile = blockIdx.x * NT + s;
      if ((int)blockIdx.x < n_iter && s < NT && tile < n_tiles) {
        float o[3], g[3], m;
        residual_load(tile, o, g, m);
        residual(o, g, m, yb[s]);
      }
    }
    for (int it = blockIdx.x; it < n_iter; it += gridDim.x) {
      for (int l = a.n_hidden - 1; l >= 0; --l) {
        const bool top = l == a.n_hidden - 1;
#pragma unroll 1
        for (int s = 0; s < 2; ++s) {
          const int tile = it * NT + s;
          if (s >= NT || tile >= n_tiles) break;
          const uint32_t ts = tbase + s * 256;
          uint8_t* image = images + s * kLayerBytes;
          const uint8_t* slope = slopes + s * 32 * 256;
          const int64_t grow = (int64_t)tile * 128 + rw;
          const float y0 = s == 0 ? yb[0][0] : yb[1][0], y1 = s == 0 ? yb[0][1] : yb[1][1];
          const float y2 = s == 0 ? yb[0][2] : yb[1][2];
          // the slot's next tile: its outputs and targets load while this step waits
          float ro[3], rg[3], rm;
          const int next = (it + (int)gridDim.x) * NT + s;
          const bool more = l == 0 && it + (int)gridDim.x < n_iter && next < n_tiles;
          if (more) residual_load(next, ro, rg, rm);
          pipe_sync(3 + s);
          tc::tc_fence_after();
          if (top) {
            // output layer: dWout[i][c] += sum over the warp's rows of ybar_i a[c], column c = lane
#pragma unroll 8
            for (int r2 = 0; r2 < 32; ++r2) {
              const float av = __uint_as_float(
                  (uint32_t)*reinterpret_cast<const uint16_t*>(image + tc::sw128_offset(lg * 32 + r2, 32 * h + lane, kW)) << 16);
              gwo[0] = fmaf(__shfl_sync(0xffffffffu, y0, r2), av, gwo[0]);
              gwo[1] = fmaf(__shfl_sync(0xffffffffu, y1, r2), av, gwo[1]);
              if (d == 3) gwo[2] = fmaf(__shfl_sync(0xffffffffu, y2, r2), av, gwo[2]);
            }
            if (prim && h == 0) {
              gbo[0] += y0;
              gbo[1] += y1;
              gbo[2] += y2;
            }
            __syncwarp();   // every lane has read the warp's rows before they are replaced
          }
#pragma unroll 1
          for (int c0 = 32 * h; c0 < 32 * h + 32; c0 += 16) {
            float z[16];
            if (top) {
#pragma unroll
              for (int i = 0; i < 16; ++i) {
                float sacc = fmaf(sWout[c0 + i], y0, 0.f);
                sacc = fmaf(sWout[kW + c0 + i], y1, sacc);
                if (d == 3) sacc = fmaf(sWout[2 * kW + c0 + i], y2, sacc);
                z[i] = sacc;
              }
            } else {
              tc::tmem_ld16(ts + c0, z);
            }
            // slope s: act'(z) = s, or 1 where s < 0; the curvature term of a tangent row is its own
            // activation where s >= 0; the primal row adds its point's terms
            uint4* own0 = reinterpret_cast<uint4*>(image + tc::sw128_offset(rw, c0, kW));
            uint4* own1 = reinterpret_cast<uint4*>(image + tc::sw128_offset(rw, c0 + 8, kW));
            uint32_t sw[8], aw[8];
            {
              const uint4 v0 = *reinterpret_cast<const uint4*>(slope + stage_chunk(lg * ppg + q, c0 / 8));
              const uint4 v1 = *reinterpret_cast<const uint4*>(slope + stage_chunk(lg * ppg + q, c0 / 8 + 1));
              const uint4 u0 = *own0, u1 = *own1;
              sw[0] = v0.x, sw[1] = v0.y, sw[2] = v0.z, sw[3] = v0.w, sw[4] = v1.x, sw[5] = v1.y, sw[6] = v1.z, sw[7] = v1.w;
              aw[0] = u0.x, aw[1] = u0.y, aw[2] = u0.z, aw[3] = u0.w, aw[4] = u1.x, aw[5] = u1.y, aw[6] = u1.z, aw[7] = u1.w;
            }
            // The sum goes in the order of the rows, as train_bwd_tc adds them: it is rounded to BF16 next, and
            // another order falls on the other side of a rounding here and there (pairwise sums moved the
            // latent gradients of 2,105 points by 3e-5).  R = 4: the four lanes of a point take four columns each
            // of its primal row, 16 shuffles per 16 columns; R = 5: the primal lane adds what it is sent, a
            // shuffle per column and tangent row.  Gradients of 65,536 points, R = 4: 635 us; 709 with the
            // R = 5 form, whose 48 shuffles then set the time; 679 with pairwise sums.
            float term[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const float sp = (i & 1) ? bf16_hi(sw[i / 2]) : bf16_lo(sw[i / 2]);
              const float at = (i & 1) ? bf16_hi(aw[i / 2]) : bf16_lo(aw[i / 2]);
              const float zb = (sp < 0.f ? 1.f : sp) * z[i];
              term[i] = prim ? zb : (sp >= 0.f ? at : 0.f) * z[i];
              z[i] = zb;
              if (R == 5) {
                float sum = term[i];
#pragma unroll
                for (int j = 1; j < R; ++j) sum += __shfl_down_sync(0xffffffffu, term[i], j);
                z[i] = prim ? sum : zb;
              }
            }
            float p4[4];                                 // R = 4: columns 4 k .. 4 k + 3 of the point's primal row
            if (R == 4) {
              quad_transpose(term, k);
#pragma unroll
              for (int c = 0; c < 4; ++c) p4[c] = ((term[c] + term[4 + c]) + term[8 + c]) + term[12 + c];
            }
            // bias gradients: the primal rows' adjoints summed per column (column lane % 8, the rows
            // in four parts)
#pragma unroll
            for (int c = 0; c < 16; c += 8) {
              __syncwarp();
              if (R == 4 && (k >> 1) == c / 8)
                *reinterpret_cast<float4*>(wscratch + q * 8 + 4 * (k & 1)) = make_float4(p4[0], p4[1], p4[2], p4[3]);
              if (R == 5 && prim) {
                float4* o = reinterpret_cast<float4*>(wscratch + q * 8);
                o[0] = make_float4(z[c], z[c + 1], z[c + 2], z[c + 3]);
                o[1] = make_float4(z[c + 4], z[c + 5], z[c + 6], z[c + 7]);
              }
              __syncwarp();
              float v = 0.f;
#pragma unroll
              for (int pr = 0; pr < ppg; pr += 4)
                if (pr + 4 <= ppg || pr + (lane >> 3) < ppg) v += wscratch[(pr + (lane >> 3)) * 8 + (lane & 7)];
              v += __shfl_xor_sync(0xffffffffu, v, 8);
              v += __shfl_xor_sync(0xffffffffu, v, 16);
              if (lane < 8) wbias[l * 32 + (c0 & 31) + c + lane] += v;
            }
            if (l >= 1) {
              auto pack2 = [](float v0, float v1) {
                const __nv_bfloat162 b2 = __floats2bfloat162_rn(v0, v1);
                return *reinterpret_cast<const uint32_t*>(&b2);
              };
              if (R == 5 || k > 0) {
                uint32_t w[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) w[j] = pack2(z[2 * j], z[2 * j + 1]);
                *own0 = make_uint4(w[0], w[1], w[2], w[3]);
                *own1 = make_uint4(w[4], w[5], w[6], w[7]);
              }
              if (R == 4)   // the primal row (nothing of its columns is read after the barrier of the bias sums)
                *reinterpret_cast<uint2*>(image + tc::sw128_offset(rw - k, c0 + 4 * k, kW)) =
                    make_uint2(pack2(p4[0], p4[1]), pack2(p4[2], p4[3]));
            } else if (R == 4) {
              // first-layer adjoints (FP32, row-major): the point's four lanes exchange their 16 columns so that
              // each store of the warp writes 64 contiguous bytes of eight rows
              quad_transpose(z, k);
#pragma unroll
              for (int c = 0; c < 4; ++c) z[c] = p4[c];
#pragma unroll
              for (int r4 = 0; r4 < 4; ++r4)
                *reinterpret_cast<float4*>(a.zb0 + (grow - k + r4) * kW + c0 + 4 * k) =
                    make_float4(z[4 * r4], z[4 * r4 + 1], z[4 * r4 + 2], z[4 * r4 + 3]);
            } else {
              // the same by four neighbouring lanes, whatever their points
              const int j = lane & 3;
              quad_transpose(z, j);
#pragma unroll
              for (int r4 = 0; r4 < 4; ++r4)
                *reinterpret_cast<float4*>(a.zb0 + (grow - j + r4) * kW + c0 + 4 * j) =
                    make_float4(z[4 * r4], z[4 * r4 + 1], z[4 * r4 + 2], z[4 * r4 + 3]);
            }
          }
          tc::fence_async_smem();
          tc::tc_fence_before();
          pipe_arrive(1 + s);
          if (more) {
            float y[3];
            residual(ro, rg, rm, y);
#pragma unroll
            for (int i = 0; i < 3; ++i) {
              if (s == 0) yb[0][i] = y[i];
              else yb[1][i] = y[i];
            }
          }
        }
      }
    }
    // gradients of the output layer (column 32 h + lane) and of the biases
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      if (i >= d) break;
      atomicAdd(&a.gparams[a.gWout_off + i * kW + 32 * h + lane], gwo[i]);
      float v = gbo[i];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0 && h == 0) atomicAdd(&a.gparams[a.gbout_off + i], v);
    }
    __syncwarp();
    for (int l = 0; l < a.n_hidden; ++l) atomicAdd(&a.gparams[a.gb_off[l] + 32 * h + lane], wbias[l * 32 + lane]);
    if (h == 0) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) my_loss += __shfl_down_sync(0xffffffffu, my_loss, o);
      if (lane == 0) atomicAdd(a.loss, my_loss);
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  if (warp == 0) tc::tmem_free<512>(tail->tmem);
}

// ------------------------------------------- weight gradients (split-K GEMM)
// dW_l[out][in] = sum_rows Zbar[out][row] A[in][row]; Zbar = zbstore[l], A = astore[l]
// (the activations entering square layer l + 1).  Grid (n_tc, splits), 128 threads. 
__global__ void __launch_bounds__(128, 1) train_dw_gemm(const __nv_bfloat16* zbstore, const __nv_bfloat16* astore,
                                                        int64_t rows_total, int64_t k_per_split, float* gparams,
                                                        const int64_t* w_off, uint32_t* status) {
  __shared__ __align__(1024) uint8_t sA[kW * 128];
  __shared__ __align__(1024) uint8_t sB[kW * 128];
  __shared__ uint64_t bar;
  __shared__ uint32_t tslot;
  __shared__ int abort_flag;
  const int t = threadIdx.x, warp = t >> 5;
  const int l = blockIdx.x;
  const __nv_bfloat16* Z = zbstore + (int64_t)l * kW * rows_total;
  const __nv_bfloat16* A = astore + (int64_t)l * kW * rows_total;
  const int64_t k0 = (int64_t)blockIdx.y * k_per_split;
  const int64_t k1 = min(rows_total, k0 + k_per_split);
  if (t == 0) {
    tc::mbar_init(&bar, 1);
    abort_flag = 0;
    tc::fence_mbar_init();
  }
  if (warp == 0) tc::tmem_alloc<kW>(&tslot);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = tslot;
  constexpr uint32_t idesc = tc::idesc_bf16_f32(128, kW);
  uint32_t phase = 0;
  bool any = false;
  for (int64_t kb = k0; kb < k1; kb += 64) {
    // stage 128 x 64 blocks of both operands (K-major, 128-byte swizzle)
    for (int e = t; e < kW * 8; e += blockDim.x) {
      const int row = e >> 3, c = e & 7;
      uint4 za = make_uint4(0, 0, 0, 0), zb = make_uint4(0, 0, 0, 0);
      if (kb + c * 8 < k1) {
        za = *reinterpret_cast<const uint4*>(Z + (int64_t)row * rows_total + kb + c * 8);
        zb = *reinterpret_cast<const uint4*>(A + (int64_t)row * rows_total + kb + c * 8);
      }
      *reinterpret_cast<uint4*>(sA + tc::sw128_offset(row, c * 8, kW)) = za;
      *reinterpret_cast<uint4*>(sB + tc::sw128_offset(row, c * 8, kW)) = zb;
    }
    tc::fence_async_smem();
    tc::tc_fence_before();
    __syncthreads();
    if (t == 0) {
      tc::tc_fence_after();
      const uint32_t a_base = tc::smem_addr(sA), b_base = tc::smem_addr(sB);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk)
        tc::mma_bf16(tmem, tc::smem_desc_sw128(a_base + kk * 32), tc::smem_desc_sw128(b_base + kk * 32), idesc,
                     (any || kk > 0) ? 1u : 0u);
      tc::mma_commit(&bar);
    }
    any = true;
    if (!tc::mbar_wait(&bar, phase)) {
      raise_status(status, STATUS_TIMEOUT);
      atomicExch(&abort_flag, 1);
    }
    phase ^= 1u;
    tc::tc_fence_after();
    __syncthreads();
    if (abort_flag) break;
  }
  if (any && !abort_flag) {
    float* g = gparams + w_off[l + 1];
    for (int ch = 0; ch < kW / 32; ++ch) {
      float v[32];
      tc::tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + ch * 32, v);
      float4* g4 = reinterpret_cast<float4*>(g + t * kW + ch * 32);
#pragma unroll
      for (int i = 0; i < 8; ++i) atomicAdd(g4 + i, make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]));
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  if (warp == 0) tc::tmem_free<kW>(tmem);
}

// The same over the tile images of train_bwd_pipe and decoder_bf16: 64 rows of an image are two 8 KB
// halves of 64 features, rows of 128 bytes in the 128-byte swizzle, which is the transposed (feature
// contiguous) operand form of the MMA, K steps of 16 rows 2 KB apart.  Blocks of 64 rows of both
// operands (32 KB) stream through kDwStages shared-memory stages by bulk copies: thread 0 copies,
// thread 32 issues the MMAs.  Grid (n_tc, splits), two CTAs per SM.
constexpr int kDwStages = 3;
constexpr int kDwStageBytes = 4 * 8192;
size_t dw_image_smem_bytes() { return 1024 + (size_t)kDwStages * kDwStageBytes; }
__global__ void __launch_bounds__(128, 2) train_dw_gemm_image(const __nv_bfloat16* zbstore, const __nv_bfloat16* astore,
                                                              int64_t rows_total, int64_t k_per_split, float* gparams,
                                                              const int64_t* w_off, uint32_t* status) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* stages = smem_raw + ((1024u - (tc::smem_addr(smem_raw) & 1023u)) & 1023u);
  __shared__ uint64_t full[kDwStages], empty[kDwStages], done;
  __shared__ uint32_t tslot;
  __shared__ int abort_flag;
  const int t = threadIdx.x, warp = t >> 5;
  const int l = blockIdx.x;
  const uint8_t* Z = (const uint8_t*)(zbstore + (int64_t)l * kW * rows_total);
  const uint8_t* A = (const uint8_t*)(astore + (int64_t)l * kW * rows_total);
  const int64_t k0 = (int64_t)blockIdx.y * k_per_split;
  const int64_t k1 = min(rows_total, k0 + k_per_split);
  const int n_blk = (int)((k1 - k0) / 64);                 // rows_total and k_per_split are multiples of 64
  if (t == 0) {
    for (int i = 0; i < kDwStages; ++i) {
      tc::mbar_init(&full[i], 1);
      tc::mbar_init(&empty[i], 1);
    }
    tc::mbar_init(&done, 1);
    abort_flag = 0;
    tc::fence_mbar_init();
  }
  if (warp == 0) tc::tmem_alloc<kW>(&tslot);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = tslot;
  uint32_t fetched = 0;   // stages this thread started to fill
  if (t == 0) {
    fetched = ring_fill<kDwStages>(
        (uint32_t)n_blk,
        [&](uint32_t st, uint32_t phase) { return pipe_wait(status, &abort_flag, &empty[st], phase); },
        [&](uint32_t st, uint32_t b) {
          const int64_t row = k0 + 64 * (int64_t)b;
          const int64_t at = (row >> 7) * kLayerBytes + (row & 64) * 128;   // half of 64 features: 16 KB apart
          uint8_t* dst = stages + st * kDwStageBytes;
          tc::mbar_expect_tx(&full[st], (uint32_t)kDwStageBytes);
          tc::bulk_g2s(dst, Z + at, 8192, &full[st]);
          tc::bulk_g2s(dst + 8192, Z + at + kLayerBytes / 2, 8192, &full[st]);
          tc::bulk_g2s(dst + 16384, A + at, 8192, &full[st]);
          tc::bulk_g2s(dst + 24576, A + at + kLayerBytes / 2, 8192, &full[st]);
        });
  }
  if (t == 32) {
    constexpr uint32_t idesc = tc::idesc_bf16_f32(128, kW) | (1u << 15) | (1u << 16);   // both operands transposed
    for (int b = 0; b < n_blk; ++b) {
      const int st = b % kDwStages;
      pipe_wait(status, &abort_flag, &full[st], (uint32_t)((b / kDwStages) & 1));
      const uint32_t a_base = tc::smem_addr(stages + st * kDwStageBytes), b_base = a_base + 16384;
#pragma unroll
      for (int kk = 0; kk < 4; ++kk)
        tc::mma_bf16(tmem, tc::smem_desc_sw128_mn(a_base + kk * 2048, 8192),
                     tc::smem_desc_sw128_mn(b_base + kk * 2048, 8192), idesc, (b > 0 || kk > 0) ? 1u : 0u);
      tc::mma_commit(&empty[st]);
    }
    tc::mma_commit(&done);
  }
  __syncwarp();
  bool ok = tc::mbar_wait(&done, 0);
  if (!ok) raise_status(status, STATUS_TIMEOUT);
  ok = __all_sync(0xffffffffu, ok && !*(volatile int*)&abort_flag);
  tc::tc_fence_after();
  if (n_blk > 0 && ok) {
    float* g = gparams + w_off[l + 1];
    for (int ch = 0; ch < kW / 32; ++ch) {
      float v[32];
      tc::tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + ch * 32, v);
      float4* g4 = reinterpret_cast<float4*>(g + t * kW + ch * 32);
#pragma unroll
      for (int i = 0; i < 8; ++i) atomicAdd(g4 + i, make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]));
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  if (fetched > 0 && *(volatile int*)&abort_flag)   // after a timeout the last copies land before the CTA exits
    ring_land<kDwStages>(fetched, [&](uint32_t st, uint32_t phase) { (void)tc::mbar_wait(&full[st], phase); });
  tc::tc_fence_after();
  if (warp == 0) tc::tmem_free<kW>(tmem);
}

// First-layer weight gradient dW0[f][j] = sum_rows zbar0[f][row] in[row][j] and the latent
// adjoints of the primal rows (d loss / d xhat) and of the JVP rows (d loss / d u),
// sum_f zbar0[f][row] W0[f][d + j], from one pass over zbar0.  in[row] is the layer-0 input of
// the row: [Xn, xhat] (primal), e_k / X_range_k (X tangent k), [0, u] (JVP).
// One 128-row training tile at a time (rows k Pt + q: kind k of point q): its 128 x 128 block of
// zbar0 is staged in shared memory by float4 loads (512 contiguous bytes per feature), the
// points' inputs beside it.  Thread (f, half) sums the weight gradient of feature f over half
// of the tile's points in registers for every tile the CTA takes, and adds it to dW0 once;
// the latent adjoints take (row, 4 latents) per thread.
constexpr int kMaxIn = 40;
constexpr int kDw0Stride = 132;       // floats per staged feature row (128 rows + pad; float4 aligned)
constexpr int kDw0MaxPt = 64;         // points per tile (R >= 2)
template <int D>
__global__ void __launch_bounds__(256) train_dw0_lat(const float* zb0, int64_t rows_total, Batch b, int r, int Pt,
                                                     const float* norm, const float* W0, float* gW0, float* g_lat_pt,
                                                     float* g_u_pt) {
  constexpr int d = D;
  extern __shared__ __align__(16) float dsm[];
  float* sz = dsm;                                   // [128 f][kDw0Stride]: zbar0 of the tile's rows
  float* sin0 = sz + kW * kDw0Stride;                // [kDw0MaxPt][kMaxIn]: primal inputs of the points
  float* su = sin0 + kDw0MaxPt * kMaxIn;             // [kDw0MaxPt][32]: JVP directions
  float* sWl = su + kDw0MaxPt * 32;                  // [128][36]: latent columns of W0 (float4 rows)
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int K = d + r;
  for (int e = t; e < kW * 36; e += blockDim.x) {
    const int ff = e / 36, j = e % 36;
    sWl[e] = j < r ? W0[ff * K + d + j] : 0.f;
  }
  const int f = t & (kW - 1), half = t >> 7;
  const int q_lo = half ? (Pt + 1) / 2 : 0, q_hi = half ? Pt : (Pt + 1) / 2;
  float inv_range[D];
#pragma unroll
  for (int a2 = 0; a2 < D; ++a2) inv_range[a2] = 1.f / norm[D + a2];
  float acc[kMaxIn];
#pragma unroll
  for (int j = 0; j < kMaxIn; ++j) acc[j] = 0.f;
  const int64_t n_tiles = rows_total / 128;
  for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const int64_t row0 = tile * 128;
    __syncthreads();   // the previous tile's staged values are consumed
    // zbar0 rows of the tile: warp w stages features w, w + 8, ..., one float4 per lane
    for (int ff = warp; ff < kW; ff += 8) {
      const float4 v = *reinterpret_cast<const float4*>(zb0 + (int64_t)ff * rows_total + row0 + 4 * lane);
      *reinterpret_cast<float4*>(sz + ff * kDw0Stride + 4 * lane) = v;
    }
    // the points' primal inputs [Xn, xhat] and JVP directions
    for (int e = t; e < Pt * kMaxIn; e += blockDim.x) {
      const int q = e / kMaxIn, j = e % kMaxIn;
      const int64_t pnt = tile * Pt + q;
      float in = 0.f;
      if (pnt < b.B && j < K) in = j < d ? (b.X[pnt * d + j] - norm[j]) / norm[d + j] : b.xh[pnt * r + (j - d)];
      sin0[q * kMaxIn + j] = in;
    }
    for (int e = t; e < Pt * 32; e += blockDim.x) {
      const int q = e >> 5, j = e & 31;
      const int64_t pnt = tile * Pt + q;
      su[e] = (pnt < b.B && j < r) ? b.u[pnt * r + j] : 0.f;
    }
    __syncthreads();
    // (a) weight gradient of feature f over this thread's points (rows of invalid points are zero)
    const float* zf = sz + f * kDw0Stride;
    // four points at a time with float4 reads of the staged adjoints where the rows allow it (a
    // quarter warp's 16-byte reads then fall in distinct banks; the scalar reads of lanes 132
    // floats apart conflict 4 ways)
    const bool vec4 = (Pt & 3) == 0 && (q_lo & 3) == 0 && (q_hi & 3) == 0;
    for (int q4 = q_lo; vec4 && q4 < q_hi; q4 += 4) {
      const float4 zp4 = *reinterpret_cast<const float4*>(zf + q4);
      float4 zt4[D];
#pragma unroll
      for (int a2 = 0; a2 < D; ++a2) zt4[a2] = *reinterpret_cast<const float4*>(zf + (1 + a2) * Pt + q4);
      const float4 zj4 = *reinterpret_cast<const float4*>(zf + (D + 1) * Pt + q4);
#pragma unroll
      for (int u4 = 0; u4 < 4; ++u4) {
        const int q = q4 + u4;
        const float zp = u4 == 0 ? zp4.x : u4 == 1 ? zp4.y : u4 == 2 ? zp4.z : zp4.w;
        const float zj = u4 == 0 ? zj4.x : u4 == 1 ? zj4.y : u4 == 2 ? zj4.z : zj4.w;
        const float* in = sin0 + q * kMaxIn;
#pragma unroll
        for (int j = 0; j < kMaxIn; j += 4) {
          if (j < K) {
            const float4 v = *reinterpret_cast<const float4*>(in + j);
            acc[j] = fmaf(zp, v.x, acc[j]);
            acc[j + 1] = fmaf(zp, v.y, acc[j + 1]);
            acc[j + 2] = fmaf(zp, v.z, acc[j + 2]);
            acc[j + 3] = fmaf(zp, v.w, acc[j + 3]);
          }
        }
#pragma unroll
        for (int a2 = 0; a2 < D; ++a2) {
          const float zt = u4 == 0 ? zt4[a2].x : u4 == 1 ? zt4[a2].y : u4 == 2 ? zt4[a2].z : zt4[a2].w;
          acc[a2] = fmaf(zt, inv_range[a2], acc[a2]);
        }
        const float* uq = su + q * 32;
#pragma unroll
        for (int j = 0; j < 32; j += 4) {
          if (j < r) {
            const float4 v = *reinterpret_cast<const float4*>(uq + j);
            acc[D + j] = fmaf(zj, v.x, acc[D + j]);
            acc[D + j + 1] = fmaf(zj, v.y, acc[D + j + 1]);
            acc[D + j + 2] = fmaf(zj, v.z, acc[D + j + 2]);
            acc[D + j + 3] = fmaf(zj, v.w, acc[D + j + 3]);
          }
        }
      }
    }
    for (int q = q_lo; !vec4 && q < q_hi; ++q) {
      const float zp = zf[q];                   // primal row
      const float* in = sin0 + q * kMaxIn;
#pragma unroll
      for (int j = 0; j < kMaxIn; j += 4) {
        if (j < K) {
          const float4 v = *reinterpret_cast<const float4*>(in + j);
          acc[j] = fmaf(zp, v.x, acc[j]);
          acc[j + 1] = fmaf(zp, v.y, acc[j + 1]);
          acc[j + 2] = fmaf(zp, v.z, acc[j + 2]);
          acc[j + 3] = fmaf(zp, v.w, acc[j + 3]);
        }
      }
#pragma unroll
      for (int a2 = 0; a2 < D; ++a2)                 // X-tangent rows: one input each
        acc[a2] = fmaf(zf[(1 + a2) * Pt + q], inv_range[a2], acc[a2]);
      const float zj = zf[(D + 1) * Pt + q];               // JVP row: [0, u] (u zero-padded to 32)
      const float* uq = su + q * 32;
#pragma unroll
      for (int j = 0; j < 32; j += 4) {
        if (j < r) {
          const float4 v = *reinterpret_cast<const float4*>(uq + j);
          acc[D + j] = fmaf(zj, v.x, acc[D + j]);
          acc[D + j + 1] = fmaf(zj, v.y, acc[D + j + 1]);
          acc[D + j + 2] = fmaf(zj, v.z, acc[D + j + 2]);
          acc[D + j + 3] = fmaf(zj, v.w, acc[D + j + 3]);
        }
      }
    }
    // (b) latent adjoints of the primal (k = 0) and JVP (k = d + 1) rows: (row, 4 latents) per thread
    const int n_groups = (r + 3) / 4;
    for (int o = t; o < 2 * Pt * n_groups; o += blockDim.x) {
      const int g = o % n_groups, rr = o / n_groups;
      const int q = rr % Pt, jvp = rr / Pt;
      const int64_t pnt = tile * Pt + q;
      const int row = (jvp ? d + 1 : 0) * Pt + q;
      float v0 = 0.f, v1 = 0.f, v2 = 0.f, v3 = 0.f;
#pragma unroll 8
      for (int ff = 0; ff < kW; ++ff) {
        const float z = sz[ff * kDw0Stride + row];
        const float4 w = *reinterpret_cast<const float4*>(sWl + ff * 36 + 4 * g);
        v0 = fmaf(z, w.x, v0);
        v1 = fmaf(z, w.y, v1);
        v2 = fmaf(z, w.z, v2);
        v3 = fmaf(z, w.w, v3);
      }
      if (pnt < b.B) {
        float* dst = (jvp ? g_u_pt : g_lat_pt) + pnt * r + 4 * g;
        const int nj = min(4, r - 4 * g);
        if (nj > 0) dst[0] = v0;
        if (nj > 1) dst[1] = v1;
        if (nj > 2) dst[2] = v2;
        if (nj > 3) dst[3] = v3;
      }
    }
  }
  // combine the two halves of each feature, then one atomic per weight
  __syncthreads();
  float* red = sz;   // reused as [128][kMaxIn + 1]
  if (half == 1) {
#pragma unroll
    for (int j = 0; j < kMaxIn; ++j) red[f * (kMaxIn + 1) + j] = acc[j];
  }
  __syncthreads();
  if (half == 0) {
#pragma unroll
    for (int j = 0; j < kMaxIn; ++j)
      if (j < K) atomicAdd(&gW0[f * K + j], acc[j] + red[f * (kMaxIn + 1) + j]);
  }
}

size_t dw0_smem_bytes() {
  return (size_t)(kW * kDw0Stride + kDw0MaxPt * kMaxIn + kDw0MaxPt * 32 + kW * 36) * sizeof(float);
}

// The same gradients from zbar0 as train_bwd_pipe stores it: row-major in decoder_bf16's row order (R = D + 2
// consecutive rows per point, floor(32 / R) points per 32 rows), so that a tile is 64 consecutive KB.  One
// CTA per SM; tile i + 1 arrives by asynchronous copies (its inputs in registers) under the arithmetic of tile
// i.  Thread (feature pair, point group) sums the weight gradients: one shared read of an input then serves
// two features, and the eight groups' sums meet once per CTA.  The latent adjoints take (point, 4 latents,
// quarter of the features) per thread, both rows of the point at once, and four shuffled sums.  Bound by the
// latency of the shared-memory reads (16 warps); 65,536 points, r = 16, 2D: 132 us with one staged tile per CTA and one
// row or feature per thread, 94 us like this.
constexpr int kDw0Threads = 512;
constexpr int kDw0In = 32;            // d + r <= 31 on this path

template <int D>
__global__ void __launch_bounds__(kDw0Threads, 1) train_dw0_pipe(const float* __restrict__ zb0, int64_t rows_total,
                                                                 Batch b, int r, const float* norm, const float* W0,
                                                                 float* gW0, float* g_lat_pt, float* g_u_pt) {
  constexpr int R = D + 2, PPG = 32 / R, PT = 4 * PPG;             // points per lane group and per tile
  constexpr int NI = (PT * kDw0In + kDw0Threads - 1) / kDw0Threads;  // staged inputs per thread
  constexpr int NG = kDw0Threads / (kW / 2);                       // point groups
  extern __shared__ __align__(16) float dsm[];
  float* sz = dsm;                                   // two tiles [128 rows][kDw0Stride]
  float* sin0 = sz + 2 * 128 * kDw0Stride;           // [PT][32]: primal inputs of the points
  float* su = sin0 + PT * kDw0In;                    // [PT][32]: JVP directions
  float* sWl = su + PT * kDw0In;                     // [128][36]: latent columns of W0
  const int t = threadIdx.x, lane = t & 31;
  const int K = D + r;
  for (int e = t; e < kW * 36; e += kDw0Threads) {
    const int ff = e / 36, j = e % 36;
    sWl[e] = j < r ? W0[ff * K + D + j] : 0.f;
  }
  float inv_range[D];
#pragma unroll
  for (int a = 0; a < D; ++a) inv_range[a] = 1.f / norm[D + a];
  const float lo = lane < D ? norm[lane] : 0.f, range = lane < D ? norm[D + lane] : 1.f;
  const int64_t n_tiles = rows_total / 128;
  auto fetch = [&](int64_t tile, int buf) {
    const float* src = zb0 + tile * 128 * kW;
    float* dst = sz + buf * 128 * kDw0Stride;
#pragma unroll
    for (int i = 0; i < 128 * kW / 4 / kDw0Threads; ++i) {
      const int e = t + i * kDw0Threads, row = e >> 5, c = 4 * (e & 31);
      cp_async16(dst + row * kDw0Stride + c, src + row * kW + c);
    }
    cp_async_commit();
  };
  float vi[NI], vu[NI];
  // input `lane` of points t / 32, ... of a tile: X or xhat, and u
  auto load_inputs = [&](int64_t tile) {
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      const int q = (t + i * kDw0Threads) >> 5;
      const int64_t pnt = tile * PT + q;
      const bool in = q < PT && pnt < b.B;
      vi[i] = in && lane < K ? (lane < D ? b.X[pnt * D + lane] : b.xh[pnt * r + (lane - D)]) : 0.f;
      vu[i] = in && lane < r ? b.u[pnt * r + lane] : 0.f;
    }
  };
  const int fp = t & (kW / 2 - 1), pg = t / (kW / 2);
  float acc[2][kDw0In];
#pragma unroll
  for (int j = 0; j < kDw0In; ++j) acc[0][j] = acc[1][j] = 0.f;
  int64_t tile = blockIdx.x;
  if (tile < n_tiles) {
    fetch(tile, 0);
    load_inputs(tile);
  }
  for (int buf = 0; tile < n_tiles; buf ^= 1) {
    const int64_t next = tile + gridDim.x;
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      const int e = t + i * kDw0Threads;
      const bool valid = tile * PT + (e >> 5) < b.B;
      if (e < PT * kDw0In) {
        sin0[e] = lane < D ? (valid ? (vi[i] - lo) / range : 0.f) : vi[i];
        su[e] = vu[i];
      }
    }
    if (next < n_tiles) {
      fetch(next, buf ^ 1);
      cp_async_wait_but_one();
    } else {
      cp_async_wait_all();
    }
    __syncthreads();
    if (next < n_tiles) load_inputs(next);
    const float* z = sz + buf * 128 * kDw0Stride;
    // (a) weight gradients of features 2 fp, 2 fp + 1 over this thread's points (rows of points past the batch are 0)
#pragma unroll
    for (int i = 0; i < (PT + NG - 1) / NG; ++i) {
      const int q = pg + i * NG;
      if (PT % NG != 0 && q >= PT) break;
      const float* zq = z + ((q / PPG) * 32 + (q % PPG) * R) * kDw0Stride + 2 * fp;
      const float2 zp = *reinterpret_cast<const float2*>(zq);
      const float2 zj = *reinterpret_cast<const float2*>(zq + (D + 1) * kDw0Stride);
      const float* in = sin0 + q * kDw0In;
#pragma unroll
      for (int j = 0; j < kDw0In; j += 4) {
        if (j < K) {
          const float4 v = *reinterpret_cast<const float4*>(in + j);
          fma2(acc[0][j], acc[0][j + 1], v.x, v.y, zp.x);
          fma2(acc[0][j + 2], acc[0][j + 3], v.z, v.w, zp.x);
          fma2(acc[1][j], acc[1][j + 1], v.x, v.y, zp.y);
          fma2(acc[1][j + 2], acc[1][j + 3], v.z, v.w, zp.y);
        }
      }
#pragma unroll
      for (int a = 0; a < D; ++a) {                  // X-tangent rows: one input each
        const float2 zt = *reinterpret_cast<const float2*>(zq + (1 + a) * kDw0Stride);
        acc[0][a] = fmaf(zt.x, inv_range[a], acc[0][a]);
        acc[1][a] = fmaf(zt.y, inv_range[a], acc[1][a]);
      }
      const float* uq = su + q * kDw0In;             // JVP row: [0, u]
#pragma unroll
      for (int j = 0; j + D < kDw0In; j += 4) {
        if (j < r) {
          const float4 v = *reinterpret_cast<const float4*>(uq + j);
          const float vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int c = 0; c < 4; ++c)
            if (j + c + D < kDw0In) {
              acc[0][D + j + c] = fmaf(zj.x, vv[c], acc[0][D + j + c]);
              acc[1][D + j + c] = fmaf(zj.y, vv[c], acc[1][D + j + c]);
            }
        }
      }
    }
    // (b) latent adjoints of the primal and the JVP row of each point: lanes (point, 4 latents, features 16 i + 4 part ..)
    const int G = (r + 3) / 4, tasks = PT * G * 4;
    for (int o0 = t - lane; o0 < tasks; o0 += kDw0Threads) {
      const int o = min(o0 + lane, tasks - 1);
      const int part = o & 3, g = (o >> 2) % G, q = (o >> 2) / G;
      const float* zp = z + ((q / PPG) * 32 + (q % PPG) * R) * kDw0Stride + 4 * part;
      const float* zj = zp + (D + 1) * kDw0Stride;
      const float* w = sWl + 4 * part * 36 + 4 * g;
      float vp[4] = {0.f, 0.f, 0.f, 0.f}, vj[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int i = 0; i < kW / 16; ++i) {
        const float4 p4 = *reinterpret_cast<const float4*>(zp + 16 * i);
        const float4 j4 = *reinterpret_cast<const float4*>(zj + 16 * i);
        const float pa[4] = {p4.x, p4.y, p4.z, p4.w}, ja[4] = {j4.x, j4.y, j4.z, j4.w};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float4 w4 = *reinterpret_cast<const float4*>(w + (16 * i + c) * 36);
          fma2(vp[0], vp[1], w4.x, w4.y, pa[c]);
          fma2(vp[2], vp[3], w4.z, w4.w, pa[c]);
          fma2(vj[0], vj[1], w4.x, w4.y, ja[c]);
          fma2(vj[2], vj[3], w4.z, w4.w, ja[c]);
        }
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        vp[c] += __shfl_xor_sync(0xffffffffu, vp[c], 1);
        vj[c] += __shfl_xor_sync(0xffffffffu, vj[c], 1);
        vp[c] += __shfl_xor_sync(0xffffffffu, vp[c], 2);
        vj[c] += __shfl_xor_sync(0xffffffffu, vj[c], 2);
      }
      const int64_t pnt = tile * PT + q;
      if (part < 2 && o0 + lane < tasks && pnt < b.B) {
        float* dst = (part ? g_u_pt : g_lat_pt) + pnt * r + 4 * g;
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (4 * g + c < r) dst[c] = part ? vj[c] : vp[c];
      }
    }
    __syncthreads();
    tile = next;
  }
  // the point groups' sums, then one atomic per weight
  constexpr int LD = kDw0In + 1;
  static_assert(NG * LD <= 2 * kDw0Stride, "the sums fit the tile buffers");
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int j = 0; j < kDw0In; ++j) sz[(pg * kW + 2 * fp + h) * LD + j] = acc[h][j];
  __syncthreads();
  for (int e = t; e < kW * K; e += kDw0Threads) {
    const int f = e / K, j = e - f * K;
    float sum = 0.f;
#pragma unroll
    for (int g = 0; g < NG; ++g) sum += sz[(g * kW + f) * LD + j];
    atomicAdd(&gW0[e], sum);
  }
}

template <int D>
constexpr size_t dw0_pipe_smem_bytes() {
  return (size_t)(2 * 128 * kDw0Stride + 2 * 4 * (32 / (D + 2)) * kDw0In + kW * 36) * sizeof(float);
}

// V latents of a point per thread (4 as one vector reduction where r allows it), so that consecutive threads
// read consecutive words: 65,536 points, r = 16, 2,048 snapshots 30 us with a point per thread,
// 6 us like this.
template <int V>
__global__ void train_lat_scatter(Batch b, int r, const float* __restrict__ g_lat_pt, const float* __restrict__ g_u_pt,
                                  float dt_snap, float* g_lat) {
  const int per = r / V;
  const int64_t n = b.B * per;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t p = e / per;
    const int j = (int)(e - p * per) * V;
    const int s = b.snap[p], nx = b.next[p];
    if (V == 4) {
      float4 gu = *reinterpret_cast<const float4*>(g_u_pt + p * r + j);
      float4 gl = *reinterpret_cast<const float4*>(g_lat_pt + p * r + j);
      gu = make_float4(gu.x / dt_snap, gu.y / dt_snap, gu.z / dt_snap, gu.w / dt_snap);
      if (nx >= 0) {
        gl = make_float4(gl.x - gu.x, gl.y - gu.y, gl.z - gu.z, gl.w - gu.w);
        atomicAdd(reinterpret_cast<float4*>(g_lat + (int64_t)nx * r + j), gu);
      }
      atomicAdd(reinterpret_cast<float4*>(g_lat + (int64_t)s * r + j), gl);
    } else {
      const float gu = g_u_pt[p * r + j] / dt_snap;
      atomicAdd(&g_lat[(int64_t)s * r + j], g_lat_pt[p * r + j] - (nx >= 0 ? gu : 0.f));
      if (nx >= 0) atomicAdd(&g_lat[(int64_t)nx * r + j], gu);
    }
  }
}

// Adam (Kingma and Ba 2015) on two parameter ranges; zeroes the gradients.
__global__ void train_adam(float* p0, float* g0, float* m0, float* v0, int64_t n0, float* p1, float* g1, float* m1,
                           float* v1, int64_t n1, const int64_t* step, int64_t total_steps, float lr0, float lr1,
                           float beta1, float beta2, float eps, int update) {
  const int64_t t = *step;
  const float frac = total_steps > 1 ? (float)min(t, total_steps - 1) / (float)(total_steps - 1) : 0.f;
  const float lr = lr0 * powf(lr1 / lr0, frac);
  const float bc1 = 1.f - powf(beta1, (float)(t + 1)), bc2 = 1.f - powf(beta2, (float)(t + 1));
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n0 + n1; i += (int64_t)gridDim.x * blockDim.x) {
    float *p, *g, *m, *v;
    int64_t j = i;
    if (i < n0) {
      p = p0; g = g0; m = m0; v = v0;
    } else {
      j = i - n0;
      p = p1; g = g1; m = m1; v = v1;
    }
    const float gr = g[j];
    g[j] = 0.f;
    if (!update) continue;
    const float mm = beta1 * m[j] + (1.f - beta1) * gr;
    const float vv = beta2 * v[j] + (1.f - beta2) * gr * gr;
    m[j] = mm;
    v[j] = vv;
    p[j] -= lr * (mm / bc1) / (sqrtf(vv / bc2) + eps);
  }
}

__global__ void train_step_inc(int64_t* step) { *step += 1; }

// Transposed BF16 images of the square layers: image row = input feature, K = output feature.
__global__ void train_pack_transposed(const float* params, const int64_t* w_off, int n_tc, uint8_t* img) {
  const int64_t total = (int64_t)n_tc * kW * kW;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int l = (int)(i / (kW * kW));
    const int rem = (int)(i % (kW * kW));
    const int out = rem / kW, in = rem % kW;
    const float w = params[w_off[l + 1] + rem];  // W[out][in]
    *reinterpret_cast<__nv_bfloat16*>(img + (size_t)l * kLayerBytes + tc::sw128_offset(in, out, kW)) =
        __float2bfloat16_rn(w);
  }
}

}  // namespace mpmrom

using namespace mpmrom;

struct trainer_ctx {
  mpm_decoder* dec = nullptr;
  train_config cfg{};
  int d = 0, r = 0, R = 0, Pt = 0, n_sm = 0;
  int64_t B = 0, n_tiles = 0, rows_total = 0, n_snap = 0;
  int64_t i_offset = 0;   // first draw of this shard in the step's minibatch
  float n_norm = 0.f;     // points of the whole minibatch (batch x shards)
  Store st{};
  Batch b{};
  // device buffers
  int64_t* snap_base = nullptr;
  int32_t* snap_inst = nullptr;
  int32_t* snap_next = nullptr;
  int64_t* inst_off = nullptr;
  float* X = nullptr;
  float* sx = nullptr;
  float* sv = nullptr;
  float* sF = nullptr;
  float* latents = nullptr;
  float* g_lat = nullptr;
  float* m_lat = nullptr;
  float* v_lat = nullptr;
  float* gparams = nullptr;
  float* m_par = nullptr;
  float* v_par = nullptr;
  float* batch_mem = nullptr;
  int32_t* batch_idx = nullptr;
  float* fwd = nullptr;
  __nv_bfloat16* dstore = nullptr;   // primal rows' activation slopes (n_hidden, W, rows)
  __nv_bfloat16* astore = nullptr;
  __nv_bfloat16* zbstore = nullptr;
  float* zb0 = nullptr;
  float* g_lat_pt = nullptr;
  float* g_u_pt = nullptr;
  uint8_t* wtimg = nullptr;
  int64_t* d_w_off = nullptr;
  int64_t* step = nullptr;
  double* loss = nullptr;
  uint32_t* status = nullptr;
  size_t bwd_smem = 0;
  bool pipe = false;            // decoder_bf16's tile images, train_bwd_pipe, train_dw_gemm_image
  int64_t points_total = 0;     // points of all tiles, padding included (tile images)
  // encoder (Section 4.1) in place of the latent table
  bool enc = false;
  EncDesc E{};
  float* U = nullptr;           // (n_snap, L0) standardised subset positions
  float* enc_p = nullptr;       // parameters, gradients, Adam moments
  float* enc_g = nullptr;
  float* enc_m = nullptr;
  float* enc_v = nullptr;
  float* enc_ss = nullptr;      // shift (d), scale (d)
  double* enc_work = nullptr;
  cudaStream_t cap_stream = nullptr;
  cudaGraphExec_t graph = nullptr;
  cudaGraphExec_t graph_noupdate = nullptr;
};


// ---------------------------------------------------------------------------------------------
// Input and output scaling of Appendix B: per coordinate, min-max of the reference positions X
// and mean / standard deviation of every snapshot position x.  Pass 1: per-block minimum and
// maximum of X and FP64 sum of x; pass 2: FP64 sum of (x - mean)^2 with the pass-1 mean.  One
// block reduces the partials after each pass.
// ---------------------------------------------------------------------------------------------
constexpr int kScaleThreads = 256;

__device__ __forceinline__ double block_sum_d(double v, double* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
  return t;   // valid in thread 0
}

__device__ __forceinline__ float block_minmax(float v, bool is_max, float* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float u = __shfl_down_sync(0xffffffffu, v, o);
    v = is_max ? fmaxf(v, u) : fminf(v, u);
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  float t = v;
  if (threadIdx.x == 0)
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) t = is_max ? fmaxf(t, sh[w]) : fminf(t, sh[w]);
  return t;   // valid in thread 0
}

// pass 0: part[b] = {min X_a, max X_a, sum x_a}, pass 1: part[b] = {sum (x_a - mean_a)^2}
__global__ void __launch_bounds__(kScaleThreads) scale_partials(int pass, int d, const float* __restrict__ X,
                                                                int64_t nX, const float* __restrict__ x, int64_t nx,
                                                                const double* __restrict__ mean, double* part) {
  __shared__ double shd[kScaleThreads / 32];
  __shared__ float shf[kScaleThreads / 32];
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (int a = 0; a < d; ++a) {
    if (pass == 0) {
      float lo = INFINITY, hi = -INFINITY;
      for (int64_t i = i0; i < nX; i += stride) {
        const float u = X[i * d + a];
        lo = fminf(lo, u);
        hi = fmaxf(hi, u);
      }
      double s = 0.0;
      for (int64_t i = i0; i < nx; i += stride) s += (double)x[i * d + a];
      lo = block_minmax(lo, false, shf);
      hi = block_minmax(hi, true, shf);
      s = block_sum_d(s, shd);
      if (threadIdx.x == 0) {
        part[(size_t)blockIdx.x * 3 * d + 3 * a + 0] = lo;
        part[(size_t)blockIdx.x * 3 * d + 3 * a + 1] = hi;
        part[(size_t)blockIdx.x * 3 * d + 3 * a + 2] = s;
      }
    } else {
      const double m = mean[a];
      double s = 0.0;
      for (int64_t i = i0; i < nx; i += stride) {
        const double e = (double)x[i * d + a] - m;
        s = fma(e, e, s);
      }
      s = block_sum_d(s, shd);
      if (threadIdx.x == 0) part[(size_t)blockIdx.x * d + a] = s;
    }
  }
}

// one thread per coordinate: reduce the partials; pass 0 leaves the mean in stats[0..d), pass 1
// writes the decoder's scaling {X_min, X_range, mean, std} (as floats) into norm
__global__ void scale_finish(int pass, int d, int n_part, int64_t nx, const double* part, double* stats,
                             float* norm) {
  const int a = threadIdx.x;
  if (a >= d) return;
  if (pass == 0) {
    double lo = INFINITY, hi = -INFINITY, s = 0.0;
    for (int b = 0; b < n_part; ++b) {
      lo = fmin(lo, part[(size_t)b * 3 * d + 3 * a + 0]);
      hi = fmax(hi, part[(size_t)b * 3 * d + 3 * a + 1]);
      s += part[(size_t)b * 3 * d + 3 * a + 2];
    }
    stats[a] = s / (double)nx;
    stats[d + a] = lo;
    stats[2 * d + a] = hi;
  } else {
    double ss = 0.0;
    for (int b = 0; b < n_part; ++b) ss += part[(size_t)b * d + a];
    norm[a] = (float)stats[d + a];
    norm[d + a] = (float)(stats[2 * d + a] - stats[d + a]);
    norm[2 * d + a] = (float)stats[a];
    norm[3 * d + a] = (float)sqrt(ss / (double)nx);
  }
}

namespace {

mpm_status train_launch_update(trainer_ctx* c, cudaStream_t s);

mpm_status train_launch_step(trainer_ctx* c, cudaStream_t s, int update) {
  mpm_decoder* dec = c->dec;
  const int d = c->d, r = c->r;
  if (c->enc) {
    // latents of every snapshot from the encoder
    mpm_status se = enc_forward(c->E, c->enc_p, c->U, c->n_snap, c->latents, c->n_sm, s);
    if (se != MPM_OK) return se;
  }
  const int sample_blocks = (int)std::max<int64_t>(1, std::min<int64_t>((c->B + 127) / 128, (int64_t)c->n_sm * 16));
  (d == 2 ? train_sample<2> : train_sample<3>)<<<sample_blocks, 128, 0, s>>>(
      c->st, c->b, c->latents, c->cfg.dt_snap, c->cfg.seed, c->step, c->loss, c->i_offset);
  MPM_CUDA_TRY(cudaGetLastError());
  int kinds[8];
  kinds[0] = 0;
  for (int a = 0; a < d; ++a) kinds[1 + a] = 1 + a;
  kinds[1 + d] = 1000;
  mpm_status st = decoder_launch_train(dec, c->b.X, c->b.xh, c->b.u, kinds, c->R, c->B, c->fwd, c->dstore, c->astore,
                                       c->rows_total, c->points_total, s);
  if (st != MPM_OK) return st;
  BwdArgs a{};
  a.d = d;
  a.r = r;
  a.n_hidden = dec->n_hidden;
  a.n_tc = dec->n_tc;
  a.act = dec->act;
  a.R = c->R;
  a.Pt = c->Pt;
  a.n = c->B;
  a.n_norm = c->n_norm;
  a.rows_total = c->rows_total;
  a.points_total = c->points_total;
  const int L = (int)dec->w_off.size();
  a.W0 = dec->params + dec->w_off[0];
  a.Wout = dec->params + dec->w_off[L - 1];
  a.norm = dec->norm;
  a.dstore = c->dstore;
  a.astore = c->astore;
  a.wtimg = c->wtimg;
  a.fwd = c->fwd;
  a.b = c->b;
  a.lamF = c->cfg.lambda_F;
  a.lamv = c->cfg.lambda_v;
  a.zbstore = c->zbstore;
  a.zb0 = c->zb0;
  a.gparams = c->gparams;
  a.gW0_off = dec->w_off[0];
  a.gb0_off = dec->b_off[0];
  a.gWout_off = dec->w_off[L - 1];
  a.gbout_off = dec->b_off[L - 1];
  for (int l = 0; l < dec->n_hidden; ++l) a.gb_off[l] = dec->b_off[l];
  a.g_lat_pt = c->g_lat_pt;
  a.g_u_pt = c->g_u_pt;
  a.loss = c->loss;
  a.status = c->status;
  const int bw = (int)std::max<int64_t>(1, std::min<int64_t>(c->n_tiles, c->n_sm));
  if (c->pipe)
    (d == 2 ? train_bwd_pipe<2> : train_bwd_pipe<3>)<<<bw, kBwdPipeThreads, c->bwd_smem, s>>>(a);
  else
    train_bwd_tc<<<bw, kBwdThreads, c->bwd_smem, s>>>(a);
  MPM_CUDA_TRY(cudaGetLastError());
  if (dec->n_tc > 0) {
    // several CTAs per SM (four with 32 KB of shared memory each, two with the streamed images), so that
    // loads of as many K blocks are in flight per SM; the splits' partial sums meet in vector reductions
    const int splits = std::max(1, (c->pipe ? 2 : 4) * c->n_sm / dec->n_tc);
    int64_t kps = (c->rows_total + splits - 1) / splits;
    kps = (kps + 63) / 64 * 64;
    dim3 g(dec->n_tc, (unsigned)((c->rows_total + kps - 1) / kps));
    if (c->pipe)
      train_dw_gemm_image<<<g, 128, dw_image_smem_bytes(), s>>>(c->zbstore, c->astore, c->rows_total, kps, c->gparams,
                                                                c->d_w_off, c->status);
    else
      train_dw_gemm<<<g, 128, 0, s>>>(c->zbstore, c->astore, c->rows_total, kps, c->gparams, c->d_w_off, c->status);
    MPM_CUDA_TRY(cudaGetLastError());
  }
  const float* W0 = dec->params + dec->w_off[0];
  float* gW0 = c->gparams + dec->w_off[0];
  if (c->pipe) {
    const int g0 = (int)std::min<int64_t>(c->n_sm, c->rows_total / 128);
    if (d == 2)
      train_dw0_pipe<2><<<g0, kDw0Threads, dw0_pipe_smem_bytes<2>(), s>>>(c->zb0, c->rows_total, c->b, r, dec->norm, W0,
                                                                          gW0, c->g_lat_pt, c->g_u_pt);
    else
      train_dw0_pipe<3><<<g0, kDw0Threads, dw0_pipe_smem_bytes<3>(), s>>>(c->zb0, c->rows_total, c->b, r, dec->norm, W0,
                                                                          gW0, c->g_lat_pt, c->g_u_pt);
  } else {
    auto* dw0 = d == 2 ? train_dw0_lat<2> : train_dw0_lat<3>;
    dw0<<<c->n_sm * 2, 256, dw0_smem_bytes(), s>>>(c->zb0, c->rows_total, c->b, r, c->Pt, dec->norm, W0, gW0,
                                                   c->g_lat_pt, c->g_u_pt);
  }
  MPM_CUDA_TRY(cudaGetLastError());
  {
    const bool vec = r % 4 == 0;   // rows of g_lat, g_lat_pt and g_u_pt then start on 16 bytes
    const int64_t work = c->B * (vec ? r / 4 : r);
    const int g = (int)std::max<int64_t>(1, std::min<int64_t>((work + 255) / 256, (int64_t)c->n_sm * 16));
    (vec ? train_lat_scatter<4> : train_lat_scatter<1>)<<<g, 256, 0, s>>>(c->b, r, c->g_lat_pt, c->g_u_pt,
                                                                         c->cfg.dt_snap, c->g_lat);
  }
  MPM_CUDA_TRY(cudaGetLastError());
  if (c->enc) {
    // pull the per-snapshot latent gradients back through the encoder
    st = enc_backward(c->E, c->enc_p, c->U, c->n_snap, c->g_lat, c->enc_g, c->n_sm, s);
    if (st != MPM_OK) return st;
  }
  if (update) return train_launch_update(c, s);
  return MPM_OK;
}

// Adam on the decoder and on the latent table or the encoder (the gradients are consumed and
// zeroed), re-pack of the weight images, step count.
mpm_status train_launch_update(trainer_ctx* c, cudaStream_t s) {
  mpm_decoder* dec = c->dec;
  const int r = c->r;
  mpm_status st = MPM_OK;
  {
    const int64_t n0 = dec->n_params, n1 = c->enc ? (int64_t)c->E.n_params : c->n_snap * r;
    float* p1 = c->enc ? c->enc_p : c->latents;
    float* g1 = c->enc ? c->enc_g : c->g_lat;
    float* m1 = c->enc ? c->enc_m : c->m_lat;
    float* v1 = c->enc ? c->enc_v : c->v_lat;
    if (c->enc) MPM_CUDA_TRY(cudaMemsetAsync(c->g_lat, 0, sizeof(float) * c->n_snap * r, s));
    int ba = (int)std::max<int64_t>(1, std::min<int64_t>((n0 + n1 + 255) / 256, (int64_t)c->n_sm * 8));
    train_adam<<<ba, 256, 0, s>>>(dec->params, c->gparams, c->m_par, c->v_par, n0, p1, g1, m1, v1, n1, c->step,
                                  c->cfg.total_steps, c->cfg.lr0, c->cfg.lr1, 0.9f, 0.999f, 1e-8f, 1);
    MPM_CUDA_TRY(cudaGetLastError());
    st = decoder_refresh(dec, s);
    if (st != MPM_OK) return st;
    if (dec->n_tc > 0) {
      train_pack_transposed<<<std::max(1, dec->n_tc * 64), 256, 0, s>>>(dec->params, c->d_w_off, dec->n_tc, c->wtimg);
      MPM_CUDA_TRY(cudaGetLastError());
    }
    train_step_inc<<<1, 1, 0, s>>>(c->step);
    MPM_CUDA_TRY(cudaGetLastError());
  }
  return MPM_OK;
}

template <typename T>
mpm_status talloc(T** p, size_t count, bool zero = true) {
  cudaError_t e = cudaMalloc((void**)p, std::max<size_t>(count, 1) * sizeof(T));
  if (e != cudaSuccess) return set_error(MPM_ENOMEM, std::string("cudaMalloc: ") + cudaGetErrorString(e));
  if (zero) {
    e = cudaMemset(*p, 0, std::max<size_t>(count, 1) * sizeof(T));
    if (e != cudaSuccess) return set_error(MPM_ECUDA, std::string("cudaMemset: ") + cudaGetErrorString(e));
  }
  return MPM_OK;
}

mpm_status capture(trainer_ctx* c, int update, cudaGraphExec_t* out) {
  cudaGraph_t g = nullptr;
  MPM_CUDA_TRY(cudaStreamBeginCapture(c->cap_stream, cudaStreamCaptureModeThreadLocal));
  mpm_status st = train_launch_step(c, c->cap_stream, update);
  cudaError_t e = cudaStreamEndCapture(c->cap_stream, &g);
  if (st != MPM_OK) {
    if (g) cudaGraphDestroy(g);
    return st;
  }
  if (e != cudaSuccess) return set_error(MPM_ECUDA, std::string("graph capture: ") + cudaGetErrorString(e));
  e = cudaGraphInstantiate(out, g, 0);
  cudaGraphDestroy(g);
  if (e != cudaSuccess) return set_error(MPM_ECUDA, std::string("graph instantiate: ") + cudaGetErrorString(e));
  return MPM_OK;
}

}  // namespace

extern "C" {

mpm_status decoder_fit_scaling(mpm_decoder* dec, const snapshot_desc* sd, void* stream) {
  MPM_CHECK_ARG(dec && sd && sd->X && sd->x && sd->inst_offsets && sd->snap_inst, "null argument");
  MPM_CHECK_ARG(sd->dim == dec->d, "snapshot dim differs from the decoder's");
  MPM_CHECK_ARG(sd->n_inst >= 1 && sd->n_snap >= 1, "empty snapshot store");
  for (const void* ptr : {(const void*)sd->X, (const void*)sd->x}) {
    cudaPointerAttributes at{};
    if (cudaPointerGetAttributes(&at, ptr) != cudaSuccess) {
      cudaGetLastError();
      return set_error(MPM_EINVAL, "decoder_fit_scaling: X and x must be device pointers");
    }
    MPM_CHECK_ARG(at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged,
                  "decoder_fit_scaling: X and x must be device (or managed) pointers");
  }
  int64_t nx = 0;
  for (int s = 0; s < sd->n_snap; ++s) {
    const int inst = sd->snap_inst[s];
    MPM_CHECK_ARG(inst >= 0 && inst < sd->n_inst, "snap_inst out of range");
    nx += sd->inst_offsets[inst + 1] - sd->inst_offsets[inst];
  }
  const int64_t nX = sd->inst_offsets[sd->n_inst];
  MPM_CHECK_ARG(nX >= 1 && nx >= 1, "no particles");
  const int d = dec->d;
  cudaStream_t s = (cudaStream_t)stream;
  int devn = 0, n_sm = 0;
  MPM_CUDA_TRY(cudaGetDevice(&devn));
  MPM_CUDA_TRY(cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, devn));
  const int blocks = std::max(1, std::min<int>(n_sm * 4, (int)((std::max(nX, nx) + kScaleThreads - 1) / kScaleThreads)));
  double* mem = nullptr;
  MPM_CUDA_TRY(cudaMallocAsync((void**)&mem, sizeof(double) * ((size_t)blocks * 3 * d + 3 * d), s));
  double* part = mem;
  double* stats = mem + (size_t)blocks * 3 * d;
  scale_partials<<<blocks, kScaleThreads, 0, s>>>(0, d, sd->X, nX, sd->x, nx, nullptr, part);
  scale_finish<<<1, 32, 0, s>>>(0, d, blocks, nx, part, stats, nullptr);
  scale_partials<<<blocks, kScaleThreads, 0, s>>>(1, d, sd->X, nX, sd->x, nx, stats, part);
  scale_finish<<<1, 32, 0, s>>>(1, d, blocks, nx, part, stats, dec->norm);
  cudaError_t e = cudaGetLastError();
  cudaFreeAsync(mem, s);
  if (e != cudaSuccess) return set_error(MPM_ECUDA, std::string("decoder_fit_scaling: ") + cudaGetErrorString(e));
  return decoder_refresh(dec, s);
}

mpm_status trainer_create(mpm_decoder* dec, const train_config* cfg, const snapshot_desc* sd, const float* latents0,
                          trainer_ctx** out) {
  MPM_CHECK_ARG(dec && cfg && sd && out, "null argument");
  *out = nullptr;
  MPM_CHECK_ARG(dec->n_tc >= 1, "training needs at least two hidden layers (square tensor-core layers)");
  MPM_CHECK_ARG(sd->dim == dec->d, "snapshot dimension must match the decoder");
  MPM_CHECK_ARG(sd->n_inst >= 1 && sd->inst_offsets && sd->X, "instances");
  MPM_CHECK_ARG(sd->n_snap >= 1 && sd->snap_inst && sd->snap_next && sd->x && sd->v && sd->F, "snapshots");
  MPM_CHECK_ARG(cfg->batch >= 1 && cfg->dt_snap > 0 && cfg->lr0 > 0 && cfg->lr1 > 0, "batch, dt_snap, lr");
  MPM_CHECK_ARG(dec->r <= 32, "latent dimension <= 32");
  MPM_CHECK_ARG(cfg->shard_count >= 0 && cfg->shard_index >= 0 && cfg->shard_index < std::max(1, cfg->shard_count),
                "shard_index must be in [0, shard_count)");
  auto* c = new trainer_ctx();
  c->dec = dec;
  c->cfg = *cfg;
  c->d = dec->d;
  c->r = dec->r;
  c->R = c->d + 2;
  // whole points of R rows per 32 rows (decoder_bf16's order), or per 128 rows where that kernel
  // does not take the decoder (r > 28)
  c->Pt = 4 * (32 / c->R);
  c->pipe = decoder_train_pipe(dec, ((int64_t)cfg->batch + c->Pt - 1) / c->Pt * 128);
  if (!c->pipe) c->Pt = 128 / c->R;
  c->B = cfg->batch;
  c->i_offset = (int64_t)cfg->shard_index * cfg->batch;
  c->n_norm = (float)((double)cfg->batch * std::max(1, cfg->shard_count));
  c->n_tiles = (c->B + c->Pt - 1) / c->Pt;
  c->rows_total = c->n_tiles * 128;
  c->points_total = c->pipe ? c->n_tiles * c->Pt : 0;
  c->n_snap = sd->n_snap;
  int devn = 0;
  cudaGetDevice(&devn);
  cudaDeviceGetAttribute(&c->n_sm, cudaDevAttrMultiProcessorCount, devn);
  const int d = c->d, r = c->r;
  mpm_status st;
  struct Owner {  // destroys the partly built context on every early return
    trainer_ctx* c;
    ~Owner() { trainer_destroy(c); }
  } owner{c};
  // snapshot bookkeeping (host)
  std::vector<int64_t> base(sd->n_snap + 1, 0);
  for (int s = 0; s < sd->n_snap; ++s) {
    const int inst = sd->snap_inst[s];
    if (inst < 0 || inst >= sd->n_inst) return set_error(MPM_EINVAL, "snap_inst out of range");
    if (sd->snap_next[s] >= sd->n_snap) return set_error(MPM_EINVAL, "snap_next out of range");
    base[s + 1] = base[s] + (sd->inst_offsets[inst + 1] - sd->inst_offsets[inst]);
  }
  const int64_t total = base[sd->n_snap];
  const int64_t Ptot = sd->inst_offsets[sd->n_inst];
  if ((st = talloc(&c->snap_base, sd->n_snap + 1)) != MPM_OK) return st;
  if ((st = talloc(&c->snap_inst, sd->n_snap)) != MPM_OK) return st;
  if ((st = talloc(&c->snap_next, sd->n_snap)) != MPM_OK) return st;
  if ((st = talloc(&c->inst_off, sd->n_inst + 1)) != MPM_OK) return st;
  if ((st = talloc(&c->X, (size_t)Ptot * d, false)) != MPM_OK) return st;
  if ((st = talloc(&c->sx, (size_t)total * d, false)) != MPM_OK) return st;
  if ((st = talloc(&c->sv, (size_t)total * d, false)) != MPM_OK) return st;
  if ((st = talloc(&c->sF, (size_t)total * d * d, false)) != MPM_OK) return st;
  MPM_CUDA_TRY(cudaMemcpy(c->snap_base, base.data(), sizeof(int64_t) * (sd->n_snap + 1), cudaMemcpyHostToDevice));
  MPM_CUDA_TRY(cudaMemcpy(c->snap_inst, sd->snap_inst, sizeof(int32_t) * sd->n_snap, cudaMemcpyDefault));
  MPM_CUDA_TRY(cudaMemcpy(c->snap_next, sd->snap_next, sizeof(int32_t) * sd->n_snap, cudaMemcpyDefault));
  MPM_CUDA_TRY(cudaMemcpy(c->inst_off, sd->inst_offsets, sizeof(int64_t) * (sd->n_inst + 1), cudaMemcpyDefault));
  MPM_CUDA_TRY(cudaMemcpy(c->X, sd->X, sizeof(float) * Ptot * d, cudaMemcpyDefault));
  MPM_CUDA_TRY(cudaMemcpy(c->sx, sd->x, sizeof(float) * total * d, cudaMemcpyDefault));
  MPM_CUDA_TRY(cudaMemcpy(c->sv, sd->v, sizeof(float) * total * d, cudaMemcpyDefault));
  MPM_CUDA_TRY(cudaMemcpy(c->sF, sd->F, sizeof(float) * total * d * d, cudaMemcpyDefault));
  // latent table + optimiser state
  const size_t nl = (size_t)sd->n_snap * r;
  if ((st = talloc(&c->latents, nl)) != MPM_OK) return st;
  if (latents0) MPM_CUDA_TRY(cudaMemcpy(c->latents, latents0, sizeof(float) * nl, cudaMemcpyDefault));
  if ((st = talloc(&c->g_lat, nl)) != MPM_OK) return st;
  if ((st = talloc(&c->m_lat, nl)) != MPM_OK) return st;
  if ((st = talloc(&c->v_lat, nl)) != MPM_OK) return st;
  if (cfg->encoder_subset > 0) {
    c->enc = true;
    if (!enc_describe(d, r, cfg->encoder_subset, 0, &c->E))
      return set_error(MPM_EINVAL, "encoder_subset: d x subset must be in [32, 8192]");
    for (int i = 0; i < sd->n_inst; ++i)
      if (sd->inst_offsets[i + 1] - sd->inst_offsets[i] < cfg->encoder_subset)
        return set_error(MPM_EINVAL, "encoder_subset larger than an instance");
    const int np = c->E.n_params;
    if ((st = talloc(&c->U, (size_t)sd->n_snap * c->E.L[0], false)) != MPM_OK) return st;
    if ((st = talloc(&c->enc_p, np)) != MPM_OK) return st;
    if ((st = talloc(&c->enc_g, np)) != MPM_OK) return st;
    if ((st = talloc(&c->enc_m, np)) != MPM_OK) return st;
    if ((st = talloc(&c->enc_v, np)) != MPM_OK) return st;
    if ((st = talloc(&c->enc_ss, 2 * d)) != MPM_OK) return st;
    if ((st = talloc(&c->enc_work, 2 * d)) != MPM_OK) return st;
    if ((st = enc_prepare(c->E)) != MPM_OK) return st;
    if ((st = enc_moments(c->E, c->sx, c->snap_base, sd->n_snap, c->enc_work, c->enc_ss, 0)) != MPM_OK) return st;
    if ((st = enc_gather(c->E, c->sx, c->snap_base, sd->n_snap, c->enc_ss, c->U, 0)) != MPM_OK) return st;
    // Xavier-uniform initial weights (fan-in / fan-out of each layer's linear map), zero biases,
    // uniform numbers from SplitMix64 seeded with the training seed
    std::vector<float> h(np, 0.f);
    uint64_t state = cfg->seed ^ 0x656e636f646572ull;
    auto uni = [&](float lim) {
      state += 0x9E3779B97F4A7C15ull;
      uint64_t z = state;
      z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
      z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
      z ^= z >> 31;
      return lim * (2.f * (float)((z >> 40) * (1.0 / 16777216.0)) - 1.f);
    };
    const float lc = std::sqrt(6.f / (kEncKernel + 1));
    for (int l = 0; l < c->E.n_conv; ++l)
      for (int k = 0; k < kEncKernel; ++k) h[7 * l + k] = uni(lc);
    const int dc = c->E.L[c->E.n_conv];
    const float l1 = std::sqrt(6.f / (dc + kEncFC)), l2 = std::sqrt(6.f / (kEncFC + r));
    for (int i = 0; i < kEncFC * dc; ++i) h[c->E.oW1 + i] = uni(l1);
    for (int i = 0; i < r * kEncFC; ++i) h[c->E.oW2 + i] = uni(l2);
    MPM_CUDA_TRY(cudaMemcpy(c->enc_p, h.data(), sizeof(float) * np, cudaMemcpyHostToDevice));
  }
  if ((st = talloc(&c->gparams, dec->n_params)) != MPM_OK) return st;
  if ((st = talloc(&c->m_par, dec->n_params)) != MPM_OK) return st;
  if ((st = talloc(&c->v_par, dec->n_params)) != MPM_OK) return st;
  // batch
  const int64_t B = c->B;
  const size_t per_pt = (size_t)(d + 2 * r + d + d + d * d + 1);
  if ((st = talloc(&c->batch_mem, per_pt * B)) != MPM_OK) return st;
  if ((st = talloc(&c->batch_idx, (size_t)3 * B)) != MPM_OK) return st;
  float* m = c->batch_mem;
  c->b.B = B;
  c->b.X = m;
  m += B * d;
  c->b.xh = m;
  m += B * r;
  c->b.u = m;
  m += B * r;
  c->b.tx = m;
  m += B * d;
  c->b.tv = m;
  m += B * d;
  c->b.tF = m;
  m += B * d * d;
  c->b.mask = m;
  c->b.snap = c->batch_idx;
  c->b.next = c->batch_idx + B;
  c->b.part = c->batch_idx + 2 * B;
  // activation stores
  const size_t rows = (size_t)c->rows_total;
  if ((st = talloc(&c->fwd, (size_t)c->R * B * d)) != MPM_OK) return st;
  if ((st = talloc(&c->dstore, (size_t)dec->n_hidden * kW * (c->pipe ? (size_t)c->points_total : rows))) != MPM_OK)
    return st;
  if ((st = talloc(&c->astore, (size_t)dec->n_hidden * kW * rows)) != MPM_OK) return st;
  if ((st = talloc(&c->zbstore, (size_t)dec->n_tc * kW * rows)) != MPM_OK) return st;
  if ((st = talloc(&c->zb0, (size_t)kW * rows)) != MPM_OK) return st;
  if ((st = talloc(&c->g_lat_pt, (size_t)B * r)) != MPM_OK) return st;
  if ((st = talloc(&c->g_u_pt, (size_t)B * r)) != MPM_OK) return st;
  if ((st = talloc(&c->wtimg, (size_t)dec->n_tc * kLayerBytes)) != MPM_OK) return st;
  if ((st = talloc(&c->d_w_off, dec->w_off.size())) != MPM_OK) return st;
  MPM_CUDA_TRY(cudaMemcpy(c->d_w_off, dec->w_off.data(), sizeof(int64_t) * dec->w_off.size(), cudaMemcpyHostToDevice));
  if ((st = talloc(&c->step, 1)) != MPM_OK) return st;
  if ((st = talloc(&c->loss, 1)) != MPM_OK) return st;
  if ((st = talloc(&c->status, 1)) != MPM_OK) return st;
  c->st.d = d;
  c->st.r = r;
  c->st.n_snap = sd->n_snap;
  c->st.snap_base = c->snap_base;
  c->st.snap_inst = c->snap_inst;
  c->st.snap_next = c->snap_next;
  c->st.inst_off = c->inst_off;
  c->st.X = c->X;
  c->st.x = c->sx;
  c->st.v = c->sv;
  c->st.F = c->sF;
  c->bwd_smem = 1024 + kMaxTC * kLayerBytes + kLayerBytes + (size_t)2 * kExchRows * kChunkStride * 4 +
                2 * 64 * 128 * 2 + 128 * 3 * 4 + kW * 4 + sizeof(DecSmemTail);
  MPM_CUDA_TRY(cudaFuncSetAttribute(train_bwd_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)c->bwd_smem));
  if (c->pipe) {
    c->bwd_smem = bwd_pipe_smem_bytes();
    for (auto* f : {train_bwd_pipe<2>, train_bwd_pipe<3>})
      MPM_CUDA_TRY(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)c->bwd_smem));
    MPM_CUDA_TRY(cudaFuncSetAttribute(train_dw_gemm_image, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)dw_image_smem_bytes()));
  }
  for (auto* f : {train_dw0_lat<2>, train_dw0_lat<3>})
    MPM_CUDA_TRY(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dw0_smem_bytes()));
  MPM_CUDA_TRY(cudaFuncSetAttribute(train_dw0_pipe<2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)dw0_pipe_smem_bytes<2>()));
  MPM_CUDA_TRY(cudaFuncSetAttribute(train_dw0_pipe<3>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)dw0_pipe_smem_bytes<3>()));
  train_pack_transposed<<<std::max(1, dec->n_tc * 64), 256>>>(dec->params, c->d_w_off, dec->n_tc, c->wtimg);
  MPM_CUDA_TRY(cudaGetLastError());
  MPM_CUDA_TRY(cudaDeviceSynchronize());
  MPM_CUDA_TRY(cudaStreamCreateWithFlags(&c->cap_stream, cudaStreamNonBlocking));
  owner.c = nullptr;
  *out = c;
  return MPM_OK;
}

void trainer_destroy(trainer_ctx* c) {
  if (!c) return;
  if (c->graph) cudaGraphExecDestroy(c->graph);
  if (c->graph_noupdate) cudaGraphExecDestroy(c->graph_noupdate);
  if (c->cap_stream) cudaStreamDestroy(c->cap_stream);
  void* bufs[] = {c->snap_base, c->snap_inst, c->snap_next, c->inst_off, c->X, c->sx, c->sv, c->sF, c->latents,
                  c->g_lat, c->m_lat, c->v_lat, c->gparams, c->m_par, c->v_par, c->batch_mem, c->batch_idx, c->fwd,
                  c->dstore, c->astore, c->zbstore, c->zb0, c->g_lat_pt, c->g_u_pt, c->wtimg, c->d_w_off, c->step,
                  c->loss, c->status, c->U, c->enc_p, c->enc_g, c->enc_m, c->enc_v, c->enc_ss, c->enc_work};
  for (void* p : bufs) cudaFree(p);
  delete c;
}

mpm_status decoder_train(trainer_ctx* c, int n_steps, void* stream) {
  MPM_CHECK_ARG(c, "null context");
  MPM_CHECK_ARG(n_steps >= 0, "n_steps >= 0");
  if (!c->graph) {
    mpm_status st = capture(c, 1, &c->graph);
    if (st != MPM_OK) return st;
  }
  for (int i = 0; i < n_steps; ++i) MPM_CUDA_TRY(cudaGraphLaunch(c->graph, (cudaStream_t)stream));
  return MPM_OK;
}

mpm_status trainer_loss(trainer_ctx* c, double* loss, int64_t* step, void* stream) {
  MPM_CHECK_ARG(c, "null context");
  cudaStream_t s = (cudaStream_t)stream;
  double h = 0.0;
  MPM_CUDA_TRY(cudaMemcpyAsync(&h, c->loss, sizeof(double), cudaMemcpyDeviceToHost, s));
  if (step) MPM_CUDA_TRY(cudaMemcpyAsync(step, c->step, sizeof(int64_t), cudaMemcpyDefault, s));
  MPM_CUDA_TRY(cudaStreamSynchronize(s));
  if (loss) *loss = h / (double)c->n_norm;
  return MPM_OK;
}

mpm_status trainer_gradient_sizes(const trainer_ctx* c, int64_t* n_params, int64_t* n_second) {
  MPM_CHECK_ARG(c, "null context");
  if (n_params) *n_params = c->dec->n_params;
  if (n_second) *n_second = c->enc ? (int64_t)c->E.n_params : c->n_snap * c->r;
  return MPM_OK;
}

mpm_status trainer_compute_gradients(trainer_ctx* c, float* g_params, float* g_second, void* stream) {
  MPM_CHECK_ARG(c && g_params && g_second, "null argument");
  cudaStream_t s = (cudaStream_t)stream;
  mpm_status st = train_launch_step(c, s, 0);
  if (st != MPM_OK) return st;
  const size_t n1 = c->enc ? (size_t)c->E.n_params : (size_t)c->n_snap * c->r;
  float* g1 = c->enc ? c->enc_g : c->g_lat;
  MPM_CUDA_TRY(cudaMemcpyAsync(g_params, c->gparams, sizeof(float) * c->dec->n_params, cudaMemcpyDeviceToDevice, s));
  MPM_CUDA_TRY(cudaMemcpyAsync(g_second, g1, sizeof(float) * n1, cudaMemcpyDeviceToDevice, s));
  MPM_CUDA_TRY(cudaMemsetAsync(c->gparams, 0, sizeof(float) * c->dec->n_params, s));
  MPM_CUDA_TRY(cudaMemsetAsync(c->g_lat, 0, sizeof(float) * c->n_snap * c->r, s));
  if (c->enc) MPM_CUDA_TRY(cudaMemsetAsync(c->enc_g, 0, sizeof(float) * c->E.n_params, s));
  return MPM_OK;
}

mpm_status trainer_apply_gradients(trainer_ctx* c, const float* g_params, const float* g_second, void* stream) {
  MPM_CHECK_ARG(c && g_params && g_second, "null argument");
  cudaStream_t s = (cudaStream_t)stream;
  const size_t n1 = c->enc ? (size_t)c->E.n_params : (size_t)c->n_snap * c->r;
  float* g1 = c->enc ? c->enc_g : c->g_lat;
  MPM_CUDA_TRY(cudaMemcpyAsync(c->gparams, g_params, sizeof(float) * c->dec->n_params, cudaMemcpyDeviceToDevice, s));
  MPM_CUDA_TRY(cudaMemcpyAsync(g1, g_second, sizeof(float) * n1, cudaMemcpyDeviceToDevice, s));
  return train_launch_update(c, s);
}

mpm_status trainer_get_latents(trainer_ctx* c, float* latents, void* stream) {
  MPM_CHECK_ARG(c && latents, "null argument");
  MPM_CUDA_TRY(cudaMemcpyAsync(latents, c->latents, sizeof(float) * c->n_snap * c->r, cudaMemcpyDefault,
                               (cudaStream_t)stream));
  return MPM_OK;
}

mpm_status trainer_status_word(trainer_ctx* c, uint32_t* out, int clear, void* stream) {
  MPM_CHECK_ARG(c && out, "null argument");
  cudaStream_t s = (cudaStream_t)stream;
  uint32_t h = 0;
  MPM_CUDA_TRY(cudaMemcpyAsync(&h, c->status, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
  if (clear) MPM_CUDA_TRY(cudaMemsetAsync(c->status, 0, sizeof(uint32_t), s));
  MPM_CUDA_TRY(cudaStreamSynchronize(s));
  *out = h;
  return MPM_OK;
}

mpm_status trainer_gradients(trainer_ctx* c, float* g_params, float* g_latents, float* g_encoder, int32_t* batch_snap,
                             int32_t* batch_part, double* loss, void* stream) {
  MPM_CHECK_ARG(c, "null context");
  cudaStream_t s = (cudaStream_t)stream;
  // one forward + backward on the batch of the current step, no update
  mpm_status st = train_launch_step(c, s, 0);
  if (st != MPM_OK) return st;
  if (g_params) MPM_CUDA_TRY(cudaMemcpyAsync(g_params, c->gparams, sizeof(float) * c->dec->n_params, cudaMemcpyDefault, s));
  if (g_latents) MPM_CUDA_TRY(cudaMemcpyAsync(g_latents, c->g_lat, sizeof(float) * c->n_snap * c->r, cudaMemcpyDefault, s));
  if (g_encoder && c->enc)
    MPM_CUDA_TRY(cudaMemcpyAsync(g_encoder, c->enc_g, sizeof(float) * c->E.n_params, cudaMemcpyDefault, s));
  if (batch_snap) MPM_CUDA_TRY(cudaMemcpyAsync(batch_snap, c->b.snap, sizeof(int32_t) * c->B, cudaMemcpyDefault, s));
  if (batch_part) MPM_CUDA_TRY(cudaMemcpyAsync(batch_part, c->b.part, sizeof(int32_t) * c->B, cudaMemcpyDefault, s));
  double h = 0.0;
  MPM_CUDA_TRY(cudaMemcpyAsync(&h, c->loss, sizeof(double), cudaMemcpyDeviceToHost, s));
  MPM_CUDA_TRY(cudaMemsetAsync(c->gparams, 0, sizeof(float) * c->dec->n_params, s));
  MPM_CUDA_TRY(cudaMemsetAsync(c->g_lat, 0, sizeof(float) * c->n_snap * c->r, s));
  if (c->enc) MPM_CUDA_TRY(cudaMemsetAsync(c->enc_g, 0, sizeof(float) * c->E.n_params, s));
  MPM_CUDA_TRY(cudaStreamSynchronize(s));
  if (loss) *loss = h / (double)c->n_norm;
  return MPM_OK;
}

mpm_status trainer_encoder_params(trainer_ctx* c, float* params, float* shift_scale, int64_t* n_params, void* stream) {
  MPM_CHECK_ARG(c, "null context");
  MPM_CHECK_ARG(c->enc, "the trainer has no encoder (train_config.encoder_subset = 0)");
  cudaStream_t s = (cudaStream_t)stream;
  if (n_params) *n_params = c->E.n_params;
  if (params) MPM_CUDA_TRY(cudaMemcpyAsync(params, c->enc_p, sizeof(float) * c->E.n_params, cudaMemcpyDefault, s));
  if (shift_scale) MPM_CUDA_TRY(cudaMemcpyAsync(shift_scale, c->enc_ss, sizeof(float) * 2 * c->d, cudaMemcpyDefault, s));
  MPM_CUDA_TRY(cudaStreamSynchronize(s));
  return MPM_OK;
}

mpm_status trainer_set_encoder_params(trainer_ctx* c, const float* params, const float* shift_scale, void* stream) {
  MPM_CHECK_ARG(c, "null context");
  MPM_CHECK_ARG(c->enc, "the trainer has no encoder (train_config.encoder_subset = 0)");
  cudaStream_t s = (cudaStream_t)stream;
  if (params) MPM_CUDA_TRY(cudaMemcpyAsync(c->enc_p, params, sizeof(float) * c->E.n_params, cudaMemcpyDefault, s));
  if (shift_scale) {
    MPM_CUDA_TRY(cudaMemcpyAsync(c->enc_ss, shift_scale, sizeof(float) * 2 * c->d, cudaMemcpyDefault, s));
    mpm_status st = enc_gather(c->E, c->sx, c->snap_base, c->n_snap, c->enc_ss, c->U, s);
    if (st != MPM_OK) return st;
  }
  MPM_CUDA_TRY(cudaMemsetAsync(c->enc_m, 0, sizeof(float) * c->E.n_params, s));
  MPM_CUDA_TRY(cudaMemsetAsync(c->enc_v, 0, sizeof(float) * c->E.n_params, s));
  MPM_CUDA_TRY(cudaStreamSynchronize(s));
  return MPM_OK;
}

mpm_status trainer_encode(trainer_ctx* c, const float* x, int64_t n, int64_t n_particles, float* latents,
                          void* stream) {
  MPM_CHECK_ARG(c, "null context");
  MPM_CHECK_ARG(c->enc, "the trainer has no encoder (train_config.encoder_subset = 0)");
  MPM_CHECK_ARG(n >= 0 && n_particles >= c->E.n_sub, "n >= 0 and n_particles >= the encoder subset");
  if (n == 0) return MPM_OK;
  MPM_CHECK_ARG(x && latents, "null argument");
  cudaStream_t s = (cudaStream_t)stream;
  const int d = c->d;
  float *xd = nullptr, *Ud = nullptr, *ld = nullptr;
  int64_t* base = nullptr;
  std::vector<int64_t> hb(n + 1);
  for (int64_t i = 0; i <= n; ++i) hb[i] = i * n_particles;
  mpm_status st = MPM_OK;
  cudaError_t e = cudaMalloc((void**)&xd, sizeof(float) * n * n_particles * d);
  if (e == cudaSuccess) e = cudaMalloc((void**)&Ud, sizeof(float) * n * c->E.L[0]);
  if (e == cudaSuccess) e = cudaMalloc((void**)&ld, sizeof(float) * n * c->r);
  if (e == cudaSuccess) e = cudaMalloc((void**)&base, sizeof(int64_t) * (n + 1));
  if (e == cudaSuccess) e = cudaMemcpyAsync(xd, x, sizeof(float) * n * n_particles * d, cudaMemcpyDefault, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(base, hb.data(), sizeof(int64_t) * (n + 1), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) {
    st = enc_gather(c->E, xd, base, n, c->enc_ss, Ud, s);
    if (st == MPM_OK) st = enc_forward(c->E, c->enc_p, Ud, n, ld, c->n_sm, s);
    if (st == MPM_OK) e = cudaMemcpyAsync(latents, ld, sizeof(float) * n * c->r, cudaMemcpyDefault, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  }
  cudaFree(xd);
  cudaFree(Ud);
  cudaFree(ld);
  cudaFree(base);
  if (e != cudaSuccess) return set_error(MPM_ECUDA, std::string("trainer_encode: ") + cudaGetErrorString(e));
  return st;
}

}  // extern "C"
