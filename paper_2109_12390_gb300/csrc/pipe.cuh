// Pieces of the alternating-tile pipelines (decoder_tc3, decoder_bf16, train_bwd_pipe): sixteen
// epilogue warps take the tile slots of a CTA in turn, one warp per slot issues its MMAs.  Barriers,
// packed FP32 arithmetic, and the mapping of a call's rows to tiles.
#pragma once

#include "decoder_common.cuh"
#include "ring.cuh"

namespace mpmrom {

constexpr int kEpiThreads = 512;          // epilogue threads
constexpr int kAtomBytes = kW * 128;      // 128 rows x 64 BF16

// Bounded wait; after a timeout anywhere in the CTA no further waits are made.  Whether the phase was seen complete.
__device__ __forceinline__ bool pipe_wait(uint32_t* status, int* abort, uint64_t* bar, uint32_t phase) {
  if (*(volatile int*)abort) return false;
  if (tc::mbar_wait(bar, phase)) return true;
  raise_status(status, STATUS_TIMEOUT);
  atomicExch(abort, 1);
  return false;
}

// Barriers 1 + s: the epilogue warps arrive when slot s's next operand is complete (and its
// accumulator read), the slot's issuer warp waits.  Barriers 3 + s: the issuer arrives when the
// accumulator is complete, the epilogue warps wait (blocked, where polling the MMA barrier would
// take issue slots).  Barrier 5: the column parts' output sums are in shared memory.
__device__ __forceinline__ void pipe_arrive(int id) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "n"(kEpiThreads + 32) : "memory");
}
__device__ __forceinline__ void pipe_sync(int id) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(kEpiThreads + 32) : "memory");
}
__device__ __forceinline__ void pipe_combine(int part) {
  if (part == 3) asm volatile("bar.sync 5, %0;" ::"n"(kEpiThreads) : "memory");
  else asm volatile("bar.arrive 5, %0;" ::"n"(kEpiThreads) : "memory");
}

// 2^x on the special-function unit, results below the normal range flushed to zero
__device__ __forceinline__ float ex2_ftz(float x) {
  float e;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(x));
  return e;
}
// Pairs of FP32 operations in one instruction (each rounded as the scalar operation)
__device__ __forceinline__ void add2(float& a0, float& a1, float b0, float b1) {
  asm("{\n .reg .b64 a, b;\n mov.b64 a, {%0, %1};\n mov.b64 b, {%2, %3};\n add.rn.f32x2 a, a, b;\n"
      " mov.b64 {%0, %1}, a;\n}\n"
      : "+f"(a0), "+f"(a1)
      : "f"(b0), "f"(b1));
}
__device__ __forceinline__ void mul2(float& a0, float& a1, float b) {
  asm("{\n .reg .b64 a, b;\n mov.b64 a, {%0, %1};\n mov.b64 b, {%2, %2};\n mul.rn.f32x2 a, a, b;\n"
      " mov.b64 {%0, %1}, a;\n}\n"
      : "+f"(a0), "+f"(a1)
      : "f"(b));
}
__device__ __forceinline__ void fma2(float& a0, float& a1, float b0, float b1, float c) {   // a += b c
  asm("{\n .reg .b64 a, b, c;\n mov.b64 a, {%0, %1};\n mov.b64 b, {%2, %3};\n mov.b64 c, {%4, %4};\n"
      " fma.rn.f32x2 a, b, c, a;\n mov.b64 {%0, %1}, a;\n}\n"
      : "+f"(a0), "+f"(a1)
      : "f"(b0), "f"(b1), "f"(c));
}
// Biases enter the primal rows with a factor 1 and the others with a factor 0 (a select of the value or of the
// address costs the epilogues 2 to 5 %), so an infinite one, a unit that is switched off, becomes the largest
// finite number: the same activation and derivatives on either side, and no NaN on the rows without it.
__device__ __forceinline__ float finite_bias(float b) {
  constexpr float big = 3.402823466e38f;
  return b < -big ? -big : b > big ? big : b;
}
// What the rows of a call need of their activations (a template parameter: one variant's code per
// kernel keeps the epilogue loop small)
enum { PIPE_PRIMAL = 0, PIPE_TANGENT = 1, PIPE_SECANT = 2, PIPE_IDENTITY = 3 };
constexpr float kLog2e = 1.4426950408889634f;   // __expf(z) is 2^(z kLog2e)

// One thread's row of a tile slot (rows and points are counted in 32 bits: pipe_launch's callers take
// another kernel for 2^31 rows or more).
struct PipeRow {
  int cls, psrc, kidx;   // class, lane of the point's primal row, output block (-1: not written)
  int p;                 // point
};
// Its raw first-layer inputs 8 c .. 8 c + 7 in the padded layout (coordinates at 0 .. 3, latents from
// kTcLat): latents or directions, and coordinates of primal rows as stored; hot is the one-hot entry
// of a tangent row (-1: none).
struct PipeIn {
  float v[8];
  int hot;
  bool primal;
};

// Row of a lane in the lane group whose first row is g0 (rows in (point, kind) order, U per group).
// TRAIN: whole points, U <= 32 of the group's lanes (the others idle).
template <int MODE, bool TRAIN>
__device__ __forceinline__ PipeRow pipe_row(const DecArgs& a, int g0, int U, int n_rows, int lane, int& kind) {
  PipeRow rs;
  kind = -1;
  rs.cls = -1;
  rs.psrc = lane;
  rs.kidx = -1;
  if (TRAIN) {
    const int q = lane / a.R, k = lane - q * a.R;
    rs.p = g0 / a.R + q;
    if (lane < U && g0 + lane < n_rows) {
      kind = a.kinds[k];
      rs.cls = kind_class(kind);
      rs.kidx = k;
      rs.psrc = lane - k;
    }
    return rs;
  }
  if (MODE == PIPE_PRIMAL) {
    rs.p = g0 + lane;
    if (rs.p < n_rows) kind = rs.cls = rs.kidx = 0;
    return rs;
  }
  const int p0 = (int)((uint32_t)g0 / (uint32_t)a.R);   // point of the group's first row
  const int row = U == 32 ? g0 + lane : lane == 0 ? p0 * a.R : g0 + lane - 1;
  const uint32_t off = (uint32_t)(row - p0 * a.R);      // 0 .. R + 30
  const int dp = (int)(off / (uint32_t)a.R), k = (int)off - dp * a.R;
  rs.p = p0 + dp;
  if (row < n_rows) {
    kind = a.kinds[k];
    rs.cls = kind_class(kind);
    rs.kidx = (U != 32 && lane == 0) ? -1 : k;
    rs.psrc = U == 32 ? lane - k : max(lane - k, 0);    // before the group's first row: lane 0's copy
  }
  return rs;
}

// The row's inputs (loads only: pipe_finish does the arithmetic, so that the loads stay in flight).
// vec4: latent and direction rows are 16-byte aligned and r is a multiple of 4.
template <int MODE, bool TRAIN = false>
__device__ __forceinline__ PipeRow pipe_load(const DecArgs& a, int g0, int U, int n_rows, int lane, int c, bool vec4,
                                             PipeIn& in) {
  int kind;
  const PipeRow rs = pipe_row<MODE, TRAIN>(a, g0, U, n_rows, lane, kind);
  const float *vec = nullptr, *xp = nullptr;   // latent part, coordinates
  in.hot = -1;
  in.primal = rs.cls == 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) in.v[j] = 0.f;
  if (rs.cls >= 0) {
    int64_t xrow = rs.p;
    int li = 0;
    if (a.n_dev && a.n_rep <= 1) {
      if (a.idx) xrow = a.idx[rs.p];           // one latent row: point p is row idx[p]
    } else if (!a.n_dev) {
      li = a.lat ? a.lat[rs.p] : a.lat_per_point ? rs.p : 0;
    } else {
      RowInfo ri;
      ri.p = rs.p;
      row_source(a, ri, xrow, li);
    }
    if (rs.cls == 0) {
      vec = a.latents + (int64_t)li * a.r;
      xp = a.X + xrow * a.d;
    } else if (rs.cls == 1 && kind != KIND_JVP) {
      in.hot = kind - 1 < a.d ? kind - 1 : kind - 1 - a.d + kTcLat;
    } else {
      vec = a.dirs + dir_offset(a, kind, li);
    }
  }
  const int i0 = 8 * c - kTcLat;               // latent index of the first input
  if (c == 0 && xp) {
#pragma unroll
    for (int j = 0; j < 3; ++j)
      if (j < a.d) in.v[j] = xp[j];
  }
  if (vec) {
    if (vec4) {
      if (c > 0 && i0 < a.r) {
        const float4 q = *reinterpret_cast<const float4*>(vec + i0);
        in.v[0] = q.x;
        in.v[1] = q.y;
        in.v[2] = q.z;
        in.v[3] = q.w;
      }
      if (i0 + 4 < a.r) {
        const float4 q = *reinterpret_cast<const float4*>(vec + i0 + 4);
        in.v[4] = q.x;
        in.v[5] = q.y;
        in.v[6] = q.z;
        in.v[7] = q.w;
      }
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (i0 + j >= 0 && i0 + j < a.r) in.v[j] = vec[i0 + j];
    }
  }
  return rs;
}
template <int MODE>
__device__ __forceinline__ void pipe_finish(int d, const float* norm, int c, PipeIn& in) {
  if (c == 0) {
#pragma unroll
    for (int j = 0; j < 3; ++j)
      if (j < d) in.v[j] = in.primal ? (in.v[j] - norm[j]) / norm[d + j] : in.hot == j ? 1.f / norm[d + j] : 0.f;
  }
  if (MODE != PIPE_PRIMAL) {
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (8 * c + j == in.hot && in.hot >= kTcLat) in.v[j] = 1.f;
  }
}
__device__ __forceinline__ bool pipe_vec4(const DecArgs& a) {
  return (a.r & 3) == 0 && (((uintptr_t)a.latents | (uintptr_t)a.dirs) & 15u) == 0;
}

}  // namespace mpmrom
