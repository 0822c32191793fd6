// Row helpers of the 2D tile kernels (TMA per-step and batched): a thread owns
// a few columns of a shared-memory box (80 floats wide: 8 halo columns each
// side of a 64-column tile) and slides a register window of 2R+1 rows down its
// run of rows.
//
// The zero-sum Laplacian of a cell is the sum over the y, then the x taps of
// w_m [(a + b) - 2c] (pair form, 3 FP operations per tap) or
// w_m [(a - c) + (b - c)] (difference form, rounding relative to the
// differences: for fields with a large smooth part).  The low part of a
// compensated pair (a field of the order of the rounding error of its high
// part) takes the cheapest form, sum_m w_m (a + b) - w_c c with the centre
// weight w_c = 4 sum_m w_m summed in FP32 (R additions and a multiply, so up to
// R + 1 roundings): 2 FP operations per tap; the rounded w_c departs from a
// zero-sum stencil by a relative ~R 2^-24 of a field that is itself ~2^-24 of
// the state.
#pragma once

#include "stencil.cuh"

namespace pat {

// ------------------------------------------------ NP column pairs per thread
// A thread owns 2 NP columns (NP packed FP32x2 pairs, the first at a multiple of 2 NP) of RUN consecutive
// rows; `own` points at the thread's first cell in a shared-memory box.

// 2 NP consecutive floats of a box row
template <int NP>
struct Cells {
  float2 v[NP];
  __device__ __forceinline__ void load(const float* __restrict__ p) {
    if (NP == 1) {
      v[0] = *reinterpret_cast<const float2*>(p);
    } else {
#pragma unroll
      for (int k = 0; k < NP / 2; ++k) {
        const float4 q = *reinterpret_cast<const float4*>(p + 4 * k);
        v[2 * k] = lo2(q);
        v[NP == 1 ? 0 : 2 * k + 1] = hi2(q);
      }
    }
  }
  __device__ __forceinline__ void store(float* __restrict__ p) const {
    if (NP == 1) {
      *reinterpret_cast<float2*>(p) = v[0];
    } else {
#pragma unroll
      for (int k = 0; k < NP / 2; ++k)
        *reinterpret_cast<float4*>(p + 4 * k) = make_float4(v[2 * k].x, v[2 * k].y, v[NP == 1 ? 0 : 2 * k + 1].x,
                                                            v[NP == 1 ? 0 : 2 * k + 1].y);
    }
  }
  // global loads: streamed (read once per launch, no L1 allocation) and read-only
  __device__ __forceinline__ void stream(const float* p) {
    if (NP == 1) {
      asm volatile("ld.global.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(v[0].x), "=f"(v[0].y) : "l"(p));
    } else {
#pragma unroll
      for (int k = 0; k < NP / 2; ++k) {
        const float4 q = ld_stream4(p + 4 * k);
        v[2 * k] = lo2(q);
        v[NP == 1 ? 0 : 2 * k + 1] = hi2(q);
      }
    }
  }
  __device__ __forceinline__ void ldg(const float* p) {
    if (NP == 1) {
      v[0] = __ldg(reinterpret_cast<const float2*>(p));
    } else {
#pragma unroll
      for (int k = 0; k < NP / 2; ++k) {
        const float4 q = __ldg(reinterpret_cast<const float4*>(p + 4 * k));
        v[2 * k] = lo2(q);
        v[NP == 1 ? 0 : 2 * k + 1] = hi2(q);
      }
    }
  }
  __device__ __forceinline__ void fill(float a) {
#pragma unroll
    for (int k = 0; k < NP; ++k) v[k] = dup2(a);
  }
  __device__ __forceinline__ float get(int j) const { return (j & 1) ? v[j / 2].y : v[j / 2].x; }
};

template <int NP>
__device__ __forceinline__ void store_cells(float* __restrict__ p, const float (&a)[2 * NP]) {
  Cells<NP> c;
#pragma unroll
  for (int k = 0; k < NP; ++k) c.v[k] = make_float2(a[2 * k], a[2 * k + 1]);
  c.store(p);
}

// The thread's row with R columns either side: aligned pieces of the own width, the own piece handed in (it is
// in the window already).
template <int R, int NP>
struct Row {
  static constexpr int W = 2 * NP, HP = (R + W - 1) / W;  // pieces either side
  Cells<NP> piece[2 * HP + 1];
  __device__ __forceinline__ void load(const float* __restrict__ own, const Cells<NP>& c) {
#pragma unroll
    for (int k = 0; k < 2 * HP + 1; ++k) {
      if (k == HP)
        piece[k] = c;
      else
        piece[k].load(own + W * (k - HP));
    }
  }
  __device__ __forceinline__ float at(int o) const {  // offset from the thread's first column
    const int i = o + W * HP;
    return piece[i / W].get(i % W);
  }
  __device__ __forceinline__ float2 pair(int o) const { return make_float2(at(o), at(o + 1)); }
};

// a + b of two pairs.  An odd shift straddles two aligned register pairs: packed arithmetic would first move
// both halves, so those take two scalar additions (the same rounding).
__device__ __forceinline__ float2 add_pair(float2 a, float2 b, bool aligned) {
  return aligned ? __fadd2_rn(a, b) : make_float2(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y));
}

// Laplacian of pair p of the row: y taps from the window (win[i] = row - R + i), x taps from the row, in
// that order, added to acc; each lane rounds as the scalar form would.
template <int R, bool DIFF, int NP>
__device__ __forceinline__ float2 stencil_pair(const Cells<NP> (&win)[2 * R + 1], const Row<R, NP>& f, int p,
                                               const float2 (&w2)[R + 1], float2 acc = make_float2(0.f, 0.f)) {
  const float2 c = win[R].v[p];
  const float2 nc = __fmul2_rn(c, dup2(-1.f));
#pragma unroll
  for (int m = 1; m <= R; ++m) acc = __ffma2_rn(w2[m], pair_term2<DIFF>(win[R + m].v[p], win[R - m].v[p], c, nc), acc);
#pragma unroll
  for (int m = 1; m <= R; ++m) {
    const bool even = m % 2 == 0;
    const float2 rt = f.pair(2 * p + m), lt = f.pair(2 * p - m);
    float2 t;
    if (DIFF)
      t = __fadd2_rn(add_pair(rt, nc, even), add_pair(lt, nc, even));
    else
      t = __ffma2_rn(c, dup2(-2.f), add_pair(rt, lt, even));
    acc = __ffma2_rn(w2[m], t, acc);
  }
  return acc;
}

// The low part's stencil of pair p of the row, centre weight -nwc.
template <int R, int NP>
__device__ __forceinline__ float2 stencil_low(const Cells<NP> (&win)[2 * R + 1], const Row<R, NP>& f, int p,
                                              const float2 (&w2)[R + 1], float2 nwc) {
  float2 acc = __fmul2_rn(nwc, win[R].v[p]);
#pragma unroll
  for (int m = 1; m <= R; ++m) acc = __ffma2_rn(w2[m], __fadd2_rn(win[R + m].v[p], win[R - m].v[p]), acc);
#pragma unroll
  for (int m = 1; m <= R; ++m)
    acc = __ffma2_rn(w2[m], add_pair(f.pair(2 * p + m), f.pair(2 * p - m), m % 2 == 0), acc);
  return acc;
}

// The low part's stencil of the thread's RUN rows (box pitch BW): lo[rr].
template <int R, int RUN, int BW, int NP>
__device__ __forceinline__ void stencil_run_pair(const float* __restrict__ own, const float2 (&w2)[R + 1], float2 nwc,
                                                 Cells<NP> (&lo)[RUN]) {
  Cells<NP> win[2 * R + 1];
#pragma unroll
  for (int i = 0; i < 2 * R; ++i) win[i].load(own + (i - R) * BW);
#pragma unroll
  for (int rr = 0; rr < RUN; ++rr) {
    win[2 * R].load(own + (rr + R) * BW);
    Row<R, NP> f;
    f.load(own + rr * BW, win[R]);
#pragma unroll
    for (int p = 0; p < NP; ++p) lo[rr].v[p] = stencil_low<R, NP>(win, f, p, w2, nwc);
#pragma unroll
    for (int i = 0; i < 2 * R; ++i) win[i] = win[i + 1];
  }
}

}  // namespace pat
