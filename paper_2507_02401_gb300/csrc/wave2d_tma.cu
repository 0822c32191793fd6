// 2D wave step with TMA-fed tile pipelines: one launch per time step of the
// increment form (paper Sec. 2, Eq. wave_equation, eliminated to p only)
//
//   forward:  D^{n+1} = D^n + c_lap (kappa_hi + kappa_lo) L P^n,   P^{n+1} = P^n + D^{n+1}
//   adjoint:  G^m = G^{m+1} + S^T r_m + c_lap L(kappa Q^{m+1}),    Q^m = Q^{m+1} + G^m
//             (final step: x = G^0 = G^1 + S^T r_0 + 1/2 L(kappa Q^1))
//
// The adjoint runs in the variable Z = kappa Q (constant or varying medium):
// Z^m = Z^{m+1} + kappa G^m, and the stencil acts on Z directly.  In a closed
// box Z integrates G over time and grows far beyond the result, so Z is kept
// as a compensated pair Z + Z_lo (TwoSum), the stencil sees both parts
// (Z through the difference form (a - c) + (b - c), whose rounding is relative
// to the differences, Z_lo through the cheapest sum form), and G is plain.
// FP32 emulation of the 512^2, 1500-step, order-8 adjoint with noisy data
// simulated from a phantom: 1.9e-5 for the plain pair-form recurrence
// (constant and varying medium), 1.5e-5 with the difference form alone,
// 7e-7 with the compensated Z.  Each step also adds S^T r_{m-1}, the sensor
// injection of the step after it, to the G it has just stored (lists per tile).
//
// Persistent CTAs walk 64 x 32 tiles (64 x 64 in the forward on very large
// fields, see below); one thread issues the TMA load of the next tile's boxes
// (80 x (32+2R) floats, halo included, zero outside the grid: P for the forward, Z and Z_lo for the adjoint) into the second of two
// shared-memory stages while the CTA computes the current one.  Each thread
// owns 4 columns x 4 consecutive rows: y neighbours come from a sliding
// register window of 2R+1 rows, x neighbours from the shared-memory row; its
// own D / G cells are loaded straight into registers before the wait for the
// boxes, as is kappa in the forward from order 4 on; kappa otherwise and G_lo
// two rows ahead of their use.
// Compulsory DRAM traffic per point-update: forward P and D read, P^{n+1} and
// D^{n+1} written (16 B), plus kappa hi/lo (8 B) for a varying medium;
// adjoint Z, Z_lo, G read and written (24 B), plus kappa (4 B) for a varying
// medium.
#include <cudaTypedefs.h>

#include <type_traits>

#include "internal.h"
#include "stencil.cuh"
#include "tile2d.cuh"
#include "tma.cuh"

namespace pat {
namespace {

// 64 x 32 tiles, 128 threads, each with 2 NP columns x RUN rows.  Measured at order 8, K / K* us per step, on
// 4000 x 3600 | 1400^2 | 1024^2 cells:
//   4 columns x 4 rows, 64 x 32 tiles (3 CTAs per SM)   39.8 / 69.9 | 7.2 / 12.0 | 4.5 / 8.5
//   2 columns x 8 rows, 64 x 64 tiles (2 CTAs per SM)   42.0 / 76.9 | 8.0 / 14.5 | 4.7 / 8.3
//   2 columns x 8 rows, 64 x 32 tiles (3 CTAs)          42.0 / 73.1 | 8.0 / 12.5 | 4.8 / 8.9
//   4 columns x 8 rows, 64 x 64 tiles (2 to 3 CTAs)     40.0 / 93.1 | 6.8 / 16.6 | 5.8 / 9.5
// The first needs the fewest shared-memory wavefronts per cell of those that leave 12 warps on an SM in the
// adjoint, whose two stencils keep the FP32 and shared-memory pipes about half busy each.
//
// Forward steps of a constant medium, on rows of whole 128-byte lines and fields of 256 MiB or more, take tiles twice
// as tall, a CTA of 256 threads each, two CTAs per SM: there DRAM is the bound, and it serves 64 rows of a tile better
// than 32.  K us per step, tall | not: order 8 16384^2 653 | 786, 12000^2 350 | 386, 8192^2 159 | 161, 4096^2 41.8 |
// 40.4; order 2 627 | 726, 339 | 378, 150 | 163, 37.2 | 35.1.  Rows that are no multiple of 128 bytes do not gain
// (12000 x 12004 order 8 503 | 497), nor do varying media (12000^2 order 2 563 | 508) and the adjoint.
constexpr int TX = 64, NP = 2, TCOLS = TX / (2 * NP), RUN = 4;
__host__ __device__ constexpr int tile_y(bool tall) { return tall ? 64 : 32; }
__host__ __device__ constexpr int threads_of(bool tall) { return TCOLS * (tile_y(tall) / RUN); }
// CTAs per SM to leave registers for: a fourth pays up to order 4 (1024^2 order 4 K* 6.3 against 7.4 us), except
// in the full form, which spills then (1000 x 875 order 4 K* 7.8 against 6.8 us)
constexpr int min_ctas(int R, bool full, bool grad, bool tall) { return grad || tall ? 2 : R <= 3 && !full ? 4 : 3; }
constexpr int XH = 8;            // box columns left of the tile (>= R, 16-byte aligned)
constexpr int BW = TX + 2 * XH;  // box width, 80 floats

template <int R, int NBOX = 1, bool TALL = false>
struct G2 {
  static constexpr int BH = tile_y(TALL) + 2 * R;
  static constexpr int PBOX = BW * BH;       // floats (multiple of 32: 128-byte aligned)
  static constexpr int STAGE = NBOX * PBOX;  // the adjoint stages Z and Z_lo
  static constexpr size_t USED = sizeof(float) * 2 * STAGE + 16;
  // Tall tiles: two CTAs per SM and no room for a third, which the next step's grid, launched programmatically, would
  // take on some SMs and leave others with one of its CTAs (order 2, whose registers leave that room: 12000^2 339 us
  // per step so, 358 with it).
  static constexpr size_t SMEM = TALL && R == 1 ? 100 * 1024 : USED;
};

// Sensor s = b + t * gridDim.x is sampled by thread t of CTA b (the sensors spread over every CTA).
__device__ __forceinline__ void fused_sample2(const StepArgs& a, long long bid, int t) {
  const long long gs = bid + (long long)t * gridDim.x;
  if (a.y == nullptr || gs >= a.ns) return;
  const int s = (int)gs;
  float v = 0.f;
  for (int k = 0; k < a.corners; ++k) v = fmaf(a.sens_w[s * a.corners + k], a.cur[a.sens_cell[s * a.corners + k]], v);
  a.y[(long long)s * a.nt + a.t_sample] = v;
}

// MODE 0: constant medium, forward; 1: varying medium, forward; 2: adjoint (either medium) in
// Z = kappa Q with Z compensated.  SP 0: no absorbing layer; 1: layer, forward update; 2: layer,
// adjoint update.  With the layer's per-cell factors a = (1-q)/(1+q), b = 1/(1+q), q = sigma dt/2:
//   forward  D' = a D + b inc (first step: D' = (a-1) P + b inc),  P' = P + D'
//   adjoint  G' = G + inc,  Q' = a Q + b G', i.e. Z' = a Z + b kappa G'  (final step: x = G' + ((a-1)/b) Q)
// Tiles that do not reach the layer use a = b = 1 without loading the factors.
// FULL (rows of no multiple of 4 cells): the forward's stencil takes the difference form and the adjoint keeps G as a
// compensated pair too (G_lo in dbuf_lo), with the rounding of kappa G carried into Z_lo.
// GRAD (adjoint): adds this step's term gcoef Z^m .* L P^{m-1} of the medium gradient to a compensated sum.
// The sums are pairs of FP32 (TwoSum with the product's rounding error, ~2^-47): FP64 arithmetic runs at 2
// operations per clock and SM here, and dividing by kappa once at the end replaces a division per step.
template <int R, int MODE, int SP, bool FULL, bool GRAD = false, bool TALL = false>
__global__ void __launch_bounds__(threads_of(TALL), min_ctas(R, FULL, GRAD, TALL)) step2d_tma_kernel(const StepArgs a, const __grid_constant__ CUtensorMap mp,
                                                             const __grid_constant__ CUtensorMap ml, int* status,
                                                             long long timeout_ns) {
  constexpr bool VARC = MODE == 1, ADJ = MODE == 2;
  constexpr int TY = tile_y(TALL), THREADS = threads_of(TALL);
  constexpr bool ALL_K = VARC && R > 1 && !FULL;
  using G = G2<R, ADJ ? 2 : 1, TALL>;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  float* stage0 = reinterpret_cast<float*>(smem_raw);
  uint64_t* bars = reinterpret_cast<uint64_t*>(stage0 + 2 * G::STAGE);

  const int t = threadIdx.x;

  const int nx = a.nx, ny = a.ny, pitch = a.pitch;
  const int tiles_x = (nx + TX - 1) / TX;
  const int ntiles = tiles_x * ((ny + TY - 1) / TY);
  const int c0 = (t % TCOLS) * 2 * NP, r0 = (t / TCOLS) * RUN;
  const bool load_d = !a.d_zero;
  const bool kv = a.kappa != nullptr;  // adjoint: varying medium (per-cell kappa)
  const unsigned stage_bytes = (unsigned)G::STAGE * 4u;

  if (t == 0) {
    mbar_init(&bars[0], 1);
    mbar_init(&bars[1], 1);
    fence_mbar_init();
  }
  __syncthreads();

  auto issue = [&](int tile, int s) {
    float* st = stage0 + s * G::STAGE;
    const int tt = a.flip ? ntiles - 1 - tile : tile;
    const int gx0 = (tt % tiles_x) * TX, gy0 = (tt / tiles_x) * TY;
    mbar_expect_tx(&bars[s], stage_bytes);
    tma_load_2d(st, &mp, gx0 - XH, gy0 - R, &bars[s]);
    if (ADJ) tma_load_2d(st + G::PBOX, &ml, gx0 - XH, gy0 - R, &bars[s]);
  };
  griddep_wait();  // everything above overlaps the previous step's last CTAs
  griddep_trigger();
  int first = blockIdx.x;
  if (t == 0 && first < ntiles) issue(first, 0);
  fused_sample2(a, blockIdx.x, t);  // while the first tile's boxes are in flight

  const float ckh = a.c_lap * a.kappa0, ckl = a.c_lap * a.kappa0_lo;
  float2 w2[R + 1];  // stencil weights, packed
#pragma unroll
  for (int m = 0; m <= R; ++m) w2[m] = dup2(a.w[m]);
  float wc = 0.f;  // centre weight of the Z_lo stencil (sum form)
#pragma unroll
  for (int m = 1; m <= R; ++m) wc += a.w[m];
  const float2 nwc = dup2(-(wc * 4.f));
  int k = 0;
  bool ok = true;
  int issued = (first < ntiles) ? 1 : 0;
  for (int tile = first; tile < ntiles; tile += gridDim.x, ++k) {
    const int s = k & 1;
    if (t == 0) {
      fence_proxy_async_shared();  // the other stage was last read through the generic proxy
      const int nxt = tile + gridDim.x;
      if (nxt < ntiles) {
        issue(nxt, s ^ 1);
        ++issued;
      }
    }
    const int tt = a.flip ? ntiles - 1 - tile : tile;
    const int gx0 = (tt % tiles_x) * TX, gy0 = (tt / tiles_x) * TY;
    const int gx = gx0 + c0;
    // own-cell fields straight into registers, in flight while the boxes land: D or G of every row; kappa
    // and G_lo (fetch) two rows ahead of their use, or, in the forward of a varying medium from order 4 on, kappa of
    // every row as well (K us per step, all rows | two ahead: 12000^2 order 8 524 | 556, order 6 with a layer 540 |
    // 609, 4096^2 order 8 57 | 62; order 2 530 | 494)
    Cells<NP> d2[RUN], kh2[RUN], kl2[RUN], gl2[RUN], lp2[RUN], sh2[RUN], sl2[RUN];
    // (the adjoint's final step takes kappa inside the layer; a partial tile has cells beyond the field, so every
    // access to a field by cell is under a test like fetch's)
    const bool need_k = VARC || (ADJ && kv && (SP || !a.final_step));
    auto fetch = [&](int rr) {
      const int gy = gy0 + r0 + rr;
      const long long gi = (long long)gy * pitch + gx;
      const bool in = gy < ny && gx < nx;
      kh2[rr].fill(0.f);
      kl2[rr].fill(0.f);
      gl2[rr].fill(0.f);
      if (need_k && in) kh2[rr].ldg(a.kappa + gi);
      if ((VARC || FULL) && need_k && in) kl2[rr].ldg(a.kappa_lo + gi);
      if (ADJ && FULL && in) gl2[rr].stream(a.dbuf_lo + gi);
      if (GRAD && in) {
        lp2[rr].stream(a.lp + gi);
        sh2[rr].stream(a.gsum_hi + gi);
        sl2[rr].stream(a.gsum_lo + gi);
      }
    };
#pragma unroll
    for (int rr = 0; rr < RUN; ++rr) {
      const int gy = gy0 + r0 + rr;
      d2[rr].fill(0.f);
      if (load_d && gy < ny && gx < nx) d2[rr].stream(a.dbuf + (long long)gy * pitch + gx);
    }
#pragma unroll
    for (int rr = 0; rr < (ALL_K ? RUN : 2); ++rr) fetch(rr);
    const bool good = mbar_wait(&bars[s], (k >> 1) & 1, timeout_ns);
    if (__syncthreads_or(!good)) {
      if (t == 0) atomicCAS(status, (int)PAT_OK, (int)PAT_ERR_TIMEOUT);
      ok = false;
      break;
    }
    const float* P = stage0 + s * G::STAGE;  // P (forward) or Z (adjoint)
    const float* PL = P + G::PBOX;           // adjoint: Z_lo
    // absorbing layer: does the tile reach it (its factors are then loaded row by row)
    const bool layer = SP != 0 && (gx0 < a.sp_w || gx0 + TX > nx - a.sp_w || gy0 < a.sp_w || gy0 + TY > ny - a.sp_w);

    // the tile's update; instantiated separately for tiles inside and outside the layer, so that
    // tiles outside it run exactly the code of the kernel without a layer
    auto update = [&](auto in_layer) {
      constexpr bool LAYER = decltype(in_layer)::value;
      Cells<NP> lo[RUN];  // adjoint: the Z_lo part of the stencil, first pass
      if (ADJ) stencil_run_pair<R, RUN, BW>(PL + (r0 + R) * BW + XH + c0, w2, nwc, lo);
      // sliding window over this thread's columns: win[i] = box row (row - R + i)
      const float* own = P + (r0 + R) * BW + XH + c0;
      Cells<NP> win[2 * R + 1];
#pragma unroll
      for (int i = 0; i < 2 * R; ++i) win[i].load(own + (i - R) * BW);
#pragma unroll
      for (int rr = 0; rr < RUN; ++rr) {
        win[2 * R].load(own + (rr + R) * BW);
        Row<R, NP> f;
        f.load(own + rr * BW, win[R]);
        const int gy = gy0 + r0 + rr;
        const long long gi = (long long)gy * pitch + gx;
        const bool in = gy < ny && gx < nx;
        if (!ALL_K && rr + 2 < RUN) fetch(rr + 2);
        Cells<NP> sa2, sb2, zl2;
        sa2.fill(1.f);
        sb2.fill(1.f);
        if (LAYER && in) {
          sa2.ldg(a.sp_a + gi);
          sb2.ldg(a.sp_b + gi);
        }
        if (ADJ) zl2.load(PL + (r0 + rr + R) * BW + XH + c0);  // own Z_lo cells
        // forward: zero-sum pair form (a + b) - 2c per tap; adjoint (and FULL): difference form
        Cells<NP> st2;
#pragma unroll
        for (int p = 0; p < NP; ++p) st2.v[p] = stencil_pair<R, ADJ || FULL>(win, f, p, w2);
        float dn[2 * NP], pn[2 * NP], pl[2 * NP], gn[2 * NP];
#pragma unroll
        for (int j = 0; j < 2 * NP; ++j) {
          const float c = win[R].get(j);  // own P or Z
          const float fa = sa2.get(j), fb = sb2.get(j);
          if (!ADJ) {
            const float acc = st2.get(j);
            const float inc = VARC ? fmaf(a.c_lap * kh2[rr].get(j), acc, (a.c_lap * kl2[rr].get(j)) * acc)
                                   : fmaf(ckh, acc, ckl * acc);
            if (!LAYER)
              dn[j] = d2[rr].get(j) + inc;
            else  // forward in the layer
              dn[j] = load_d ? fmaf(fa, d2[rr].get(j), fb * inc) : fmaf(fa - 1.f, c, fb * inc);
            pn[j] = c + dn[j];
            pl[j] = gn[j] = 0.f;
          } else {
            const float acc = st2.get(j) + lo[rr].get(j);
            const float zl = zl2.get(j);
            const float kap = kv ? kh2[rr].get(j) : a.kappa0;
            float g, gl = 0.f;  // G' = G + L Z (S^T r injected into G beforehand)
            if (FULL && !a.final_step)
              g = two_sum(d2[rr].get(j), a.c_lap * acc + gl2[rr].get(j), gl);
            else
              g = fmaf(a.c_lap, acc, FULL ? d2[rr].get(j) + gl2[rr].get(j) : d2[rr].get(j));
            dn[j] = g;
            gn[j] = gl;
            if (a.final_step) {
              pn[j] = g;
              if (LAYER && in && fa != 1.f)  // x = G' + ((a-1)/b) Q,  Q = (Z + Z_lo) / kappa
                pn[j] = fmaf((fa - 1.f) / fb, (c + zl) / kap, g);
              pl[j] = 0.f;
            } else {
              float u, ul = 0.f;  // kappa G', and what its rounding dropped (FULL)
              if (FULL) {
                const float kl = kv ? kl2[rr].get(j) : a.kappa0_lo;
                u = kap * g;
                ul = fmaf(kap, g, -u) + fmaf(kap, gl, kl * g);
              } else {
                u = kv ? kap * g : fmaf(a.kappa0, g, a.kappa0_lo * g);
              }
              if (LAYER && (fa != 1.f || fb != 1.f)) {  // Z' = a Z + b kappa G'
                pn[j] = fmaf(fa, c, fb * u);
                pl[j] = FULL ? fmaf(fa, zl, fb * ul) : fa * zl;
              } else {
                float e;
                pn[j] = two_sum(c, u, e);
                pl[j] = zl + (FULL ? e + ul : e);
              }
            }
          }
        }
        if (in) {
          store_cells<NP>(a.next + gi, pn);
          if (!ADJ && FULL && a.lp != nullptr) st2.store(a.lp + gi);
          if (!a.final_step) {
            store_cells<NP>(a.dbuf + gi, dn);
            if (ADJ) store_cells<NP>(a.next_lo + gi, pl);
            if (ADJ && FULL) store_cells<NP>(a.dbuf_lo + gi, gn);
            if (GRAD) {
              float sh[2 * NP], sl[2 * NP];
#pragma unroll
              for (int j = 0; j < 2 * NP; ++j) {
                const float l = a.gcoef * lp2[rr].get(j);
                const float ph = pn[j] * l;
                const float pe = fmaf(pl[j], l, fmaf(pn[j], l, -ph));
                float e;
                sh[j] = two_sum(sh2[rr].get(j), ph, e);
                sl[j] = sl2[rr].get(j) + (e + pe);
              }
              store_cells<NP>(a.gsum_hi + gi, sh);
              store_cells<NP>(a.gsum_lo + gi, sl);
            }
          }
        }
#pragma unroll
        for (int i = 0; i < 2 * R; ++i) win[i] = win[i + 1];
      }
    };
    if (SP != 0 && layer)
      update(std::true_type{});
    else
      update(std::false_type{});
    __syncthreads();  // this stage is refilled by the next iteration's TMA
    if (ADJ && a.inj_r) {  // G + S^T r for the next step, on this tile's cells (stored above, before the barrier)
      const int e1 = a.inj_tile_ptr[tt + 1];
      for (int e = a.inj_tile_ptr[tt] + t; e < e1; e += THREADS) {
        const InjCell c = a.inj_tile[e];
        float v = 0.f;
        for (int q = c.beg; q < c.end; ++q) v = fmaf(a.ent_w[q], a.inj_r[(long long)a.ent_sensor[q] * a.nt + a.inj_t], v);
        a.dbuf[c.local] += v;
      }
    }
  }
  // after a timed-out wait: give the copies in flight a bounded chance to land
  if (t == 0 && !ok)
    for (int j = max(0, issued - 2); j < issued; ++j) mbar_wait(&bars[j & 1], (j >> 1) & 1, timeout_ns);
}

template <int R, bool FULL>
const void* kernel_r(int mode, int sp) {
  switch (mode * 3 + sp) {
    case 0: return reinterpret_cast<const void*>(&step2d_tma_kernel<R, 0, 0, FULL>);
    case 1: return reinterpret_cast<const void*>(&step2d_tma_kernel<R, 0, 1, FULL>);
    case 3: return reinterpret_cast<const void*>(&step2d_tma_kernel<R, 1, 0, FULL>);
    case 4: return reinterpret_cast<const void*>(&step2d_tma_kernel<R, 1, 1, FULL>);
    case 6: return reinterpret_cast<const void*>(&step2d_tma_kernel<R, 2, 0, FULL>);
    case 8: return reinterpret_cast<const void*>(&step2d_tma_kernel<R, 2, 2, FULL>);
    case 9: return reinterpret_cast<const void*>(&step2d_tma_kernel<R, 2, 0, FULL, true>);
    default: return nullptr;  // mismatched layer modes are not instantiated
  }
}

template <int R>
const void* kernel_tall(int mode, int sp) {  // forward, constant medium
  if (mode != 0) return nullptr;
  return sp == 0   ? reinterpret_cast<const void*>(&step2d_tma_kernel<R, 0, 0, false, false, true>)
         : sp == 1 ? reinterpret_cast<const void*>(&step2d_tma_kernel<R, 0, 1, false, false, true>)
                   : nullptr;
}

template <int R>
const void* kernel_form(int mode, int sp, Form2d form) {
  return form == Form2d::Tall ? kernel_tall<R>(mode, sp)
         : form == Form2d::Full ? kernel_r<R, true>(mode, sp)
                                : kernel_r<R, false>(mode, sp);
}

const void* kernel_for(int R, int mode, int sp, Form2d form) {
  switch (R) {
    case 1: return kernel_form<1>(mode, sp, form);
    case 3: return kernel_form<3>(mode, sp, form);
    case 5: return kernel_form<5>(mode, sp, form);
    case 7: return kernel_form<7>(mode, sp, form);
    default: return nullptr;
  }
}

template <int R>
size_t smem_r(int mode, Form2d form) {
  return mode >= 2 ? G2<R, 2>::SMEM : form == Form2d::Tall ? G2<R, 1, true>::SMEM : G2<R>::SMEM;
}

size_t smem_for(int R, int mode, Form2d form) {
  return R == 1 ? smem_r<1>(mode, form) : R == 3 ? smem_r<3>(mode, form) : R == 5 ? smem_r<5>(mode, form) : smem_r<7>(mode, form);
}

}  // namespace

void tma2d_tile(int* tx, int* ty) {
  *tx = TX;
  *ty = tile_y(false);
}

bool tma2d_tall(int pitch, long long cells) { return pitch % 32 == 0 && cells >= 1LL << 26; }

bool tma2d_supported(int R) { return R == 1 || R == 3 || R == 5 || R == 7; }

cudaError_t tma2d_encode(const float* base, int nx, int pitch, int ny, int R, bool tall, CUtensorMap* halo) {
  auto fn = tma_encoder();
  if (!fn) return cudaErrorNotSupported;
  const cuuint64_t dims[2] = {(cuuint64_t)nx, (cuuint64_t)ny};
  const cuuint64_t strides[1] = {(cuuint64_t)pitch * 4};
  const cuuint32_t estr[2] = {1, 1};
  const cuuint32_t box_h[2] = {(cuuint32_t)BW, (cuuint32_t)(tile_y(tall) + 2 * R)};
  const CUresult r = fn(halo, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(base), dims, strides, box_h, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// Persistent grid: as many CTAs as fit on the device, at most one per tile (0: the kernel does not run there).
int tma2d_ctas(int nx, int ny, int R, int mode, int sp, Form2d form) {
  static PerDevice resident[3][4][3][8];
  const bool tall = form == Form2d::Tall;
  const int fit = resident[(int)form][mode][sp][R].get(current_device(), [&] {
    int dev = 0, sms = 0, per = 0;
    const void* fn = kernel_for(R, mode, sp, form);
    const size_t smem = smem_for(R, mode, form);
    if (!fn || cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, threads_of(tall), smem) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    return per * sms;
  });
  const int ntiles = ((nx + TX - 1) / TX) * ((ny + tile_y(tall) - 1) / tile_y(tall));
  return ntiles < fit ? ntiles : fit;
}

long long tma2d_threads(int nx, int ny, int R, int mode, int sp, Form2d form) {
  return (long long)tma2d_ctas(nx, ny, R, mode, sp, form) * threads_of(form == Form2d::Tall);
}

cudaError_t step2d_tma_launch(int R, int mode, int sp, Form2d form, const StepArgs& a, const CUtensorMap& p,
                              const CUtensorMap& lo, int* status, long long timeout_ns, cudaStream_t st) {
  const void* fn = kernel_for(R, mode, sp, form);
  if (!fn) return cudaErrorInvalidValue;
  const int nctas = tma2d_ctas(a.nx, a.ny, R, mode, sp, form);  // the first call sets the kernel's attributes
  if (nctas <= 0) return cudaErrorInvalidConfiguration;
  CUtensorMap map = p, mapl = lo;
  StepArgs args = a;
  void* params[] = {&args, &map, &mapl, &status, &timeout_ns};
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(nctas);
  cfg.blockDim = dim3(threads_of(form == Form2d::Tall));
  cfg.dynamicSmemBytes = smem_for(R, mode, form);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];  // starts while the previous step drains (the kernel waits for it itself)
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelExC(&cfg, fn, params);
}

}  // namespace pat
