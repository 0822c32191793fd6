// Persistent 2D wave kernel for grids of up to one 128 x 64 tile per SM (1.2
// million cells on 152 SMs): K or K* (paper Sec. 2, Eq. wave_equation,
// eliminated to p only) in one cooperative launch, the wavefield on chip.  The
// recurrences, the state variables and the exchange protocol (tagged 64-bit
// words, two slots, bounded waits) are those of the kernel with 64 x 32 tiles
// (wave2d_persist.cu), which serves the grids whose tiles fit; what differs is
// the tile and where its state lives.
//
// A step's 8192 cells per SM are bound by FP32 and shared-memory issue rather
// than by the exchange, so a thread owns two blocks of 2 columns x 4 rows and
// slides a register window down each.  The 352 blocks of the tile's 8-cell
// frame belong to as many threads (11 warps), whose second block is an interior
// one; the other 160 threads own two interior blocks.  Interior stencils
// (R <= 7) need no halo: first every interior block is computed, then the
// frame's threads take the neighbours' words, which have arrived meanwhile, and
// compute the frame while the others serve the sensors.  P, Z and Z_lo are read
// from shared memory (two slots of the whole tile); D or G stays in registers.
// The adjoint keeps G as a compensated pair as well, as the per-step engine
// does on rows of no multiple of 4 cells; the sensor injections S^T r are added to its low
// part G_lo, which sits in shared memory and joins the next increment anyway:
// to the frame's cells before the mid-step barrier (the frame reads them after
// it), to the interior's after it.
//
// us per step, K / K*, at 1024^2 (128 of 152 SMs): order 2 1.7 / 3.3, order 4
// 2.5 / 4.5, order 6 3.3 / 6.1, order 8 4.2 / 7.6; a launch per step takes
// 3.5 / 5.7, 4.3 / 6.3, 4.1 / 8.1, 4.5 / 8.5.  One 2 x 8 block per thread, with
// frame threads that compute no interior: 4.9 / 10.8 at order 8 (two halves
// bound by latency, on 10 and 6 warps).
#include <type_traits>

#include "internal.h"
#include "persist2d.cuh"
#include "stencil.cuh"
#include "tile2d.cuh"

namespace pat {
namespace {

constexpr int TX = 128, TY = 64, RUN = 4;
constexpr int NTHREADS = (TX / 2) * (TY / RUN) / 2;  // 512: two blocks each
constexpr int XOFF = 8;                              // left halo columns in shared memory (>= R + 1)
constexpr int PITCH = TX + 2 * XOFF;
constexpr int GX = TX / 2, GY = TY / RUN;            // blocks across and down the tile
constexpr int EDGE = 8, EX = EDGE / 2, EY = EDGE / RUN;  // frame depth: cells, block columns, block rows
constexpr int NFRAME = 2 * EY * GX + (GY - 2 * EY) * 2 * EX;  // 352 blocks, one per thread t < NFRAME
constexpr int NREST = NTHREADS - NFRAME;
constexpr int MANY = (1 << 19) - 1;                  // sensors of one cell that fit its kept word
constexpr int KEEP = 8;                              // words of shared memory per thread
static_assert(EDGE >= kMaxR && NFRAME % 32 == 0, "interior stencils need no halo; whole warps");

// Thread (= frame block) at block row ty, block column tx (the inverse of block_cell).
__device__ __forceinline__ int frame_thread(int ty, int tx) {
  if (ty < EY) return ty * GX + tx;
  if (ty >= GY - EY) return (ty - (GY - 2 * EY)) * GX + tx;
  return 2 * EY * GX + (ty - EY) * 2 * EX + (tx < EX ? tx : tx - (GX - 2 * EX));
}

// First cell (row, column) of block v of thread t: frame blocks (v = 0, t < NFRAME) are numbered along the top
// rows, the bottom rows, then the sides; interior blocks row by row.
__device__ __forceinline__ void block_cell(int t, int v, int& row, int& col) {
  int ty, tx;
  if (v == 0 && t < 2 * EY * GX) {
    ty = t < EY * GX ? t / GX : t / GX + GY - 2 * EY;
    tx = t % GX;
  } else if (v == 0 && t < NFRAME) {
    const int u = t - 2 * EY * GX, c = u % (2 * EX);
    ty = EY + u / (2 * EX);
    tx = c < EX ? c : c + GX - 2 * EX;
  } else {
    const int u = v == 0 ? t - NFRAME : t + NREST;
    ty = EY + u / (GX - 2 * EX);
    tx = EX + u % (GX - 2 * EX);
  }
  row = ty * RUN;
  col = tx * 2;
}

template <int R, bool ADJ>
struct Geo {
  static constexpr int NF = ADJ ? 2 : 1;
  static constexpr int SBUF = (TY + 2 * R) * PITCH;  // one shared-memory field buffer
  // exchange: a frame thread publishes its rows as pairs of words; pair (row rr, thread f) is pair rr NFRAME + f of
  // the slot, so that a warp's store is one contiguous run
  static constexpr int SLOT = 2 * RUN * NFRAME;      // words per tile and slot
  static constexpr int D = (R + 1) / 2;              // column pairs a west or east neighbour needs
  static constexpr int NS = R * GX, WE = TY * D;     // pairs from one north or south / west or east neighbour
  static constexpr int PER = (2 * NS + 2 * WE + NFRAME - 1) / NFRAME;  // pairs a frame thread takes at most
  static_assert(PER + 4 <= KEEP && 2 * D <= XOFF && SLOT / 2 <= 4096 && SBUF <= (1 << 14), "fields of a duty word");
};

// Pair u of a tile's halo: [13:0] float offset in the own buffer, [25:14] pair of the neighbour's slot, [27:26]
// region (north, south, west, east).
template <int R, bool ADJ>
__device__ __forceinline__ unsigned halo_pair(int u) {
  using G = Geo<R, ADJ>;
  int region, src, dst;
  if (u < 2 * G::NS) {
    region = u < G::NS ? 0 : 1;
    const int v = u % G::NS, i = v / GX, p = v % GX;
    const int row = region == 0 ? TY - R + i : i;
    src = (row % RUN) * NFRAME + frame_thread(row / RUN, p);
    dst = (region == 0 ? i : R + TY + i) * PITCH + XOFF + 2 * p;
  } else {
    const int w = u - 2 * G::NS;
    region = w < G::WE ? 2 : 3;
    const int v = w % G::WE, row = v / G::D, g = v % G::D;
    src = (row % RUN) * NFRAME + frame_thread(row / RUN, region == 2 ? GX - G::D + g : g);
    dst = (R + row) * PITCH + (region == 2 ? XOFF - 2 * G::D : XOFF + TX) + 2 * g;
  }
  return (unsigned)region << 26 | (unsigned)src << 14 | (unsigned)dst;
}

template <int R, bool ADJ, bool VARC, bool SP>
__global__ void __launch_bounds__(NTHREADS, 1) wave2d_persist_large_kernel(const Persist2DArgs a) {
  using G = Geo<R, ADJ>;
  extern __shared__ float4 smem4[];
  float* S0 = reinterpret_cast<float*>(smem4);  // [slot][field]
  float* J = S0 + 2 * G::NF * G::SBUF;          // adjoint: G_lo + S^T r of the step's cells, TY x TX
  // words that a thread needs once per step, out of the registers of the update: [0, 4) the first cell of its
  // injection list, [4, 4 + PER) a frame thread's halo duty
  unsigned* keep = reinterpret_cast<unsigned*>(J + (ADJ ? TX * TY : 0)) + threadIdx.x;  // stride NTHREADS
  // forward, varying medium: the tile's kappa and its rounding residual (the adjoint has no room for them and reads
  // 64 KB per tile and step from L2, 1.0 us of its step at orders 2 to 6; from L2 the forward took 0.4 us more)
  constexpr bool KSM = VARC && !ADJ;
  float* ks = J + (ADJ ? TX * TY : 0) + KEEP * NTHREADS;
  __shared__ int s_abort;

  const int t = threadIdx.x;
  const bool frame = t < NFRAME;
  const int tile = blockIdx.x;
  const int tix = tile % a.tiles_x, tiy = tile / a.tiles_x;
  const int gx0 = tix * TX, gy0 = tiy * TY;
  const int nx = a.nx, ny = a.ny, nt = a.nt;
  struct Block {
    int r0, c0, gx, rows;  // first cell in the tile, column in the grid, rows inside the grid
    bool in0, in1;
    long long gi0;         // first cell in kappa and the layer's factors (padded rows)
  };
  auto block = [&](int v) {
    Block b;
    block_cell(t, v, b.r0, b.c0);
    b.gx = gx0 + b.c0;
    b.in0 = b.gx < nx;
    b.in1 = b.gx + 1 < nx;
    b.rows = min(max(ny - gy0 - b.r0, 0), RUN);
    b.gi0 = (long long)(gy0 + b.r0) * a.pitch + b.gx;
    return b;
  };
  u64* xbuf = reinterpret_cast<u64*>(a.xbuf);
  const float2(&w2)[R + 1] = reinterpret_cast<const float2(&)[R + 1]>(a.w2);
  float wc = 0.f;  // centre weight of the Z_lo stencil (sum form)
#pragma unroll
  for (int m = 1; m <= R; ++m) wc += a.w[m];
  const float2 nwc = dup2(-(wc * 4.f));
  const bool layer = SP && (gx0 < a.sp_w || gx0 + TX > nx - a.sp_w || gy0 < a.sp_w || gy0 + TY > ny - a.sp_w);

  for (int i = t; i < 2 * G::NF * G::SBUF + (ADJ ? TX * TY : 0); i += NTHREADS) S0[i] = 0.f;
  if (t == 0) s_abort = 0;
  __syncthreads();

  auto Sbuf = [&](int slot) { return S0 + slot * G::NF * G::SBUF; };
  auto Xslot = [&](int tl, int slot) { return xbuf + ((size_t)tl * 2 + slot) * G::SLOT; };
  Cells<1> d[2][RUN];  // D (forward); G (adjoint)
  // frame blocks: rows that a neighbour needs
  auto publish = [&](const Block& b, u64* X, int rr, float2 hi, float2 lo, unsigned step) {
    if (b.c0 < R || b.c0 + 2 > TX - R || b.r0 + rr < R || b.r0 + rr >= TY - R)
      st_word2(X + 2 * (rr * NFRAME + t), pack<ADJ>(hi.x, lo.x, step), pack<ADJ>(hi.y, lo.y, step));
  };
#pragma unroll
  for (int v = 0; v < 2; ++v) {  // state 0: x (forward), zero (adjoint)
    const Block b = block(v);
#pragma unroll
    for (int rr = 0; rr < RUN; ++rr) {
      d[v][rr].fill(0.f);
      if (KSM) {
        float2 h = make_float2(0.f, 0.f), l = h;
        if (rr < b.rows && b.in0) {
          h = __ldg(reinterpret_cast<const float2*>(a.kappa + b.gi0 + (long long)rr * a.pitch));
          l = __ldg(reinterpret_cast<const float2*>(a.kappa_lo + b.gi0 + (long long)rr * a.pitch));
        }
        *reinterpret_cast<float2*>(ks + (b.r0 + rr) * TX + b.c0) = h;
        *reinterpret_cast<float2*>(ks + TX * TY + (b.r0 + rr) * TX + b.c0) = l;
      }
      float2 p = make_float2(0.f, 0.f);
      if (!ADJ && rr < b.rows) {
        const float* x = a.in + (long long)(gy0 + b.r0 + rr) * nx + b.gx;
        if (b.in0) p.x = x[0];
        if (b.in1) p.y = x[1];
      }
      if (!ADJ) *reinterpret_cast<float2*>(Sbuf(0) + (b.r0 + rr + R) * PITCH + XOFF + b.c0) = p;
      if (v == 0 && frame) publish(b, Xslot(tile, 0), rr, p, make_float2(0.f, 0.f), 0u);
    }
  }

  // ---- halo duty of the frame's threads
  unsigned mine = 0;  // pairs whose neighbour exists
  if (frame)
    for (int j = 0; j < G::PER; ++j) {
      const int u = t + j * NFRAME;
      if (u >= 2 * G::NS + 2 * G::WE) break;
      const unsigned h = halo_pair<R, ADJ>(u);
      const int region = h >> 26;
      keep[(4 + j) * NTHREADS] = h;
      if (region == 0 ? tiy > 0 : region == 1 ? tiy < a.tiles_y - 1 : region == 2 ? tix > 0 : tix < a.tiles_x - 1)
        mine |= 1u << j;
    }
  // halo of state k; false if the wait ran out.  Every poll issues the loads of all pending pairs before it
  // checks a tag.
  auto load_halo = [&](int k) -> bool {
    float* S = Sbuf(k & 1);
    unsigned pending = mine;
    unsigned long long t0 = 0;
    for (unsigned it = 0; pending && it < (1u << 28); ++it) {
      u64 w[G::PER][2];
#pragma unroll
      for (int j = 0; j < G::PER; ++j)
        if (pending & (1u << j)) {
          const unsigned h = keep[(4 + j) * NTHREADS];
          const int region = h >> 26;
          const int nb = tile + (region == 0 ? -a.tiles_x : region == 1 ? a.tiles_x : region == 2 ? -1 : 1);
          ld_word2(Xslot(nb, k & 1) + 2 * (h >> 14 & 0xfffu), w[j][0], w[j][1]);
        }
#pragma unroll
      for (int j = 0; j < G::PER; ++j)
        if ((pending & (1u << j)) && tag_ok<ADJ>(w[j][0], (unsigned)k) && tag_ok<ADJ>(w[j][1], (unsigned)k)) {
          float* q = S + (keep[(4 + j) * NTHREADS] & 0x3fffu);
          *reinterpret_cast<float2*>(q) = make_float2(word_hi(w[j][0]), word_hi(w[j][1]));
          if (ADJ) *reinterpret_cast<float2*>(q + G::SBUF) = make_float2(word_lo(w[j][0]), word_lo(w[j][1]));
          pending &= ~(1u << j);
        }
      if (!pending) return true;
      if (it == 0) t0 = global_timer_ns();
      if (a.poll_ns > 0) __nanosleep(a.poll_ns);
      if ((it & 31u) == 31u) {
        if (ld_relaxed_gpu(a.abort) != 0) return false;
        if ((long long)(global_timer_ns() - t0) > a.timeout_ns) return false;
      }
    }
    return pending == 0;
  };

  // ---- sensors.  Adjoint: the frame's threads inject into the frame's cells, the others into the interior's
  // (lists [tile][frame, interior]); forward: the others sample.
  const int lt = frame ? t : t - NFRAME, ln = frame ? NFRAME : NREST;
  int e0 = 0, e1 = 0;
  if (ADJ || !frame) {
    const int* ptr = ADJ ? a.tile_inj_ptr + 2 * tile + (frame ? 0 : 1) : a.tile_samp_ptr + tile;
    e0 = ptr[0] + lt;
    e1 = ptr[1];
    if (ADJ && e0 < e1) {
      const InjCell ic = a.inj[e0];
      const bool any = ic.beg < ic.end;
      keep[0] = (unsigned)ic.local | (unsigned)min(ic.end - ic.beg, MANY) << 13;  // TX TY = 2^13 cells
      keep[NTHREADS] = (unsigned)ic.beg;
      keep[2 * NTHREADS] = any ? (unsigned)a.ent_sensor[ic.beg] : 0u;
      keep[3 * NTHREADS] = __float_as_uint(any ? a.ent_w[ic.beg] : 0.f);
    }
  }
  // first value r_n of the thread's list, n = nt-1-k (in flight during an update), and S^T r_n to its cells
  auto fetch_r = [&](int k) { return e0 < e1 ? a.in[(long long)(int)keep[2 * NTHREADS] * nt + (nt - 1 - k)] : 0.f; };
  auto inject = [&](int k, float r) {
    if (e0 >= e1) return;
    const int n = nt - 1 - k, beg = (int)keep[NTHREADS];
    int cnt = (int)(keep[0] >> 13);
    if (cnt == MANY) cnt = a.inj[e0].end - beg;
    float s = __uint_as_float(keep[3 * NTHREADS]) * r;
    for (int i = beg + 1; i < beg + cnt; ++i) s = fmaf(a.ent_w[i], a.in[(long long)a.ent_sensor[i] * nt + n], s);
    J[keep[0] & 0x1fff] += s;
    for (int e = e0 + ln; e < e1; e += ln) {
      const InjCell ic = a.inj[e];
      s = 0.f;
      for (int i = ic.beg; i < ic.end; ++i) s = fmaf(a.ent_w[i], a.in[(long long)a.ent_sensor[i] * nt + n], s);
      J[ic.local] += s;
    }
  };
  auto sample = [&](int k) {  // y[:, k] = S P^k
    for (int e = e0; e < e1; e += ln) {
      const SampEntry se = a.samp[e];
      const float* b = Sbuf(k & 1) + (se.ly + R) * PITCH + XOFF + se.lx;
      if (se.part < 0)
        a.out[(long long)se.sensor * nt + k] = se.w[0] * b[0] + se.w[1] * b[1] + se.w[2] * b[PITCH] + se.w[3] * b[PITCH + 1];
      else
        a.part[(long long)se.part * nt + k] = se.w[0] * b[0];
    }
  };

  // ---- state k + 1 of the thread's block v (k = nt - 1: the adjoint's result)
  auto update = [&](auto vc, int k) {
    constexpr int v_ = decltype(vc)::value;
    const Block b = block(v_);
    const int r0 = b.r0, c0 = b.c0, rows = b.rows, gx = b.gx;
    const bool in0 = b.in0, in1 = b.in1;
    const long long gi0 = b.gi0;
    const bool last = k == nt - 1;
    const float* own = Sbuf(k & 1) + (r0 + R) * PITCH + XOFF + c0;
    float* nxt = Sbuf((k + 1) & 1) + (r0 + R) * PITCH + XOFF + c0;
    u64* X = Xslot(tile, (k + 1) & 1);
    const float cf = !ADJ && k == 0 ? 0.5f : 1.f;
    float2 kh[RUN], kl[RUN];
    auto fetch = [&](int rr) {  // two rows ahead of its use
      kh[rr] = VARC ? make_float2(0.f, 0.f) : dup2(a.kappa0);
      kl[rr] = VARC ? make_float2(0.f, 0.f) : dup2(a.kappa0_lo);
      if (KSM) {
        kh[rr] = *reinterpret_cast<const float2*>(ks + (r0 + rr) * TX + c0);
        kl[rr] = *reinterpret_cast<const float2*>(ks + TX * TY + (r0 + rr) * TX + c0);
      } else if (VARC && rr < rows && in0) {
        kh[rr] = __ldg(reinterpret_cast<const float2*>(a.kappa + gi0 + (long long)rr * a.pitch));
        kl[rr] = __ldg(reinterpret_cast<const float2*>(a.kappa_lo + gi0 + (long long)rr * a.pitch));
      }
    };
    fetch(0);
    fetch(1);
    if (ADJ) {  // the Z_lo part of the stencil goes to G_lo's place (in registers it would spill)
      float* gl = J + r0 * TX + c0;
      const float2 lf = dup2(last ? 0.5f : 1.f);
      const float* lw = own + G::SBUF;
      Cells<1> win[2 * R + 1];
#pragma unroll
      for (int i = 0; i < 2 * R; ++i) win[i].load(lw + (i - R) * PITCH);
#pragma unroll
      for (int rr = 0; rr < RUN; ++rr) {
        win[2 * R].load(lw + (rr + R) * PITCH);
        Row<R, 1> f;
        f.load(lw + rr * PITCH, win[R]);
        float2* q = reinterpret_cast<float2*>(gl + rr * TX);
        *q = __ffma2_rn(lf, stencil_low<R, 1>(win, f, 0, w2, nwc), *q);
#pragma unroll
        for (int i = 0; i < 2 * R; ++i) win[i] = win[i + 1];
      }
    }
    Cells<1> win[2 * R + 1];
#pragma unroll
    for (int i = 0; i < 2 * R; ++i) win[i].load(own + (i - R) * PITCH);
#pragma unroll
    for (int rr = 0; rr < RUN; ++rr) {
      win[2 * R].load(own + (rr + R) * PITCH);
      Row<R, 1> f;
      f.load(own + rr * PITCH, win[R]);
      if (rr + 2 < RUN) fetch(rr + 2);
      const float2 L = stencil_pair<R, true, 1>(win, f, 0, w2);
      float2 fa = dup2(1.f), fb = dup2(1.f);
      if (SP && layer && rr < rows && in0) {
        fa = __ldg(reinterpret_cast<const float2*>(a.sp_a + gi0 + (long long)rr * a.pitch));
        fb = __ldg(reinterpret_cast<const float2*>(a.sp_b + gi0 + (long long)rr * a.pitch));
      }
      float2 v, vl = make_float2(0.f, 0.f), jv = vl, zl = vl, gl = vl;
      if (ADJ) {
        jv = *reinterpret_cast<const float2*>(J + (r0 + rr) * TX + c0);
        zl = *reinterpret_cast<const float2*>(own + G::SBUF + rr * PITCH);
      }
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const bool in = rr < rows && (j ? in1 : in0);
        const float c = win[R].get(j), ka = f2get(kh[rr], j), kb = f2get(kl[rr], j), a1 = f2get(fa, j),
                    b1 = f2get(fb, j);
        float nd, ng = 0.f, nv, nl = 0.f;
        if (!ADJ) {
          // D += cf (kappa_hi + kappa_lo) L, the product rounded once before it meets D
          const float l = f2get(L, j), inc = fmaf(cf * ka, l, (cf * kb) * l);
          if (SP)
            nd = k == 0 ? fmaf(a1 - 1.f, c, b1 * inc) : fmaf(a1, d[v_][rr].get(j), b1 * inc);
          else
            nd = d[v_][rr].get(j) + inc;
          nv = c + nd;
        } else {
          const float l = f2get(L, j), z0 = f2get(zl, j);
          if (last) {  // x = S^T r_0 + G^1 + 1/2 L Z^1
            float xv = d[v_][rr].get(j) + fmaf(0.5f, l, f2get(jv, j));
            if (SP && a1 != 1.f) xv = fmaf((a1 - 1.f) / b1, (c + z0) / (ka + kb), xv);  // + ((a-1)/b) Q
            if (in) a.out[(long long)(gy0 + r0 + rr) * nx + gx + j] = xv;
            continue;
          }
          nd = two_sum(d[v_][rr].get(j), f2get(jv, j) + l, ng);  // G += S^T r + L Z (compensated)
          const float u = ka * nd;                                           // kappa G, and what its rounding dropped
          const float ul = fmaf(ka, nd, -u) + fmaf(ka, ng, kb * nd);
          if (SP && (a1 != 1.f || b1 != 1.f)) {  // Z = a Z + b kappa G inside the layer
            nv = fmaf(a1, c, b1 * u);
            nl = fmaf(a1, z0, b1 * ul);
          } else {
            float e;
            nv = two_sum(c, u, e);  // Z += kappa G (compensated)
            nl = z0 + (e + ul);
          }
        }
        if (!in) nd = ng = nv = nl = 0.f;
        if (j == 0) {
          d[v_][rr].v[0].x = nd;
          v.x = nv;
          vl.x = nl;
          gl.x = ng;
        } else {
          d[v_][rr].v[0].y = nd;
          v.y = nv;
          vl.y = nl;
          gl.y = ng;
        }
      }
      if (!last) {
        *reinterpret_cast<float2*>(nxt + rr * PITCH) = v;
        if (ADJ) {
          *reinterpret_cast<float2*>(nxt + G::SBUF + rr * PITCH) = vl;
          *reinterpret_cast<float2*>(J + (r0 + rr) * TX + c0) = gl;
        }
        if (v_ == 0 && frame) publish(b, X, rr, v, vl, (unsigned)(k + 1));
      }
#pragma unroll
      for (int i = 0; i < 2 * R; ++i) win[i] = win[i + 1];
    }
  };

  using First = std::integral_constant<int, 0>;
  using Second = std::integral_constant<int, 1>;
  if (ADJ && !frame) inject(0, fetch_r(0));
  __syncthreads();  // state 0 and the interior's first injections
  for (int k = 0; k < nt; ++k) {
    const bool advance = ADJ || k < nt - 1;  // the forward's last state is only sampled
    // half 0: the interior, while the halo of state k arrives; half 1: the frame.  A loop, so that the long
    // update of the first blocks has one copy in the instruction cache.
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
      // the frame's injection of step k, or the interior's of the next
      const bool inj = ADJ && frame == (half == 0) && k + half < nt;
      const float r = inj ? fetch_r(k + half) : 0.f;
      if (half == 0 && advance) update(Second{}, k);
      if (frame == (half == 1) && advance) update(First{}, k);
      if (inj) inject(k + half, r);
      if (!ADJ && half == 1 && !frame) sample(k);
      if (half == 0 && frame && !load_halo(k)) {
        s_abort = 1;
        atomicCAS(a.status, (int)PAT_OK, (int)PAT_ERR_TIMEOUT);
        atomicExch(a.abort, 1);
      }
      __syncthreads();  // half 0: the halo of state k; half 1: state k + 1
      if (half == 0 && s_abort) return;
    }
  }
}

template <int R>
void* pick_r(bool adj, bool varc, bool layer) {
  if (varc) {
    if constexpr (R < 7) {
      if (adj)
        return layer ? (void*)wave2d_persist_large_kernel<R, true, true, true>
                     : (void*)wave2d_persist_large_kernel<R, true, true, false>;
      return layer ? (void*)wave2d_persist_large_kernel<R, false, true, true>
                   : (void*)wave2d_persist_large_kernel<R, false, true, false>;
    }
    return nullptr;
  }
  if (adj)
    return layer ? (void*)wave2d_persist_large_kernel<R, true, false, true>
                 : (void*)wave2d_persist_large_kernel<R, true, false, false>;
  return layer ? (void*)wave2d_persist_large_kernel<R, false, false, true>
               : (void*)wave2d_persist_large_kernel<R, false, false, false>;
}

void* pick(int R, bool adj, bool varc, bool layer) {
  return R == 1   ? pick_r<1>(adj, varc, layer)
         : R == 3 ? pick_r<3>(adj, varc, layer)
         : R == 5 ? pick_r<5>(adj, varc, layer)
         : R == 7 ? pick_r<7>(adj, varc, layer)
                  : nullptr;
}

size_t smem_bytes(int R, bool adj, bool varc) {
  const size_t sbuf = (size_t)(TY + 2 * R) * PITCH, cells = (size_t)TX * TY;
  return (2 * (adj ? 2 : 1) * sbuf + (adj ? cells : varc ? 2 * cells : 0) + (size_t)KEEP * NTHREADS) * sizeof(float);
}

}  // namespace

int persist2dl_tile_x() { return TX; }
int persist2dl_tile_y() { return TY; }
int persist2dl_edge() { return EDGE; }
size_t persist2dl_xbuf_words(int ntiles) { return (size_t)ntiles * 2 * 2 * RUN * NFRAME; }

// One per SM: the launch bounds give every variant, with the layer or without, the registers for that, and the layer
// needs no shared memory, so one variant is asked (asking loads a kernel, 0.3 to 0.5 ms the first time).
int persist2dl_max_ctas(int R, bool adj, bool varc) {
  static PerDevice kept[kMaxR + 1][2][2];
  return kept[R][adj][varc].get(current_device(), [&] {
    void* f = pick(R, adj, varc, false);
    int dev = 0, sms = 0, per_sm = 0;
    const size_t smem = smem_bytes(R, adj, varc);
    if (!f || cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, NTHREADS, smem) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    return per_sm > 0 ? sms : 0;
  });
}

// Where this kernel beats a launch per step, in 64 x 32 tiles per SM (the per-step kernel's time goes up with every
// further round of tiles; this kernel's does not depend on the grid).  us per step K + K*, here | per step:
//   order 2          1.4 + 1.9 to 1.7 + 3.4 | 2.9 + 4.2 to 3.6 + 5.7 (570^2 to 1024^2)       always
//   order 4          2.5 + 4.5 | 3.1 + 5.0 (570^2), 3.1 + 4.6 (720^2), 4.1 + 6.3 (1024^2)    always
//   order 4 varying  2.6 + 5.5 | 3.3 + 4.7 (720^2: 1.8 tiles), 4.0 + 6.5 (800^2: 2.1)        above 2
//   order 6          3.3 + 6.0 | 3.3 + 6.1 (720^2), 3.9 + 6.1 (800^2), 4.1 + 8.1 (1024^2)    above 2
//   order 6 varying  3.5 + 7.1 | 4.0 + 6.6 (900^2: 2.9 tiles), 5.1 + 8.4 (1024^2: 3.4)       above 3
//   order 8          4.3 + 7.6 | 4.4 + 7.1 (900^2), 4.5 + 8.4 (1024^2)                       above 3
// Order 8 with a varying medium (4.7 + 9.5 | 5.4 + 8.6 at 1024^2, kappa read from L2) stays with the per-step kernel.
int persist2dl_min_tiles(int R, bool varc) { return R == 1 ? 0 : R == 3 ? (varc ? 2 : 0) : R == 5 ? (varc ? 3 : 2) : 3; }

cudaError_t persist2dl_launch(int R, bool adj, bool varc, bool layer, const Persist2DArgs& a, int nctas,
                              cudaStream_t st) {
  void* f = pick(R, adj, varc, layer);
  if (!f) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes(R, adj, varc));
  if (e != cudaSuccess) return e;
  void* args[] = {(void*)&a};
  return cudaLaunchCooperativeKernel(f, dim3(nctas), dim3(NTHREADS), args, smem_bytes(R, adj, varc), st);
}

}  // namespace pat
