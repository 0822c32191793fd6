// Persistent 2D wave kernel: one cooperative launch runs a whole time loop
// of K (forward) or K* (adjoint) with the wavefield held on chip.
//
// Method (paper Sec. 2, Eq. wave_equation, p_t(0) = 0, pressure zero outside
// the grid): the staggered leapfrog of order 2M, written without the velocity
// as a second-order recurrence in increment form
//
//   forward:  D^1 = kappa/2 L P^0,  D^{n+1} = D^n + kappa L P^n,  P^{n+1} = P^n + D^{n+1},
//             y[s, n] = S_s P^n  (bilinear sensor sampling), n = 0 .. nt-1;
//   adjoint:  G^{nt} = Q^{nt} = 0;  for n = nt-1 .. 1:
//             G^n = G^{n+1} + S^T r_n + L(kappa Q^{n+1}),  Q^n = Q^{n+1} + G^n;
//             x = S^T r_0 + G^1 + 1/2 L(kappa Q^1),
//
// which is the exact transpose of the forward program.  The increment form
// keeps FP32 rounding from being amplified in the low-frequency modes.
//
// Precision.  kappa is applied as an unevaluated pair kappa_hi + kappa_lo:
// with a constant medium a rounded kappa is the same everywhere and shifts
// the phase of every mode coherently, step after step.  In the adjoint the
// state Q integrates G over time and, in a closed (reflecting) box, grows far
// beyond the result.  The adjoint therefore runs in Z = kappa Q,
//   G^n = G^{n+1} + S^T r_n + L Z^{n+1},  Z^n = Z^{n+1} + kappa G^n,
// with Z kept as a compensated pair Z + Z_lo (TwoSum) that is exchanged and
// fed to the stencil as two FP32 fields (Z through the difference form, whose
// rounding is relative to the differences, Z_lo through the pair form); G is
// plain.
//
// GB300 mapping.  The grid is cut into 64 x 32 tiles, one CTA per tile, all
// co-resident (cooperative launch).  Each of 512 threads keeps its 2 x 2 cells'
// state in registers for the whole loop; the CTA keeps the current field plus
// an R-deep halo in shared memory (double buffered).  Ten warps own the tile's
// 8-cell frame, six its 48 x 16 interior, whose stencils (R <= 7) need no halo
// (K of order 2: six warps a 4-cell frame, ten the rest): while the frame's
// warps wait for the neighbours' strips the interior is computed, and while
// they compute the frame the interior's warps sample the sensors.  (One step of
// 256 threads with 2 x 4 cells each, all of them behind the halo: 2.69 us (K)
// and 3.22 us (K*) at 512^2, order 8, of which 1.3 and 1.6 us are left with the
// 3-point stencil of order 2; now 1.75 and 2.44 us.)  After each step the
// threads that own boundary cells write their blocks straight to an L2-resident
// exchange buffer (relaxed GPU-scope stores; 93.4 against 92.3 reconstruction
// iterations/s at 512^2 when they were staged in shared memory and handed to
// the TMA engine), every value packed with the step it belongs to into one
// 64-bit word; an aligned 64-bit access is single-copy atomic, so a neighbour
// that reads a word with the expected tag has the right value: no flags, no
// fences, one L2 round
// trip per exchange and two CTA barriers per step.  Every wait is bounded by a
// global-timer limit and a shared abort flag; a CTA that gives up records
// PAT_ERR_TIMEOUT, raises the abort flag and leaves the loop, so the launch
// always ends.
#include <algorithm>

#include "internal.h"
#include "persist2d.cuh"
#include "stencil.cuh"
#include "tile2d.cuh"

namespace pat {
namespace {

constexpr int TX = 64;
constexpr int TY = 32;
constexpr int NTHREADS = (TX / 2) * (TY / 2);  // 512: each thread owns 2 rows x 2 columns
constexpr int XOFF = 8;                         // left halo columns in shared memory (>= R, multiple of 4)
constexpr int PITCH = TX + 16;                  // 8 halo columns each side

// The tile's frame: the cells whose stencils reach beyond it.  Its threads, whole warps, wait for the halo.  EDGE is
// even and at least R.  Order 2 has the choice: K with 4 cells (six warps wait, ten work meanwhile: 512^2 1.08 us per
// step, 1.26 with 8 cells, 1.25 with 2), K* with 8, its two stencils taking longer than the halo (640 x 512, two
// CTAs on some SMs: 1.81 us, 1.92 with 4, 1.97 with 2).
template <int R, bool ADJ>
struct Frame {
  static constexpr int EDGE = R == 1 && !ADJ ? 4 : 8;
  static constexpr int RCOUNT = R == 1 ? 32 : 64;  // threads serving one neighbour (warps 0 .. 3 or 0 .. 7)
  static constexpr int BLOCKS = (TX * 2 * EDGE + (TY - 2 * EDGE) * 2 * EDGE) / 4;  // 176 or 320 blocks of 2 x 2
  static constexpr int N = (BLOCKS + 31) / 32 * 32;  // the last warp filled up with interior blocks
  static_assert(EDGE >= R && EDGE % 2 == 0 && N >= 4 * RCOUNT && N < NTHREADS, "interior stencils need no halo");
};

// Thread of the frame that owns row pair rp, column pair cp (the inverse of cells_of).
template <int R, bool ADJ>
__device__ __forceinline__ int frame_thread(int rp, int cp) {
  constexpr int EDGE = Frame<R, ADJ>::EDGE, E2 = EDGE / 2, MIDR = (TY - 2 * EDGE) / 2, MID = (TX - 2 * EDGE) / 2;
  if (rp < E2) return rp * (TX / 2) + cp;
  if (rp >= E2 + MIDR) return (rp - MIDR) * (TX / 2) + cp;
  return EDGE * TX / 2 + (rp - E2) * EDGE + (cp < E2 ? cp : cp - MID);
}

// First cell (row, column) of thread t: the frame's top and bottom rows, then its side columns, then the interior.
template <int R, bool ADJ>
__device__ __forceinline__ void cells_of(int t, int& row, int& col) {
  constexpr int EDGE = Frame<R, ADJ>::EDGE;
  constexpr int BAND = EDGE * TX / 4;           // threads of the top (and of the bottom) rows
  constexpr int SIDE = EDGE;                    // column pairs of the two sides in one row pair
  constexpr int MID = (TX - 2 * EDGE) / 2;      // column pairs of the interior in one row pair
  if (t < 2 * BAND) {
    const int rp = t / (TX / 2);
    row = 2 * (rp < EDGE / 2 ? rp : rp + (TY - 2 * EDGE) / 2);
    col = 2 * (t % (TX / 2));
  } else if (t < Frame<R, ADJ>::BLOCKS) {
    const int u = t - 2 * BAND, cp = u % SIDE;
    row = EDGE + 2 * (u / SIDE);
    col = 2 * (cp < SIDE / 2 ? cp : cp + MID);
  } else {
    const int u = t - Frame<R, ADJ>::BLOCKS;
    row = EDGE + 2 * (u / MID);
    col = EDGE + 2 * (u % MID);
  }
}

template <int R, bool ADJ>
struct Geo {
  static constexpr int NF = ADJ ? 2 : 1;           // shared-memory fields: P, or (W_hi, W_lo)
  static constexpr int ROWS = TY + 2 * R;
  static constexpr int SBUF = ROWS * PITCH;        // one shared-memory field buffer
  // exchange: every frame thread within R cells of the edge (D = (R + 1) / 2 block rows or columns) publishes
  // its 2 x 2 block as four consecutive words.  R = 1, where half of such a block is not needed: the tile's four
  // edges as strips of words, [top TX][bottom TX][left TY][right TY] (with an 8-cell frame, order 2 K us per step:
  // 512^2 1.21 with strips, 1.23 with blocks; 64^2 0.81 and 0.89; 768 x 704, two CTAs per SM, 1.34 and 1.52).
  static constexpr int D = (R + 1) / 2;
  static constexpr int SLOT = R == 1 ? 2 * (TX + TY) : 4 * Frame<R, ADJ>::BLOCKS;  // words per tile, slot and right-hand side
  static constexpr int RCOUNT = Frame<R, ADJ>::RCOUNT;
  static constexpr int PER = (D * TX / 2 + RCOUNT - 1) / RCOUNT;  // blocks a polling thread takes at most
  static_assert(D * TY / 2 <= RCOUNT * PER, "west and east blocks fit as well");
};

// Write the thread's 2 x 2 block of the new state into the shared field
// buffer(s) Sn (second field at Sn + SBUF) and, packed and tagged, to X (its
// block of the tile's exchange slot, for R = 1 the slot itself; nullptr for
// blocks that no neighbour needs).  One 32-byte block per thread in thread order: two coalesced stores
// and no case distinction, and a reader takes whole blocks (strips of exact
// width cost up to eight predicated stores and as many 8-byte loads).
template <int R, bool ADJ>
__device__ __forceinline__ void store_state(float* Sn, u64* X, const float V[2][2], const float Vl[2][2], int r0,
                                            int c0, unsigned step) {
  constexpr int SBUF = Geo<R, ADJ>::SBUF;
  if constexpr (R == 1) {
    if (X) {
      const u64 w[2][2] = {{pack<ADJ>(V[0][0], Vl[0][0], step), pack<ADJ>(V[0][1], Vl[0][1], step)},
                           {pack<ADJ>(V[1][0], Vl[1][0], step), pack<ADJ>(V[1][1], Vl[1][1], step)}};
      if (r0 == 0) st_word2(X + c0, w[0][0], w[0][1]);
      if (r0 == TY - 2) st_word2(X + TX + c0, w[1][0], w[1][1]);
      if (c0 == 0) {
        st_word(X + 2 * TX + r0, w[0][0]);
        st_word(X + 2 * TX + r0 + 1, w[1][0]);
      }
      if (c0 == TX - 2) {
        st_word(X + 2 * TX + TY + r0, w[0][1]);
        st_word(X + 2 * TX + TY + r0 + 1, w[1][1]);
      }
    }
  } else if (X) {
    st_word2(X, pack<ADJ>(V[0][0], Vl[0][0], step), pack<ADJ>(V[0][1], Vl[0][1], step));
    st_word2(X + 2, pack<ADJ>(V[1][0], Vl[1][0], step), pack<ADJ>(V[1][1], Vl[1][1], step));
  }
#pragma unroll
  for (int rr = 0; rr < 2; ++rr) {
    *reinterpret_cast<float2*>(Sn + (r0 + rr + R) * PITCH + XOFF + c0) = make_float2(V[rr][0], V[rr][1]);
    if (ADJ)
      *reinterpret_cast<float2*>(Sn + SBUF + (r0 + rr + R) * PITCH + XOFF + c0) = make_float2(Vl[rr][0], Vl[rr][1]);
  }
}

// Laplacian of the thread's 2 x 2 cells in a shared buffer (y taps, then x taps; pair or difference form), added
// to L (ACC) or written to it.  `own` points at the thread's first cell.
template <int R, bool DIFF, bool ACC>
__device__ __forceinline__ void lap_2x2(const float* __restrict__ own, const float2 (&w2)[R + 1], float2 (&L)[2]) {
  Cells<1> col[2 * R + 2];
#pragma unroll
  for (int i = 0; i < 2 * R + 2; ++i) col[i].load(own + (i - R) * PITCH);
#pragma unroll
  for (int rr = 0; rr < 2; ++rr) {
    Cells<1> win[2 * R + 1];
#pragma unroll
    for (int i = 0; i < 2 * R + 1; ++i) win[i] = col[rr + i];
    Row<R, 1> f;
    f.load(own + rr * PITCH, win[R]);
    L[rr] = stencil_pair<R, DIFF, 1>(win, f, 0, w2, ACC ? L[rr] : dup2(0.f));
  }
}

// The blocks of a neighbour's frame that one polling thread copies: word offset in the neighbour's slot, float
// offset of the block's first cell in the own shared buffer, and which of its two rows lie in the halo.
template <int PER>
struct HaloDuty {
  int src[PER], dst[PER];
  int rows[PER];  // bit 0: first row, bit 1: second; 0: no block
};

template <int R, bool ADJ>
__device__ __forceinline__ HaloDuty<Geo<R, ADJ>::PER> halo_duty(int region, int rrank) {
  using G = Geo<R, ADJ>;
  HaloDuty<G::PER> h;
#pragma unroll
  for (int j = 0; j < G::PER; ++j) {
    const int i = rrank + j * G::RCOUNT;
    h.src[j] = h.dst[j] = h.rows[j] = 0;
    if (R == 1) {  // north and south: a pair of words per thread; west and east: one word
      if (i >= 32) continue;
      h.src[j] = region == 0 ? TX + 2 * i : region == 1 ? 2 * i : region == 2 ? 2 * TX + TY + i : 2 * TX + i;
      h.dst[j] = region == 0   ? XOFF + 2 * i
                 : region == 1 ? (TY + 1) * PITCH + XOFF + 2 * i
                 : region == 2 ? (i + 1) * PITCH + XOFF - 1
                               : (i + 1) * PITCH + XOFF + TX;
      h.rows[j] = region < 2 ? 1 : 2;  // kind
      continue;
    }
    if (region < 2) {  // north: the neighbour's last D row pairs; south: its first D
      if (i >= G::D * TX / 2) continue;
      const int b = i / (TX / 2), cp = i % (TX / 2);
      h.src[j] = 4 * frame_thread<R, ADJ>(region == 0 ? TY / 2 - G::D + b : b, cp);
      h.dst[j] = (region == 0 ? R - 2 * G::D + 2 * b : R + TY + 2 * b) * PITCH + XOFF + 2 * cp;
      // R is odd: the outermost block reaches one row beyond the halo
      h.rows[j] = region == 0 ? (b == 0 ? 2 : 3) : (b == G::D - 1 ? 1 : 3);
    } else {  // west: the neighbour's last D column pairs; east: its first D
      if (i >= G::D * TY / 2) continue;
      const int rp = i / G::D, g = i % G::D;
      h.src[j] = 4 * frame_thread<R, ADJ>(rp, region == 2 ? TX / 2 - G::D + g : g);
      h.dst[j] = (R + 2 * rp) * PITCH + (region == 2 ? XOFF - 2 * G::D : XOFF + TX) + 2 * g;
      h.rows[j] = 3;
    }
  }
  return h;
}

// Copy the halo of state `step` of NR fields from the neighbour's slots X[r]
// into the shared buffers Sc[r] (second field at Sc[r] + SBUF).  Executed by
// the threads of one region; returns false if the wait ran out.  Each
// poll first issues the loads of every block still pending (all fields), then
// checks their tags, so the L2 round trips of one poll overlap instead of
// following one another.
template <int R, bool ADJ, int NR>
__device__ __forceinline__ bool load_halo(float* const (&Sc)[NR], const u64* const (&X)[NR],
                                          const HaloDuty<Geo<R, ADJ>::PER>& h, unsigned step, const int* abort,
                                          long long timeout_ns, int poll_ns) {
  using G = Geo<R, ADJ>;
  static_assert(NR * G::PER <= 32, "pending bits");
  unsigned pending = 0;  // bit r * PER + j
#pragma unroll
  for (int r = 0; r < NR; ++r)
#pragma unroll
    for (int j = 0; j < G::PER; ++j)
      if (h.rows[j]) pending |= 1u << (r * G::PER + j);
  unsigned long long t0 = 0;
  for (unsigned it = 0; it < (1u << 28); ++it) {
    u64 w[NR][G::PER][4];
#pragma unroll
    for (int r = 0; r < NR; ++r)
#pragma unroll
      for (int j = 0; j < G::PER; ++j)
        if (pending & (1u << (r * G::PER + j))) {
          if constexpr (R == 1) {
            if (h.rows[j] == 1)
              ld_word2(X[r] + h.src[j], w[r][j][0], w[r][j][1]);
            else
              w[r][j][0] = w[r][j][1] = ld_word(X[r] + h.src[j]);
          } else {
            ld_word2(X[r] + h.src[j], w[r][j][0], w[r][j][1]);
            ld_word2(X[r] + h.src[j] + 2, w[r][j][2], w[r][j][3]);
          }
        }
#pragma unroll
    for (int r = 0; r < NR; ++r)
#pragma unroll
      for (int j = 0; j < G::PER; ++j) {
        const unsigned bit = 1u << (r * G::PER + j);
        if (!(pending & bit)) continue;
        const u64* q = w[r][j];
        if constexpr (R == 1) {
          if (tag_ok<ADJ>(q[0], step) && tag_ok<ADJ>(q[1], step)) {
            float* d = Sc[r] + h.dst[j];
            if (h.rows[j] == 1) {
              *reinterpret_cast<float2*>(d) = make_float2(word_hi(q[0]), word_hi(q[1]));
              if (ADJ) *reinterpret_cast<float2*>(d + G::SBUF) = make_float2(word_lo(q[0]), word_lo(q[1]));
            } else {
              *d = word_hi(q[0]);
              if (ADJ) d[G::SBUF] = word_lo(q[0]);
            }
            pending &= ~bit;
          }
          continue;
        }
        if (tag_ok<ADJ>(q[0], step) && tag_ok<ADJ>(q[1], step) && tag_ok<ADJ>(q[2], step) && tag_ok<ADJ>(q[3], step)) {
          float* d = Sc[r] + h.dst[j];
#pragma unroll
          for (int rr = 0; rr < 2; ++rr)
            if (h.rows[j] & (1 << rr)) {
              *reinterpret_cast<float2*>(d + rr * PITCH) = make_float2(word_hi(q[2 * rr]), word_hi(q[2 * rr + 1]));
              if (ADJ)
                *reinterpret_cast<float2*>(d + rr * PITCH + G::SBUF) =
                    make_float2(word_lo(q[2 * rr]), word_lo(q[2 * rr + 1]));
            }
          pending &= ~bit;
        }
      }
    if (__all_sync(0xffffffffu, pending == 0)) return true;
    if (it == 0) t0 = global_timer_ns();
    if (poll_ns > 0) __nanosleep(poll_ns);
    if ((it & 31u) == 31u) {
      if (ld_relaxed_gpu(abort) != 0) return false;
      if ((long long)(global_timer_ns() - t0) > timeout_ns) return false;
    }
  }
  return false;
}

// SP: absorbing layer.  With per-cell factors a, b (1 outside the layer):
//   forward  D' = a D + b inc (first step D' = (a-1) P + b inc), P' = P + D'
//   adjoint  G' = G + inc, Q' = a Q + b G', i.e. Z' = a Z + b kappa G' (final x = ... + ((a-1)/b) Q);
//   inside the layer Z_lo is only damped (the fields are being damped there).
// NR right-hand sides advance together (NR = 2: two independent fields of the same plan, e.g. two CG
// solves of one medium): every step exchanges both fields' strips in the same round trip and runs both
// updates between the same barriers.  Inputs / outputs of field r are a.in / a.out (r = 0) and a.in1 /
// a.out1 (r = 1); field r's exchange words follow field 0's in each slot.
// CTAS: CTAs per SM to leave registers for.  Order 2 has a form for two (64 registers), for grids with more tiles
// than SMs; with a layer it spills, so a grid whose tiles have an SM each takes the form for one (order 2 varying,
// K* with a layer, us per step in 64 registers -> here: 64^2 1.90 -> 1.43, 512^2 1.88 -> 1.45).
template <int R, bool ADJ, bool VARC, bool SP, int NR, int CTAS>
__global__ void __launch_bounds__(NTHREADS, CTAS) wave2d_persist_kernel(const Persist2DArgs a) {
  using G = Geo<R, ADJ>;
  constexpr int NFRAME = Frame<R, ADJ>::N;
  static_assert(NR == 1 || !SP, "several right-hand sides run without the absorbing layer");
  extern __shared__ float4 smem4[];
  float* S0 = reinterpret_cast<float*>(smem4);   // [slot][rhs][field] buffers
  float* J0 = S0 + 2 * NR * G::NF * G::SBUF;     // adjoint injection accumulators, [rhs][slot] x TY x TX
  __shared__ int s_abort;

  const int t = threadIdx.x;
  const int lane = t & 31;
  const int warp = t >> 5;
  const bool frame = t < NFRAME;
  const int tile = blockIdx.x;
  const int tix = tile % a.tiles_x;
  const int tiy = tile / a.tiles_x;
  const int gx0 = tix * TX, gy0 = tiy * TY;
  int c0, r0;
  cells_of<R, ADJ>(t, r0, c0);
  const int nx = a.nx, ny = a.ny, nt = a.nt;
  u64* xbuf = reinterpret_cast<u64*>(a.xbuf);
  float2 w2[R + 1];  // stencil weights, packed
#pragma unroll
  for (int m = 0; m <= R; ++m) w2[m] = dup2(a.w[m]);
  const float* IN[2] = {a.in, a.in1};
  float* OUT[2] = {a.out, a.out1};
  float* PART[2] = {a.part, a.part1};

  // halo duty of the first warps: 0 = north, 1 = south, 2 = west, 3 = east neighbour
  const int region = warp & 3;
  const int rrank = (warp >> 2) * 32 + lane;
  int nb = -1;
  if (warp < 4 * G::RCOUNT / 32) {
    if (region == 0 && tiy > 0) nb = tile - a.tiles_x;
    if (region == 1 && tiy < a.tiles_y - 1) nb = tile + a.tiles_x;
    if (region == 2 && tix > 0) nb = tile - 1;
    if (region == 3 && tix < a.tiles_x - 1) nb = tile + 1;
  }

  // forward: P, D ; adjoint: Z (in P, with Z_lo in Pl), G (in D); per right-hand side
  float P[NR][2][2], D[NR][2][2], Pl[NR][2][2];
  float K[2][2], Kl[2][2];
  float SA[2][2], SB[2][2];  // layer factors (SP only)
  bool valid[2][2];
#pragma unroll
  for (int rr = 0; rr < 2; ++rr)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int gx = gx0 + c0 + j, gy = gy0 + r0 + rr;
      const bool v = gx < nx && gy < ny;
      valid[rr][j] = v;
      const long long gi = (long long)gy * nx + gx;
      K[rr][j] = v ? (VARC ? a.kappa[gi] : a.kappa0) : 0.f;
      Kl[rr][j] = v ? (VARC ? a.kappa_lo[gi] : a.kappa0_lo) : 0.f;
      SA[rr][j] = (SP && v) ? a.sp_a[gi] : 1.f;
      SB[rr][j] = (SP && v) ? a.sp_b[gi] : 1.f;
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        P[r][rr][j] = (!ADJ && v) ? IN[r][gi] : 0.f;
        D[r][rr][j] = 0.f;
        Pl[r][rr][j] = 0.f;
      }
    }
  for (int i = t; i < 2 * NR * G::NF * G::SBUF; i += NTHREADS) S0[i] = 0.f;
  if (ADJ)
    for (int i = t; i < NR * 2 * TX * TY; i += NTHREADS) J0[i] = 0.f;
  if (t == 0) s_abort = 0;
  __syncthreads();

  auto Sbuf = [&](int slot, int r) { return S0 + (slot * NR + r) * G::NF * G::SBUF; };
  auto Jbuf = [&](int r, int slot) { return J0 + (r * 2 + slot) * TX * TY; };
  auto Xslot = [&](int tl, int slot, int r) { return xbuf + ((size_t)tl * 2 + slot) * NR * G::SLOT + r * G::SLOT; };
  const HaloDuty<G::PER> duty = halo_duty<R, ADJ>(region, rrank);
  // blocks within R cells of the tile's edge are published
  const bool edge = r0 < R || r0 + 2 > TY - R || c0 < R || c0 + 2 > TX - R;
  auto Xown = [&](int slot, int r) -> u64* {
    return edge ? Xslot(tile, slot, r) + (R == 1 ? 0 : 4 * t) : nullptr;
  };
#pragma unroll
  for (int r = 0; r < NR; ++r)  // publish state 0 (forward: x; adjoint: zero)
    store_state<R, ADJ>(Sbuf(0, r), Xown(0, r), P[r], Pl[r], r0, c0, 0u);

  // The interior's threads serve the tile's sensors.  Adjoint: S^T r_n, n = nt-1-k, of the injected cells into
  // step k's accumulators (KEEP: the first cell of a thread, with its first sensor, stays in registers; the form for
  // two CTAs per SM has none to spare, and kept in shared memory it takes 1.91 instead of 1.82 us at 640 x 512).
  constexpr bool KEEP = CTAS == 1;
  const int ut = t - NFRAME;
  constexpr int NINNER = NTHREADS - NFRAME;
  int e0 = 0, e1 = 0, is0 = 0;
  float iw0 = 0.f;
  InjCell ic0{0, 0, 0};
  if (!frame) {
    const int* ptr = ADJ ? a.tile_inj_ptr : a.tile_samp_ptr;
    e0 = ptr[tile] + ut;
    e1 = ptr[tile + 1];
    if (ADJ && KEEP && e0 < e1) {
      ic0 = a.inj[e0];
      if (ic0.beg < ic0.end) {
        is0 = a.ent_sensor[ic0.beg];
        iw0 = a.ent_w[ic0.beg];
      }
    }
  }
  auto inject = [&](int k) {
    const int n = nt - 1 - k;
    for (int e = e0; e < e1; e += NINNER) {
      const InjCell ic = KEEP && e == e0 ? ic0 : a.inj[e];
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        float s = 0.f;
        for (int q = ic.beg; q < ic.end; ++q) {
          const bool first = KEEP && e == e0 && q == ic.beg;
          const float w = first ? iw0 : a.ent_w[q];
          s = fmaf(w, IN[r][(long long)(first ? is0 : a.ent_sensor[q]) * nt + n], s);
        }
        Jbuf(r, k & 1)[ic.local] = s;
      }
    }
  };
  auto sample = [&](int k) {  // y[:, k] = S P^k
    for (int e = e0; e < e1; e += NINNER) {
      const SampEntry se = a.samp[e];
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const float* b = Sbuf(k & 1, r) + (se.ly + R) * PITCH + XOFF + se.lx;
        if (se.part < 0) {
          const float v = se.w[0] * b[0] + se.w[1] * b[1] + se.w[2] * b[PITCH] + se.w[3] * b[PITCH + 1];
          OUT[r][(long long)se.sensor * nt + k] = v;
        } else {
          PART[r][(long long)se.part * nt + k] = se.w[0] * b[0];
        }
      }
    }
  };
  // state k + 1 of the thread's cells (k = nt - 1: the adjoint's result)
  auto update = [&](int k) {
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const float* own = Sbuf(k & 1, r) + (r0 + R) * PITCH + XOFF + c0;
      float2 L2[2];
      lap_2x2<R, true, false>(own, w2, L2);
      if (ADJ) lap_2x2<R, false, true>(own + G::SBUF, w2, L2);
      const float L[2][2] = {{L2[0].x, L2[0].y}, {L2[1].x, L2[1].y}};

      if (k == nt - 1) {
        if (ADJ) {  // x = S^T r_0 + G^1 + 1/2 L Z^1
          const float* Jc = Jbuf(r, k & 1);
#pragma unroll
          for (int rr = 0; rr < 2; ++rr)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
              if (!valid[rr][j]) continue;
              const int lr = r0 + rr, lc = c0 + j;
              float xv = Jc[lr * TX + lc] + D[r][rr][j] + 0.5f * L[rr][j];
              if (SP && SA[rr][j] != 1.f)  // + ((a-1)/b) Q,  Q = (Z + Z_lo) / kappa
                xv = fmaf((SA[rr][j] - 1.f) / SB[rr][j], (P[r][rr][j] + Pl[r][rr][j]) / (K[rr][j] + Kl[rr][j]), xv);
              OUT[r][(long long)(gy0 + lr) * nx + gx0 + lc] = xv;
            }
        }
        continue;
      }

      float V[2][2], Vl[2][2];
      if (!ADJ) {
        const float cf = (k == 0) ? 0.5f : 1.0f;
#pragma unroll
        for (int rr = 0; rr < 2; ++rr)
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            // D += cf (kappa_hi + kappa_lo) L, the product rounded once before it meets D
            const float inc = fmaf(cf * K[rr][j], L[rr][j], (cf * Kl[rr][j]) * L[rr][j]);
            if (SP)
              D[r][rr][j] = k == 0 ? fmaf(SA[rr][j] - 1.f, P[r][rr][j], SB[rr][j] * inc)
                                   : fmaf(SA[rr][j], D[r][rr][j], SB[rr][j] * inc);
            else
              D[r][rr][j] += inc;
            P[r][rr][j] += D[r][rr][j];
            V[rr][j] = P[r][rr][j];
            Vl[rr][j] = 0.f;
          }
      } else {
        float* Jw = Jbuf(r, k & 1);
#pragma unroll
        for (int rr = 0; rr < 2; ++rr) {
          float2* jp = reinterpret_cast<float2*>(Jw + (r0 + rr) * TX + c0);
          const float2 jv = *jp;
          *jp = make_float2(0.f, 0.f);
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const float inc = f2get(jv, j) + L[rr][j];
            float g = D[r][rr][j] + inc;                         // G += S^T r + L Z
            const float u = fmaf(K[rr][j], g, Kl[rr][j] * g);    // (kappa_hi + kappa_lo) G, rounded once
            float z, zl;
            if (SP && (SA[rr][j] != 1.f || SB[rr][j] != 1.f)) {  // Z = a Z + b kappa G inside the layer
              z = fmaf(SA[rr][j], P[r][rr][j], SB[rr][j] * u);
              zl = SA[rr][j] * Pl[r][rr][j];
            } else {
              float e;
              z = two_sum(P[r][rr][j], u, e);  // Z += kappa G (compensated)
              zl = Pl[r][rr][j] + e;
            }
            if (!valid[rr][j]) g = z = zl = 0.f;
            D[r][rr][j] = g;
            P[r][rr][j] = z;
            Pl[r][rr][j] = zl;
            V[rr][j] = z;
            Vl[rr][j] = zl;
          }
        }
      }
      store_state<R, ADJ>(Sbuf((k + 1) & 1, r), Xown((k + 1) & 1, r), V, Vl, r0, c0, (unsigned)(k + 1));
    }
  };

  auto wait_halo = [&](int k) {  // halo of state k from the neighbour's slot (k & 1)
    if (nb < 0) return;
    float* sc[NR];
    const u64* xs[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      sc[r] = Sbuf(k & 1, r);
      xs[r] = Xslot(nb, k & 1, r);
    }
    if (!load_halo<R, ADJ, NR>(sc, xs, duty, (unsigned)k, a.abort, a.timeout_ns, a.poll_ns)) {
      if (lane == 0) {
        s_abort = 1;
        atomicCAS(a.status, (int)PAT_OK, (int)PAT_ERR_TIMEOUT);
        atomicExch(a.abort, 1);
      }
    }
  };
  if (ADJ && !frame) inject(0);
  __syncthreads();  // state 0 and the first injections
  for (int k = 0; k < nt; ++k) {
    if (frame) {
      wait_halo(k);
    } else {
      update(k);
      if (ADJ && k + 1 < nt) inject(k + 1);  // its accumulators were read and cleared during step k - 1
    }
    __syncthreads();  // the halo of state k
    if (s_abort) break;
    if (frame)
      update(k);
    else if (!ADJ)
      sample(k);
    if (k == nt - 1) break;
    __syncthreads();  // state k + 1
  }
}

__global__ void split_combine_kernel(const float* __restrict__ part, const int* __restrict__ split_sensor,
                                     int nsplit, int nt, float* __restrict__ y) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long long)nsplit * nt) return;
  const int q = (int)(i / nt), t = (int)(i % nt);
  const float* p = part + (long long)4 * q * nt + t;
  y[(long long)split_sensor[q] * nt + t] = ((p[0] + p[nt]) + p[2 * nt]) + p[3 * nt];
}

template <int R, bool ADJ, bool VARC, bool SP, int NR, int CTAS = 1>
void* kfn() {
  return (void*)wave2d_persist_kernel<R, ADJ, VARC, SP, NR, CTAS>;
}

template <int R, bool SP, int CTAS>
void* pick_r(bool adj, bool varc) {
  if (adj) return varc ? kfn<R, true, true, SP, 1, CTAS>() : kfn<R, true, false, SP, 1, CTAS>();
  return varc ? kfn<R, false, true, SP, 1, CTAS>() : kfn<R, false, false, SP, 1, CTAS>();
}

// ctas: CTAs per SM wanted, 1 or (order 2) 2
void* pick(int R, bool adj, bool varc, bool layer, int ctas) {
  if (ctas == 2) return R == 1 ? (layer ? pick_r<1, true, 2>(adj, varc) : pick_r<1, false, 2>(adj, varc)) : nullptr;
  switch (R) {
    case 1: return layer ? pick_r<1, true, 1>(adj, varc) : pick_r<1, false, 1>(adj, varc);
    case 3: return layer ? pick_r<3, true, 1>(adj, varc) : pick_r<3, false, 1>(adj, varc);
    case 5: return layer ? pick_r<5, true, 1>(adj, varc) : pick_r<5, false, 1>(adj, varc);
    case 7: return layer ? pick_r<7, true, 1>(adj, varc) : pick_r<7, false, 1>(adj, varc);
    default: return nullptr;
  }
}

// two right-hand sides, no absorbing layer
void* pick2(int R, bool adj, bool varc) {
#define PAT_P2D2(RR)                                                                              \
  if (R == RR) {                                                                                  \
    if (adj) return varc ? kfn<RR, true, true, false, 2>() : kfn<RR, true, false, false, 2>();    \
    return varc ? kfn<RR, false, true, false, 2>() : kfn<RR, false, false, false, 2>();           \
  }
  PAT_P2D2(1)
  PAT_P2D2(3)
  PAT_P2D2(5)
  PAT_P2D2(7)
#undef PAT_P2D2
  return nullptr;
}

size_t smem_bytes(int R, bool adj, int nr = 1) {
  const size_t sbuf = (size_t)(TY + 2 * R) * PITCH;
  const size_t nf = adj ? 2 : 1;
  return (size_t)nr * (2 * nf * sbuf + (adj ? 2 * (size_t)TX * TY : 0)) * sizeof(float);
}

cudaError_t prepare(void* f, int R, bool adj, int nr = 1) {
  return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes(R, adj, nr));
}

// CTAs of a kernel that the current device holds at once.
int resident(void* f, int R, bool adj, int nr = 1) {
  int dev = 0, sms = 0, per_sm = 0;
  if (!f || cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      prepare(f, R, adj, nr) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, NTHREADS, smem_bytes(R, adj, nr)) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return sms * per_sm;
}

}  // namespace

cudaError_t persist2d_split_combine(const float* part, const int* split_sensor, int nsplit, int nt, float* y,
                                    cudaStream_t st) {
  if (nsplit <= 0) return cudaSuccess;
  const long long n = (long long)nsplit * nt;
  split_combine_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(part, split_sensor, nsplit, nt, y);
  return cudaGetLastError();
}

bool persist2d_supported(int R, bool) { return R == 1 || R == 3 || R == 5 || R == 7; }
int persist2d_tile_x() { return TX; }
int persist2d_tile_y() { return TY; }
size_t persist2d_xbuf_words(int R, int ntiles, int nr) {
  const int slot = R == 1 ? Geo<1, true>::SLOT : Geo<3, true>::SLOT;  // 8-cell frames from R = 3 on
  return (size_t)nr * ntiles * 2 * slot;
}

static int max_ctas(int R, bool adj, bool varc) {
  static PerDevice kept[kMaxR + 1][2][2];
  return kept[R][adj][varc].get(current_device(), [&] {
    const int fit = resident(pick(R, adj, varc, false, 1), R, adj);
    return R == 1 ? std::max(fit, resident(pick(R, adj, varc, false, 2), R, adj)) : fit;
  });
}

bool persist2d_fits(int R, bool varc, long long tiles) {
  int dev = 0, sms = 0, smem = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  // more tiles than shared memory has room for need no question to the kernels (which loads them)
  if (tiles > (long long)sms * (smem / (int)smem_bytes(R, true))) return false;
  return tiles <= std::min(max_ctas(R, false, varc), max_ctas(R, true, varc));
}

cudaError_t persist2d_launch(int R, bool adj, bool varc, bool layer, const Persist2DArgs& a, int nctas,
                             cudaStream_t st) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  void* f = pick(R, adj, varc, layer, nctas > sms ? 2 : 1);
  if (!f) return cudaErrorInvalidValue;
  e = prepare(f, R, adj);
  if (e != cudaSuccess) return e;
  void* args[] = {(void*)&a};
  return cudaLaunchCooperativeKernel(f, dim3(nctas), dim3(NTHREADS), args, smem_bytes(R, adj), st);
}

int persist2d_max_ctas2(int R, bool adj, bool varc) { return resident(pick2(R, adj, varc), R, adj, 2); }

cudaError_t persist2d_launch2(int R, bool adj, bool varc, const Persist2DArgs& a, int nctas, cudaStream_t st) {
  void* f = pick2(R, adj, varc);
  if (!f) return cudaErrorInvalidValue;
  cudaError_t e = prepare(f, R, adj, 2);
  if (e != cudaSuccess) return e;
  void* args[] = {(void*)&a};
  return cudaLaunchCooperativeKernel(f, dim3(nctas), dim3(NTHREADS), args, smem_bytes(R, adj, 2), st);
}

}  // namespace pat
