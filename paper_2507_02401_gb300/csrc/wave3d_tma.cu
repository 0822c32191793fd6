// 3D wave step with TMA-fed plane pipelines (the HBM-bound volumes): one
// launch per time step of the three-level recurrence
//
//   next = c_cur cur - c_prev prev + c_lap (kappa_hi + kappa_lo) L cur
//
// (paper Sec. 2, Eq. wave_equation; forward P^{n+1} = 2P^n - P^{n-1} +
// kappa L P^n).  The adjoint Q^n = 2Q^{n+1} - Q^{n+2} + L(kappa Q^{n+1}) has
// this form for a constant kappa, and for a varying one in Z = kappa Q:
// Z^n = 2Z^{n+1} - Z^{n+2} + kappa (L Z^{n+1} + S^T r_n); its final step,
// x = (Z^1 - Z^2) / kappa + 1/2 L Z^1 + S^T r_0, leaves that variable.  So a
// varying medium adds only the reads of the own cells' kappa (hi and lo).
//
// A CTA owns a 64 x 16 column of cells and marches through a range of z
// planes.  One thread issues TMA loads of each plane of `cur` as an
// (64+16) x (16+2R) box (x/y halo included, zero outside the grid) into a
// ring of shared-memory slots, PD planes ahead of the plane being computed,
// plus the own 64 x 16 tile of `prev`; completion is tracked by one mbarrier
// per slot.  Each thread owns 2 rows x 4 columns: x/y neighbours come from the
// centre plane's slot, z neighbours from a register ring of 2R+1 planes.
// Compulsory DRAM traffic per point-update: cur and prev read once, next
// written once (12 B); halo re-reads are served by L2.
#include <cudaTypedefs.h>

#include <mutex>
#include <type_traits>

#include "internal.h"
#include "stencil.cuh"
#include "tma.cuh"

namespace pat {
namespace {

constexpr int TX = 64, TY = 16, THREADS = (TX / 4) * (TY / 2);  // 128

template <int R>
struct G3 {
  // prefetch distance in planes: one at order 6, where the shorter ring lets three CTAs share an SM
  static constexpr int PD = R == 5 ? 1 : 2;
  static constexpr int XH = R <= 4 ? 4 : 8;      // box columns left of the tile (>= R, 16-byte aligned)
  static constexpr int BW = TX + 2 * XH;         // box width, 72 or 80 floats
  static constexpr int BH = TY + 2 * R;
  static constexpr int BOX = BW * BH;            // floats a TMA load brings
  static constexpr int PLANE = (BOX + 31) / 32 * 32;  // floats per cur slot (128-byte aligned slots)
  static constexpr int NS = R + 1 + PD;  // cur slots: centre plane .. queue plane + PD
  static constexpr int PREV = TX * TY;   // floats per prev slot
  static constexpr int NSP = PD + 1;
  static constexpr size_t SMEM = sizeof(float) * ((size_t)NS * PLANE + (size_t)NSP * PREV) + 8 * (NS + NSP);
};

// Sensor s = b + t * gridDim.x is sampled by thread t of CTA b: the sensors are spread over every CTA
// of the wave (a few per CTA) instead of loading the first CTAs with all of them.
__device__ __forceinline__ void fused_sample3(const StepArgs& a, long long bid, int t) {
  const long long gs = bid + (long long)t * gridDim.x;
  if (a.y == nullptr || gs >= a.ns) return;
  const int s = (int)gs;
  float v = 0.f;
  for (int k = 0; k < a.corners; ++k) v = fmaf(a.sens_w[s * a.corners + k], a.cur[a.sens_cell[s * a.corners + k]], v);
  a.y[(long long)s * a.nt + a.t_sample] = v;
}

// Runs f(S, i + S) for S = 0 .. Q-1 while i + S < n (S a compile-time constant in each call); false as
// soon as one call returns false.
template <int S, int Q, class F>
__device__ __forceinline__ bool march(F& f, int i, int n) {
  if constexpr (S == Q) {
    return true;
  } else {
    if (i + S >= n) return true;
    if (!f(std::integral_constant<int, S>{}, i + S)) return false;
    return march<S + 1, Q>(f, i, n);
  }
}

// The adjoint's injection S^T r_m into one cell: sum of w r_m over the cell's sensor entries.
__device__ __forceinline__ float inj_sum(const StepArgs& a, const InjCell& c) {
  float v = 0.f;
  for (int q = c.beg; q < c.end; ++q) v = fmaf(a.ent_w[q], a.inj_r[(long long)a.ent_sensor[q] * a.nt + a.inj_t], v);
  return v;
}

// INJ: the adjoint's injection S^T r_m into the CTA's own cells of `next` after the step (per-CTA lists)
// Work split (column-fastest): CTA b takes column b mod columns and the (b div columns)-th of
// nchunks equal z ranges, so CTAs that run together stream neighbouring columns of the same rows.
// VARC: varying medium (a.final_step: the adjoint's last step)
template <int R, bool INJ, bool RING, bool VARC>
__global__ void __launch_bounds__(THREADS) step3d_tma_kernel(const StepArgs a, const __grid_constant__ CUtensorMap mcur,
                                                             const __grid_constant__ CUtensorMap mprev, int cols_x,
                                                             int nchunks, int* status, long long timeout_ns) {
  using G = G3<R>;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  float* ring = reinterpret_cast<float*>(smem_raw);
  float* pring = ring + G::NS * G::PLANE;
  uint64_t* bars = reinterpret_cast<uint64_t*>(pring + G::NSP * G::PREV);
  uint64_t* pbars = bars + G::NS;

  constexpr int XH = G::XH, BW = G::BW, PD = G::PD;
  const int t = threadIdx.x;
  const long long bid = blockIdx.x;

  const int nx = a.nx, ny = a.ny, nz = a.nz;
  const int pitch = a.pitch;
  const long long plane = (long long)pitch * ny;
  const int c0 = (t % (TX / 4)) * 4, r0 = (t / (TX / 4)) * 2;
  const long long ncols = (long long)cols_x * ((ny + TY - 1) / TY);
  const bool has_prev = a.prev != nullptr;
  const float ck = a.c_lap * a.kappa0, ckl = a.c_lap * a.kappa0_lo;
  const float2 ck2 = dup2(ck), ckl2 = dup2(ckl), ccur2 = dup2(a.c_cur), ncprev2 = dup2(-a.c_prev), m2 = dup2(-2.f),
               clap2 = dup2(a.c_lap);
  float2 w2[R + 1];
#pragma unroll
  for (int m = 0; m <= R; ++m) w2[m] = dup2(a.w[m]);

  bool ok_all = true;
  int issued = 0;       // cur planes issued (thread 0)
  int issued_prev = 0;  // prev planes issued
  const int col = (int)(bid % ncols);
  const long long zr = bid / ncols;
  const int z0 = (int)(zr * nz / nchunks);
  const int z1 = (int)((zr + 1) * nz / nchunks);
  const int gx0 = (col % cols_x) * TX, gy0 = (col / cols_x) * TY;
  const int nloc = z1 - z0;   // planes computed
  const int ncur = nloc + R;  // cur planes j = 0 .. ncur-1 (z = zb + j zd) go through the ring
  // march upwards from z0, or downwards from z1 - 1 (a.flip): the stencil is symmetric in z and each pair
  // is summed first, so both directions give the same bits
  const int zb = a.flip ? z1 - 1 : z0, zd = a.flip ? -1 : 1;
  if (t == 0) {
    for (int s = 0; s < G::NS + G::NSP; ++s) mbar_init(&bars[s], 1);
    fence_mbar_init();
  }
  // The CTA's injected cells (thread t takes entries t and t + THREADS; 256^3 with 4096 sensors has up to 302 in a
  // CTA).  The chain list bounds -> cell -> sensor -> r_m is walked where the thread waits anyway (the previous step's
  // end, the first copies, the first planes) and not in the march, whose instructions are the bound; what is left
  // after it is two additions per thread (and the entries beyond those, or beyond a cell's first sensor).  us per K*
  // step at 256^3, one entry walked link by link in the march -> this: order 2 30.6 -> 28.9, order 4 39.5 -> 38.0,
  // order 6 58.1 -> 54.6, order 8 79.3 -> 76.3.  The lists are the plan's: they may be read before the wait.
  constexpr int NPRE = R == 1 && VARC ? 1 : 2;  // a second one there costs the sixth CTA per SM (94 registers)
  int ie0 = 0, ie1 = 0, is[NPRE] = {};
  InjCell ic[NPRE] = {};
  float iw[NPRE] = {}, ir[NPRE] = {};
  if (INJ) {
    ie0 = a.inj_tile_ptr[bid] + t;
    ie1 = a.inj_tile_ptr[bid + 1];
#pragma unroll
    for (int j = 0; j < NPRE; ++j)
      if (ie0 + j * THREADS < ie1) ic[j] = a.inj_tile[ie0 + j * THREADS];
  }
  __syncthreads();
  griddep_wait();  // everything above overlaps the previous step's last CTAs
  griddep_trigger();
  auto issue_cur = [&](int j) {
    issued = j + 1;
    const int s = j % G::NS;
    mbar_expect_tx(&bars[s], G::BOX * 4);
    tma_load_3d(ring + s * G::PLANE, &mcur, gx0 - XH, gy0 - R, zb + j * zd, &bars[s]);
  };
  auto issue_prev = [&](int j) {
    issued_prev = j + 1;
    const int s = j % G::NSP;
    mbar_expect_tx(&pbars[s], G::PREV * 4);
    tma_load_3d(pring + s * G::PREV, &mprev, gx0, gy0, zb + j * zd, &pbars[s]);
  };
  if (t == 0) {
    for (int j = 0; j < min(R + PD, ncur); ++j) issue_cur(j);
    if (has_prev)
      for (int j = 0; j < min(PD, nloc); ++j) issue_prev(j);
  }
  fused_sample3(a, bid, t);  // the forward's sensor samples of cur, while the first copies are in flight

#pragma unroll
  for (int j = 0; j < NPRE; ++j)
    if (INJ && ic[j].beg < ic[j].end) {
      is[j] = a.ent_sensor[ic[j].beg];
      iw[j] = a.ent_w[ic[j].beg];
    }

  // register ring of the own cells: at the first plane q[k] = plane zb + (k - R) zd.  Not through the read-only
  // path (__ldg): it is for data that no one writes while the kernel lives, and this kernel starts while the
  // previous step still writes `cur`.
  float4 q[2 * R + 1][2];
#pragma unroll
  for (int i = 0; i < R; ++i)  // the R planes before zb straight from global memory
#pragma unroll
    for (int rr = 0; rr < 2; ++rr) {
      const int z = zb + (i - R) * zd, gy = gy0 + r0 + rr, gx = gx0 + c0;
      q[i][rr] = (z >= 0 && z < nz && gy < ny && gx < nx)
                     ? ld_stream4(a.cur + z * plane + (long long)gy * pitch + gx)
                     : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  // varying medium: the own cells' kappa, one plane ahead of its use
  float4 kh[2], kl[2];
  auto fetch_kappa = [&](int i) {
#pragma unroll
    for (int rr = 0; rr < 2; ++rr) {
      const int gy = gy0 + r0 + rr, gx = gx0 + c0;
      kh[rr] = kl[rr] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (i < nloc && gy < ny && gx < nx) {
        const long long gi = (zb + i * zd) * plane + (long long)gy * pitch + gx;
        kh[rr] = ld_stream4(a.kappa + gi);
        kl[rr] = ld_stream4(a.kappa_lo + gi);
      }
    }
  };
  if (VARC) fetch_kappa(0);
  bool ok = true;
#pragma unroll
  for (int i = 0; i < R; ++i) {  // planes zb .. zb + (R-1) zd from the ring
    ok = ok && (i >= ncur || mbar_wait(&bars[i % G::NS], (i / G::NS) & 1, timeout_ns));
#pragma unroll
    for (int rr = 0; rr < 2; ++rr)
      q[R + i][rr] = *reinterpret_cast<const float4*>(ring + (i % G::NS) * G::PLANE + (r0 + rr + R) * BW + XH + c0);
  }

#pragma unroll
  for (int j = 0; j < NPRE; ++j)
    if (INJ && ic[j].beg < ic[j].end) ir[j] = a.inj_r[(long long)is[j] * a.nt + a.inj_t];

  // One plane of the march.  RING: the z queue is a ring in registers, logical entry k (plane z - R + k)
  // of plane i sitting in q[(k + i) % Q]; the loop is unrolled Q times, so S = i % Q is a compile-time
  // constant in every copy and no queue entry moves between registers (fewer instructions, a Q times
  // larger loop body).  Otherwise S = 0 and the queue shifts after every plane.
  constexpr int Q = 2 * R + 1;
  auto step = [&](auto sc, int i) -> bool {
    constexpr int S = decltype(sc)::value;
    const int jq = i + R;  // queue plane
    bool good = ok && mbar_wait(&bars[jq % G::NS], (jq / G::NS) & 1, timeout_ns);
    if (has_prev) good = good && mbar_wait(&pbars[i % G::NSP], (i / G::NSP) & 1, timeout_ns);
    if (__syncthreads_or(!good)) {
      if (t == 0) atomicCAS(status, (int)PAT_OK, (int)PAT_ERR_TIMEOUT);
      return false;
    }
    // the slots refilled here were read while plane i - 1 was computed, which every thread has left at the
    // barrier above: one barrier per plane
    if (t == 0) {
      fence_proxy_async_shared();  // their reads went through the generic proxy
      if (i + R + PD < ncur) issue_cur(i + R + PD);
      if (has_prev && i + PD < nloc) issue_prev(i + PD);
    }
#pragma unroll
    for (int rr = 0; rr < 2; ++rr)
      q[(2 * R + S) % Q][rr] =
          *reinterpret_cast<const float4*>(ring + (jq % G::NS) * G::PLANE + (r0 + rr + R) * BW + XH + c0);

    const float* cen = ring + (i % G::NS) * G::PLANE;
    float2 L[2][2];  // packed pairs: cells (2p, 2p+1) of row rr
    lap_2x4_x2<R>(cen, BW, r0 + R, XH + c0, w2, L);
    const int z = zb + i * zd;
#pragma unroll
    for (int rr = 0; rr < 2; ++rr) {
      const float4 pv = has_prev ? *reinterpret_cast<const float4*>(pring + (i % G::NSP) * G::PREV + (r0 + rr) * TX + c0)
                                 : make_float4(0.f, 0.f, 0.f, 0.f);
      float2 out[2];
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        const float2 c = p ? hi2(q[(R + S) % Q][rr]) : lo2(q[(R + S) % Q][rr]);
        float2 acc = L[rr][p];
#pragma unroll
        for (int m = 1; m <= R; ++m) {
          const float2 up = p ? hi2(q[(R + m + S) % Q][rr]) : lo2(q[(R + m + S) % Q][rr]);
          const float2 dn = p ? hi2(q[(R - m + S) % Q][rr]) : lo2(q[(R - m + S) % Q][rr]);
          acc = __ffma2_rn(w2[m], __ffma2_rn(c, m2, __fadd2_rn(up, dn)), acc);
        }
        // c_cur c - c_prev prev + (ck + ckl) acc, the last product rounded once
        float2 v = __fmul2_rn(ccur2, c);
        if (has_prev) v = __ffma2_rn(ncprev2, p ? hi2(pv) : lo2(pv), v);
        if (!VARC) {
          out[p] = __fadd2_rn(v, __ffma2_rn(ck2, acc, __fmul2_rn(ckl2, acc)));
        } else {
          const float2 h = p ? hi2(kh[rr]) : lo2(kh[rr]), l = p ? hi2(kl[rr]) : lo2(kl[rr]);
          if (a.final_step)
            out[p] = make_float2(v.x / h.x + a.c_lap * acc.x, v.y / h.y + a.c_lap * acc.y);
          else
            out[p] = __fadd2_rn(v, __ffma2_rn(__fmul2_rn(clap2, h), acc, __fmul2_rn(__fmul2_rn(clap2, l), acc)));
        }
      }
      const int gy = gy0 + r0 + rr, gx = gx0 + c0;
      if (gy < ny && gx < nx)
        *reinterpret_cast<float4*>(a.next + z * plane + (long long)gy * pitch + gx) =
            make_float4(out[0].x, out[0].y, out[1].x, out[1].y);
    }
    if (VARC) fetch_kappa(i + 1);
    return true;
  };
  if constexpr (RING) {
    for (int i = 0; i < nloc; i += Q)
      if (!march<0, Q>(step, i, nloc)) {
        ok_all = false;
        break;
      }
  } else {  // the queue shifts by one plane after every step (one copy of the loop body)
    for (int i = 0; i < nloc; ++i) {
      if (!step(std::integral_constant<int, 0>{}, i)) {
        ok_all = false;
        break;
      }
#pragma unroll
      for (int k = 0; k < 2 * R; ++k) {
        q[k][0] = q[k + 1][0];
        q[k][1] = q[k + 1][1];
      }
    }
  }
  if (INJ && ok_all) {  // every thread's stores to `next` precede the injection (same CTA)
    __syncthreads();
    auto scale = [&](const InjCell& c) { return VARC && !a.final_step ? a.kappa[c.local] : 1.f; };
#pragma unroll
    for (int j = 0; j < NPRE; ++j)
      if (ie0 + j * THREADS < ie1) {
        float v = iw[j] * ir[j];
        for (int q = ic[j].beg + 1; q < ic[j].end; ++q)
          v = fmaf(a.ent_w[q], a.inj_r[(long long)a.ent_sensor[q] * a.nt + a.inj_t], v);
        a.next[ic[j].local] += scale(ic[j]) * v;
      }
    for (int e = ie0 + NPRE * THREADS; e < ie1; e += THREADS)
      a.next[a.inj_tile[e].local] += scale(a.inj_tile[e]) * inj_sum(a, a.inj_tile[e]);
  }
  // after a timed-out wait: give the copies still in flight (the last one of
  // each slot) a bounded chance to land before the CTA's shared memory goes away
  if (t == 0 && !ok_all) {
    for (int j = max(0, issued - G::NS); j < issued; ++j) mbar_wait(&bars[j % G::NS], (j / G::NS) & 1, timeout_ns);
    for (int j = max(0, issued_prev - G::NSP); j < issued_prev; ++j)
      mbar_wait(&pbars[j % G::NSP], (j / G::NSP) & 1, timeout_ns);
  }
}

using KernelFn = void (*)(const StepArgs, const CUtensorMap, const CUtensorMap, int, int, int*, long long);

// The register ring is built for R <= 3 only (tma3d_split).
template <int R, bool VARC>
KernelFn kernel_rv(bool inj, bool ring) {
  if constexpr (R <= 3) {
    if (ring) return inj ? step3d_tma_kernel<R, true, true, VARC> : step3d_tma_kernel<R, false, true, VARC>;
  }
  return inj ? step3d_tma_kernel<R, true, false, VARC> : step3d_tma_kernel<R, false, false, VARC>;
}

KernelFn kernel_for(int R, bool inj, bool ring, bool varc) {
  switch (R) {
    case 1: return varc ? kernel_rv<1, true>(inj, ring) : kernel_rv<1, false>(inj, ring);
    case 3: return varc ? kernel_rv<3, true>(inj, ring) : kernel_rv<3, false>(inj, ring);
    case 5: return varc ? kernel_rv<5, true>(inj, ring) : kernel_rv<5, false>(inj, ring);
    case 7: return varc ? kernel_rv<7, true>(inj, ring) : kernel_rv<7, false>(inj, ring);
    default: return nullptr;
  }
}

int smem_for(int R) {
  return (int)(R == 1 ? G3<1>::SMEM : R == 3 ? G3<3>::SMEM : R == 5 ? G3<5>::SMEM : G3<7>::SMEM);
}

// Co-resident CTAs of the step kernel (with and without injection and ring) on the current device; the first call
// sets the kernels' shared-memory attribute.
int resident(int R, bool varc) {
  static PerDevice kept[kMaxR + 1][2];
  return kept[R][varc].get(current_device(), [&] {
    int dev = 0, sms = 0, best = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    for (int v = 0; v < 4; ++v) {
      const KernelFn fn = kernel_for(R, v & 1, v & 2, varc);
      int per = 0;
      if (!fn ||
          cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_for(R)) != cudaSuccess ||
          cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, THREADS, smem_for(R)) != cudaSuccess) {
        cudaGetLastError();
        return 0;
      }
      best = v == 0 || per < best ? per : best;
    }
    return sms * best;
  });
}

}  // namespace

// cuTensorMapEncodeTiled through the runtime's driver entry point (no libcuda link);
// nullptr when the driver does not provide it.
void* tma_encoder_raw() {
  static void* fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = p;
    else
      cudaGetLastError();
  });
  return fn;
}


bool tma3d_supported(int R) { return R == 1 || R == 3 || R == 5 || R == 7; }

cudaError_t tma3d_encode(const float* base, int nx, int pitch, int ny, int nz, int R, CUtensorMap* cur,
                         CUtensorMap* prev) {
  auto fn = tma_encoder();
  if (!fn) return cudaErrorNotSupported;
  const cuuint64_t dims[3] = {(cuuint64_t)nx, (cuuint64_t)ny, (cuuint64_t)nz};
  const cuuint64_t strides[2] = {(cuuint64_t)pitch * 4, (cuuint64_t)pitch * ny * 4};
  const cuuint32_t estr[3] = {1, 1, 1};
  const cuuint32_t box_c[3] = {(cuuint32_t)(TX + (R <= 4 ? 8 : 16)), (cuuint32_t)(TY + 2 * R), 1};
  const cuuint32_t box_p[3] = {(cuuint32_t)TX, (cuuint32_t)TY, 1};
  CUresult r1 = fn(cur, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(base), dims, strides, box_c, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  CUresult r2 = fn(prev, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(base), dims, strides, box_p, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return (r1 == CUDA_SUCCESS && r2 == CUDA_SUCCESS) ? cudaSuccess : cudaErrorInvalidValue;
}

// Work split of a step launch: columns (64 x 16 cells) x nchunks equal z ranges, column-fastest.  Few
// columns (fewer than a quarter of the co-resident CTAs; 64 at 256^3): as many z ranges as keep every
// CTA in one wave (9 at 256^3: 576 CTAs of 28-29 planes), so no second wave leaves SMs idle at the end
// of a step.  Many columns (256 at 512^3): ranges of at least 16 planes, doubled while the grid keeps
// >= 6 CTAs per SM.  Measured at 256^3, order 4: 33.6 / 36.7 us per K / K* step against 38.0 / 40.3 us with
// 16-plane ranges in 1024 CTAs.  (Equal z-fastest shares of the (column, plane) work lost on an earlier form
// of the kernel: CTAs that run together no longer share x/y halos through L2.)
Tma3dSplit tma3d_split(int R, bool varc, int nx, int ny, int nz) {
  const int cap = resident(R, varc);
  if (cap <= 0) return Tma3dSplit{0, 0, false};
  const long long cols = (long long)((nx + TX - 1) / TX) * ((ny + TY - 1) / TY);
  int chunks;
  if (cols * 4 < cap) {
    chunks = (int)(cap / cols);
  } else {
    int dev = 0, sms = 148;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int zc = 16;
    while (zc < nz && cols * ((nz + zc * 2 - 1) / (zc * 2)) >= 6LL * sms) zc *= 2;
    chunks = (nz + zc - 1) / zc;
  }
  if (chunks > nz) chunks = nz;
  // the register-ring march saves the queue's register moves where issue is the bound (one-wave grids:
  // 33.6 / 36.7 us against 36.6 / 39.0 per K / K* step at 256^3), but its larger body costs where DRAM is
  // (many columns: 275.1 / 281.6 us against 261.5 / 270.8 at 512^3)
  return Tma3dSplit{(int)(cols * chunks), chunks, cols * 4 < cap && R <= 3};
}

// CTA holding cell (x, y, z) (the kernel's split: chunk zr holds z in [zr nz / k, (zr + 1) nz / k)).
int tma3d_cta_of(int nx, int ny, int nz, const Tma3dSplit& sp, int x, int y, int z) {
  const long long cols_x = (nx + TX - 1) / TX;
  const long long ncols = cols_x * ((ny + TY - 1) / TY);
  const long long col = (long long)(y / TY) * cols_x + x / TX;
  long long zr = (long long)z * sp.nchunks / nz;
  while (zr + 1 < sp.nchunks && (zr + 1) * nz / sp.nchunks <= z) ++zr;
  while (zr > 0 && zr * nz / sp.nchunks > z) --zr;
  return (int)(zr * ncols + col);
}

long long tma3d_threads(int nctas) { return (long long)nctas * THREADS; }

cudaError_t step3d_tma_launch(int R, const StepArgs& a, const CUtensorMap& cur, const CUtensorMap& prev,
                              const Tma3dSplit& sp, int* status, long long timeout_ns, cudaStream_t st) {
  const KernelFn fn = kernel_for(R, a.inj_r != nullptr, sp.ring, a.kappa != nullptr);
  if (!fn) return cudaErrorInvalidValue;
  return launch_pdl(fn, sp.nctas, THREADS, smem_for(R), st, a, cur, prev, (a.nx + TX - 1) / TX, sp.nchunks, status,
                    timeout_ns);
}

}  // namespace pat
