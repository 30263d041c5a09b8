// ulp_mixed.cu -- mixed-precision inner solve of Algorithm 1 (reliable-update PCG).
//
// The Krylov recurrence runs on FP32 planes: search direction d, A d, the
// residual r, the preconditioned residual s and the correction x gathered
// since the last refresh, with FP32 copies of the Eq. (UV) weights and the
// diagonal formed on the fly from them.  FP64 is kept where it decides the
// answer:
//   - the inner products behind alpha and beta are accumulated per lane as
//     double-float pairs (exact FP32 products, compensated sums) and summed
//     across lanes and tiles in FP64, so they are FP64-accurate;
//   - alpha, beta, delta and the stop tests are FP64 (the shared finisher);
//   - phi itself stays FP64: every refresh period (Algorithm 1's true-residual
//     step, every 20 iterations here) the FP32 correction is folded into phi
//     and r = b - A phi is recomputed with the FP64 weights and FP64 phi.
// Bytes per pixel per iteration: 24 (phase A) + 32 (phase B) versus 112 in FP64.
#include "ulp_flow32.cuh"
#include "ulp_host.h"

namespace ulp {

// Phase B's ring slots (kRingB32 per warp, inside the warp's share of phase A's ring).
constexpr int kLeadB32 = 3;
constexpr int kRingB32 = kLeadB32 + 1;  // elementwise: a slot is refilled one row after it was read
struct SlotB32 {
  float2 d[32], x[32], q[32], r[32], di[32];
};
static_assert(kRingB32 * sizeof(SlotB32) <= kRing32 * sizeof(Slot32), "phase B's ring fits phase A's");

// x += alpha d; then either r -= alpha q, s = M^-1 r (partials) or, on a
// refresh iteration, phi += x, x = 0 (the residual is then recomputed in FP64).
// wring: the warp's share of phase A's ring, through which the rows stream kLeadB32
// ahead (or null, and on refresh iterations: loads two rows ahead in registers).
template <int KIND>
__device__ __forceinline__ void b32_tile(const PcgArgs& a, const MapDesc& M, const FlowMap& L, int t, int lane,
                                         unsigned char* wring) {
  const TileGeo g = tile_geo(M, t, a.R);
  const size_t P = M.pitch;
  const long long it = L.iter;
  const bool refresh = (it % M.refresh) == 0;
  const float* d = (it & 1) ? M.h.d0 : M.h.d1;
  const float alpha = (float)L.alpha;
  const int j = g.j0 + 2 * lane;
  const float2 z2 = make_float2(0.f, 0.f);
  struct Row {
    float2 d, x, q, r, di;
  };
  auto load = [&](int i) {
    Row w{z2, z2, z2, z2, z2};
    if (i < g.i1) {
      const size_t off = (size_t)i * P + j;
      w.d = ldf2(d, off);
      w.x = ldf2(M.h.x, off);
      if (!refresh) {
        w.q = ldf2(M.h.q, off);
        w.r = ldf2(M.h.r, off);
        if (KIND == kJacobi) w.di = ldf2(M.h.Dinv, off);
      }
    }
    return w;
  };
  DF rs, rr;
  if (!refresh && wring) {
    // the rows stream through the warp's ring in shared memory (phase A's ring, free in
    // this phase), kLeadB32 rows ahead; the arithmetic is that of the loop below
    SlotB32* ring = reinterpret_cast<SlotB32*>(wring);
    auto issue = [&](SlotB32& sl, int i) {
      const size_t off = (size_t)i * P + j;
      cpa8(&sl.d[lane], d + off, 8);
      cpa8(&sl.x[lane], M.h.x + off, 8);
      cpa8(&sl.q[lane], M.h.q + off, 8);
      cpa8(&sl.r[lane], M.h.r + off, 8);
      if (KIND == kJacobi) cpa8(&sl.di[lane], M.h.Dinv + off, 8);
    };
#pragma unroll
    for (int k = 0; k < kLeadB32; ++k) {
      if (g.i0 + k < g.i1) issue(ring[k], g.i0 + k);
      cpa_commit();
    }
    for (int i = g.i0; i < g.i1; ++i) {
      cpa_wait<kLeadB32 - 1>();
      const SlotB32& sl = ring[(i - g.i0) % kRingB32];
      const float2 dv = sl.d[lane], qv = sl.q[lane];
      float2 xv = sl.x[lane], r = sl.r[lane];
      const float2 di = (KIND == kJacobi) ? sl.di[lane] : z2;
      if (i + kLeadB32 < g.i1) issue(ring[(i + kLeadB32 - g.i0) % kRingB32], i + kLeadB32);
      cpa_commit();
      const size_t off = (size_t)i * P + j;
      xv.x = __fmaf_rn(alpha, dv.x, xv.x);
      xv.y = __fmaf_rn(alpha, dv.y, xv.y);
      stf2(M.h.x, off, xv);
      r.x = __fmaf_rn(-alpha, qv.x, r.x);
      r.y = __fmaf_rn(-alpha, qv.y, r.y);
      stf2(M.h.r, off, r);
      if (KIND == kJacobi) {
        const float2 sv = make_float2(di.x * r.x, di.y * r.y);
        stf2(M.h.s, off, sv);
        rs.add_prod(r.x, sv.x);
        rs.add_prod(r.y, sv.y);
      }
      rr.add_prod(r.x, r.x);
      rr.add_prod(r.y, r.y);
    }
    cpa_wait_all();
    const double vrr = rr.value();
    flow_publish(a, L, t, warp_sum((KIND == kIdentity) ? vrr : rs.value()), warp_sum(vrr), 0.0, lane);
    return;
  }
  Row c0 = load(g.i0), c1 = load(g.i0 + 1);
  for (int i = g.i0; i < g.i1; ++i) {
    const Row c2 = load(i + 2);
    const size_t off = (size_t)i * P + j;
    float2 xv = c0.x;
    xv.x = __fmaf_rn(alpha, c0.d.x, xv.x);
    xv.y = __fmaf_rn(alpha, c0.d.y, xv.y);
    if (refresh) {
      double2 ph = ld2(M.f.phi, off);
      ph.x += (double)xv.x;
      ph.y += (double)xv.y;
      st2(M.f.phi, off, ph);
      stf2(M.h.x, off, z2);
    } else {
      stf2(M.h.x, off, xv);
      float2 r = c0.r;
      r.x = __fmaf_rn(-alpha, c0.q.x, r.x);
      r.y = __fmaf_rn(-alpha, c0.q.y, r.y);
      stf2(M.h.r, off, r);
      if (KIND == kJacobi) {
        const float2 s = make_float2(c0.di.x * r.x, c0.di.y * r.y);
        stf2(M.h.s, off, s);
        rs.add_prod(r.x, s.x);
        rs.add_prod(r.y, s.y);
      }
      rr.add_prod(r.x, r.x);
      rr.add_prod(r.y, r.y);
    }
    c0 = c1;
    c1 = c2;
  }
  const double vrr = rr.value();
  flow_publish(a, L, t, refresh ? 0.0 : warp_sum((KIND == kIdentity) ? vrr : rs.value()), refresh ? 0.0 : warp_sum(vrr),
               0.0, lane);
}

// phi += x, x = 0 (end of the solve).
__device__ __forceinline__ void fold_tile(const PcgArgs& a, const MapDesc& M, int t, int lane) {
  const TileGeo g = tile_geo(M, t, a.R);
  const size_t P = M.pitch;
  const int j = g.j0 + 2 * lane;
  for (int i = g.i0; i < g.i1; ++i) {
    const size_t off = (size_t)i * P + j;
    const float2 xv = ldf2(M.h.x, off);
    double2 ph = ld2(M.f.phi, off);
    ph.x += (double)xv.x;
    ph.y += (double)xv.y;
    st2(M.f.phi, off, ph);
    stf2(M.h.x, off, make_float2(0.f, 0.f));
  }
}

// phase A's row rings, phase B's in turn (dynamic: they share the block with FlowShared)
struct Rings32 {
  Slot32 s[kWarps][kRing32];
};

// The whole inner solve of every map, as k_pcg64.
template <int KIND>
__global__ void __launch_bounds__(kThreads, 2) k_pcg32(PcgArgs a) {
  extern __shared__ __align__(16) unsigned char pcg32_dsm[];
  Slot32* ring = reinterpret_cast<Rings32*>(pcg32_dsm)->s[threadIdx.x >> 5];
  __shared__ FlowShared fs;
  const int lane = threadIdx.x & 31;
  const int gw = blockIdx.x * kWarps + (threadIdx.x >> 5);
  const int NW = gridDim.x * kWarps;
  flow_begin(a, fs, blockIdx.x * kWarps, kWarps, NW);
  while (fs.alive > 0) {
    for (int t = gw; t < a.ntiles; t += NW) {
      const int m = find_map(fs.base, a.nmaps, t);
      const FlowMap& L = fs.loc[fs.slot[m]];
      if (L.done) continue;
      const MapDesc& M = a.maps[m];
      if (L.phase == kPhA) {
        const double dq = warp_sum(a32_tile_dq<KIND>(a, M, t, L.iter, L.beta, lane, ring));
        flow_publish(a, L, t, dq, 0.0, 0.0, lane);
      } else if (L.phase == kPhB) {
        b32_tile<KIND>(a, M, L, t, lane, reinterpret_cast<unsigned char*>(ring));
      } else {
        // the start: the tile's FP32 planes first (the residual reads only its own pixels of them)
        if (L.phase == kPhResInit) conv_tile<KIND>(a, M, t, lane);
        const bool init = L.phase == kPhResInit;
        double rs, rr, bb;
        res64_tile<KIND>(a, M, init, t, lane, rs, rr, bb);
        flow_publish(a, L, t, warp_sum(rs), warp_sum(rr), init ? warp_sum(bb) : 0.0, lane);
      }
    }
    if (!flow_step(a, fs)) return;
  }
  // maps active at the start: what the correction holds goes into phi
  for (int t = gw; t < a.ntiles; t += NW) {
    const int m = find_map(fs.base, a.nmaps, t);
    if (a.st[m].outer_active) fold_tile(a, a.maps[m], t, lane);
  }
}

int pcg32_max_blocks_per_sm(int kind) {
  int nb = 0;
  // the attribute is the function's on the current device: set here, which every plan creation passes
  const int smem = (int)sizeof(Rings32);
  if (kind == kIdentity) {
    cudaFuncSetAttribute(k_pcg32<kIdentity>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_pcg32<kIdentity>, kThreads, smem);
  } else if (kind == kJacobi) {
    cudaFuncSetAttribute(k_pcg32<kJacobi>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_pcg32<kJacobi>, kThreads, smem);
  }
  return nb;
}

cudaError_t launch_pcg32(const Plan& pl, int kind, const PcgArgs& a, cudaStream_t st, cudaEvent_t e0,
                         cudaEvent_t e1) {
  pl.kernel_launches += 2;
  pl.solver_launches += 1;
  launch_pcg_reset(pl, st, true);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (e0) cudaEventRecord(e0, st);
  const int blocks = pl.nsm * pl.bps;
  void* args[] = {(void*)&a};
  if (resident_fits(pl, false, kind))
    e = launch_resident(pl, false, kind, a, st);
  else if (kind == kIdentity)
    e = cudaLaunchCooperativeKernel((void*)k_pcg32<kIdentity>, blocks, kThreads, args, sizeof(Rings32), st);
  else if (kind == kJacobi)
    e = cudaLaunchCooperativeKernel((void*)k_pcg32<kJacobi>, blocks, kThreads, args, sizeof(Rings32), st);
  else
    e = cudaErrorInvalidValue;
  if (e == cudaSuccess && e1) e = cudaEventRecord(e1, st);
  return e;
}

}  // namespace ulp
