// ulp_flow.cuh -- reductions of the persistent PCG kernels without a grid barrier.
//
// Algorithm 1 needs two dot products per iteration before any block may go on (alpha from
// d^T q, beta from r^T s), so on maps of up to a few megapixels the solve's time is the
// path from the last tile's partial sum to the scalar in every block.  Here each tile
// publishes its partial sums as values that are their own flags (the slot holds a
// signalling-NaN sentinel until the value lands), and every block that owns tiles of the
// map reads all of the map's partials itself, adds them in one fixed order and advances
// its own copy of the map's scalars: one trip through L2 per phase, no atomic, no elected
// last block, no barrier.  Having read every tile's partial of a phase also tells a block
// that all tiles have finished it (each publishes after a fence behind its stores), which
// orders the planes between phases; blocks that share no map never wait for one another,
// and a block whose maps have all stopped leaves.
//
// Slots: three sets used in turn.  Publishing phase n, a tile puts the sentinel back into
// set n + 1: its values there are those of phase n - 2, which every block has read, since
// every block has published n - 1.
//
// Against counters, an elected finisher warp and a grid barrier per phase, on one GB300, us
// per Jacobi iteration (before / here): FP64 640x480 33.5 / 27.8, 1024x1024 48.6 / 46.8,
// 2048x2048 126.8 / 125.6; mixed 1024x1024 34.3 / 32.8, 2048x2048 68.0 / 66.2.  Maps that fit
// the chip go on from there (ulp_resident.cu).
#pragma once
#include "ulp_engine.cuh"
#include "ulp_sweep.cuh"

namespace ulp {

// A block's copy of one map's scalars.
struct FlowMap {
  double delta, delta0, rr, bb, alpha, beta;
  long long iter;
  int m, phase, set, done, stop_after, status, report;
};

struct FlowShared {
  int base[kMaxMaps + 1];             // first tile of each map
  unsigned char slot[kMaxMaps];       // a touched map's place in loc
  FlowMap loc[kMaxMaps];              // the maps this block owns tiles of
  double part[2][kArriveGroups];
  double sum[3];
  int n, alive, fail;
};

__device__ __forceinline__ double* flow_slots(const PcgArgs& a, int set, int q) {
  return a.flow + (size_t)(2 * set + q) * a.nflow;
}
// the third sum of a solve's start (b^T b) has slots of its own
__device__ __forceinline__ double* flow_slots_bb(const PcgArgs& a) { return a.flow + (size_t)6 * a.nflow; }

// The maps of this block's tiles (count tiles from first, and again every stride) and their
// start state; the block of a map's first tile reports the map's end.  All threads.
__device__ __forceinline__ void flow_begin(const PcgArgs& a, FlowShared& fs, int first, int count, int stride) {
  for (int m = threadIdx.x; m <= a.nmaps; m += blockDim.x)
    fs.base[m] = (m < a.nmaps) ? a.maps[m].tile_base : a.ntiles;
  __syncthreads();
  if (threadIdx.x == 0) {
    int n = 0, alive = 0;
    for (int m = 0; m < a.nmaps; ++m) {
      const int b0 = fs.base[m], b1 = fs.base[m + 1];
      bool mine = false, owner = false;
      for (int t = first; t < b1; t += stride) {
        mine |= t + count > b0;
        owner |= t <= b0 && t + count > b0;
      }
      if (!mine) continue;
      FlowMap& L = fs.loc[n];
      L = FlowMap{};
      L.m = m;
      L.phase = kPhResInit;
      L.done = a.st[m].done;
      L.report = owner;
      fs.slot[m] = (unsigned char)n++;
      if (!L.done) ++alive;
    }
    fs.n = n;
    fs.alive = alive;
    fs.fail = 0;
  }
  __syncthreads();
}

// Tile t's partial sums of the map's current phase (lane sums already added over the warp).
__device__ __forceinline__ void flow_publish(const PcgArgs& a, const FlowMap& L, int t, double v0, double v1,
                                             double v2, int lane) {
  __syncwarp();
  if (lane == 0) {
    const int next = L.set == 2 ? 0 : L.set + 1;
    st_relaxed(flow_slots(a, next, 0) + t, sentinel());
    st_relaxed(flow_slots(a, next, 1) + t, sentinel());
    __threadfence();
    st_relaxed(flow_slots(a, L.set, 0) + t, v0);
    st_relaxed(flow_slots(a, L.set, 1) + t, v1);
    if (L.phase == kPhResInit) st_relaxed(flow_slots_bb(a) + t, v2);
  }
}

// group_sums of slots that may still hold the sentinel; false if the wait ran out.
__device__ __forceinline__ bool flow_group_sums(const double* P, int n, int r, double* part,
                                                unsigned long long timeout_ns, int* err) {
  const GroupLane t(r);
  double acc[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) acc[q] = 0.0;
  bool ok = true;
  unsigned long long t_start = 0;
  for (int k = 0; t.first(k) < n; ++k) {
    double v[8];
    bool again = false;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int i = t.first(k) + 4 * kArriveGroups * q;
      v[q] = i < n ? ld_relaxed(P + i) : 0.0;
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) again |= is_sentinel(v[q]);
    if (again && t_start == 0) t_start = globaltimer();
    while (again && ok) {
      again = false;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (is_sentinel(v[q])) {
          v[q] = ld_relaxed(P + t.first(k) + 4 * kArriveGroups * q);
          again |= is_sentinel(v[q]);
        }
      }
      if (globaltimer() - t_start > timeout_ns) {
        atomicExch(err, 1);
        ok = false;
      } else if (*(volatile int*)err) {
        ok = false;
      }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) acc[q] += v[q];
  }
  group_tree(t, acc, part);
  return ok;
}

// Algorithm 1's scalars of one map after a phase (one thread): alpha = delta / d^T q, or
// delta, beta, the iteration count and the stop tests.
__device__ __forceinline__ void flow_advance(const PcgArgs& a, const MapDesc& M, FlowMap& L, const double* sum) {
  const int ph = L.phase;
  bool tests = false;
  if (ph == kPhA) {
    const double dq = sum[0];
    if (!(dq > 0.0) || !isfinite(dq)) {  // breakdown: stop after this iteration
      L.status = -3;
      L.alpha = 0.0;
      L.stop_after = 1;
    } else {
      L.alpha = L.delta / dq;
    }
    L.phase = kPhB;
  } else if (ph == kPhB && (L.iter % M.refresh) == 0) {
    L.phase = kPhRes;  // phi is complete: the true residual follows
  } else {
    if (ph == kPhResInit) {
      L.delta = L.delta0 = sum[0];
      L.bb = sum[2];
    } else {
      const double dold = L.delta;
      L.delta = sum[0];
      L.beta = sum[0] / dold;
      L.iter += 1;
    }
    L.rr = sum[1];
    L.phase = kPhA;
    tests = true;
  }
  L.set = L.set == 2 ? 0 : L.set + 1;
  if (!tests) return;
  const bool conv = (a.stop_mode == 1) ? !(L.delta > a.tol2 * L.delta0) : !(L.rr > a.tol2 * L.bb);
  if (L.stop_after) {
    L.done = 1;
  } else if (L.bb == 0.0 || conv) {
    L.done = 1;
    L.status = 0;
  } else if (L.iter >= (a.lmax > 0 ? a.lmax : 2LL * M.H * M.W)) {
    L.done = 1;
    L.status = 1;
  }
}

// After a block's tiles have published a phase of every map of its list: waits for the
// maps' other tiles, sums and advances.  False (in every thread) if a wait ran out.
__device__ __forceinline__ bool flow_step(const PcgArgs& a, FlowShared& fs) {
  const int q = threadIdx.x >> 7, r = threadIdx.x & 127, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  for (int i = 0; i < fs.n; ++i) {
    FlowMap& L = fs.loc[i];
    if (L.done) continue;
    const MapDesc& M = a.maps[L.m];
    const int cnt = L.phase == kPhA ? 1 : (L.phase == kPhResInit ? 3 : 2);
    bool ok = true;
    const bool clock = threadIdx.x == blockDim.x - 1;
    const unsigned long long t_in = clock ? globaltimer() : 0;
    if (q < cnt && q < 2)
      ok = flow_group_sums(flow_slots(a, L.set, q) + M.tile_base, M.ntiles, r, fs.part[q], a.timeout_ns, &a.bar->err);
    if (!ok) fs.fail = 1;
    __threadfence();  // the phase's stores behind the partials just read
    __syncthreads();
    // the bound is on the whole wait, so values that were there at the first look count too
    if (clock && globaltimer() - t_in > a.timeout_ns) {
      atomicExch(&a.bar->err, 1);
      fs.fail = 1;
    }
    if (warp < cnt && warp < 2) {
      const double v = warp_sum(fs.part[warp][lane]);
      if (lane == 0) fs.sum[warp] = v;
    }
    if (cnt == 3) {  // the start of a solve
      __syncthreads();
      if (q == 0)
        ok = flow_group_sums(flow_slots_bb(a) + M.tile_base, M.ntiles, r, fs.part[0], a.timeout_ns, &a.bar->err);
      if (!ok) fs.fail = 1;
      __syncthreads();
      if (warp == 0) {
        const double v = warp_sum(fs.part[0][lane]);
        if (lane == 0) fs.sum[2] = v;
      }
    }
    __syncthreads();
    if (fs.fail) return false;
    if (threadIdx.x == 0) {
      flow_advance(a, M, L, fs.sum);
      if (L.done) {
        fs.alive -= 1;
        if (L.report) {
          MapState* S = a.st + L.m;
          S->delta = L.delta;
          S->rr = L.rr;
          S->bb = L.bb;
          S->relres = (L.bb > 0.0) ? sqrt(L.rr / L.bb) : 0.0;
          S->iter = L.iter;
          S->status = L.status;
          S->done = 1;
          atomicSub(a.n_active, 1);
        }
      }
    }
    // the verdict has been read by every thread before a wait for the next map may change it
    __syncthreads();
  }
  return true;
}

// r = b - A phi, s = M^{-1} r; the lane's shares of r^T s, r^T r (and b^T b at the start).
template <int KIND>
__device__ __forceinline__ void res_tile(const PcgArgs& a, const MapDesc& M, bool init, int t, int lane, double& rs,
                                         double& rr, double& bb) {
  const TileGeo g = tile_geo(M, t, a.R);
  const size_t P = M.pitch;
  XPlane x{M.f.phi, P};
  rs = rr = bb = 0.0;
  auto epi = [&](size_t off, double2 xc, double2 ax) {
    const double2 bv = ld2(M.f.b, off);
    double2 r = make_double2(bv.x - ax.x, bv.y - ax.y);
    st2(M.f.r, off, r);
    if (KIND == kJacobi) {
      const double2 di = ld2(M.f.Dinv, off);
      const double2 s = make_double2(di.x * r.x, di.y * r.y);
      st2(M.f.s, off, s);
      rs = fma(r.x, s.x, rs);
      rs = fma(r.y, s.y, rs);
    }
    rr = fma(r.x, r.x, rr);
    rr = fma(r.y, r.y, rr);
    if (init) {
      bb = fma(bv.x, bv.x, bb);
      bb = fma(bv.y, bv.y, bb);
    }
  };
  stencil_tile(M, g.i0, g.i1, g.j0, lane, M.f.U, M.f.V, M.f.D, x, epi);
  if (KIND == kIdentity) rs = rr;
}

}  // namespace ulp
