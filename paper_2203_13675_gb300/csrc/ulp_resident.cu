// ulp_resident.cu -- the persistent Jacobi / identity PCG with the whole working set on
// the chip, for maps (or batches) whose tiles fit one per warp in the SMs' shared memory
// and registers: up to about 0.5 Mpx in FP64, 1.2 Mpx in mixed precision.
//
// Same tiles and the same arithmetic per pixel as k_pcg64 / k_pcg32.  There a phase streams
// its planes from L2 a row at a time, and with one or two warps per SM partition each row
// costs its load latency: at 640x480 the FP64 pipe (64 cycles per warp instruction and
// partition; about 70 of them per tile in phase A, 50 in phase B) was busy for a quarter of
// an iteration.  Here a warp keeps its tile's weights, D, D^-1, phi (or
// the correction), r and s in shared memory and d and q in registers across iterations.
// What crosses tiles is the rim of s: in phase B a warp stores its first and last row and
// its two edge columns into the map's s plane (r for M = I), and in phase A it reads its
// neighbours' and advances its own copy of their rim of d by the same d = s + beta d_old.
// True residuals (start and refresh iterations) go through the global planes as in the
// streaming kernels.
//
// Sums: a block adds the lane sums of its tiles of a map (FP64, fixed order) and publishes
// one partial per sum, as ulp_flow.cuh does per tile; every block of the map reads those, at
// most one per SM.  Off the path from the last tile to the scalar: phi, which moves with
// the next phase A while the rim loads are in flight, and the fence before phase B's
// partials, which finds the rim's stores already under way (they precede the dots; phase A
// stores nothing and needs none).
//
// Measured on one GB300, us per Jacobi iteration (tile partials, finisher warp and grid
// barriers / here): FP64 256x256 33.4 / 11.8, 640x480 33.0 / 14.9, 704x704 37.7 / 23.5; mixed
// 256x256 26.3 / 10.7, 1024x1024 34.5 / 20.4, 1200x1024 36.4 / 21.7.  The streaming kernels
// with published partials take 27.8 at 640x480 (FP64) and 32.8 at 1024x1024 (mixed).  Clock
// stamps in a build made for it put half of an iteration at 640x480 into the two tile phases, a
// sixth into the blocks' sums and fences, a fifth into the trips through L2 and a tenth into
// the scalars.
//
// A map's sums are grouped by where its tiles fall among the blocks, so its last bits depend on
// the batch and the number of SMs (the streaming kernels' do not).  One partial per tile in the
// streaming kernels' order instead gives their bits and was measured at 0.87-0.95 of the speed
// in FP64, 0.77-0.93 in mixed precision: every SM then adds all of the map's tile partials at
// 64 cycles per warp of FP64 values, and polls as many lines.
#include <type_traits>

#include "ulp_flow32.cuh"
#include "ulp_host.h"
#include "ulp_parts.h"

namespace ulp {

template <typename T>
struct Vec2;
template <>
struct Vec2<double> {
  using V = double2;
  static __device__ __forceinline__ V ld(const double* p, size_t o) { return ld2(p, o); }
  static __device__ __forceinline__ void st(double* p, size_t o, V v) { st2(p, o, v); }
  static __device__ __forceinline__ V make(double x, double y) { return make_double2(x, y); }
};
template <>
struct Vec2<float> {
  using V = float2;
  static __device__ __forceinline__ V ld(const float* p, size_t o) { return ldf2(p, o); }
  static __device__ __forceinline__ void st(float* p, size_t o, V v) { stf2(p, o, v); }
  static __device__ __forceinline__ V make(float x, float y) { return make_float2(x, y); }
};

// Bytes of one warp's shared memory for tiles of R rows: planes of R rows of 64 elements
// (V one row more, for the row above), then the edge columns' weights and d (3 R elements).
__host__ __device__ constexpr size_t res_warp_bytes(bool f64, int R) {
  const size_t e = f64 ? 8 : 4;
  const int planes = f64 ? 7 : 6;  // U V D Dinv phi r s; U V Dinv x r s
  return ((size_t)(planes * R + 1) * kStrip * e + (size_t)3 * R * e + 15) / 16 * 16;
}

// Which planes a kind of solve works on.
template <typename T>
__device__ __forceinline__ const T* pl_u(const MapDesc& M);
template <> __device__ __forceinline__ const double* pl_u<double>(const MapDesc& M) { return M.f.U; }
template <> __device__ __forceinline__ const float* pl_u<float>(const MapDesc& M) { return M.h.U; }
template <typename T>
__device__ __forceinline__ const T* pl_v(const MapDesc& M);
template <> __device__ __forceinline__ const double* pl_v<double>(const MapDesc& M) { return M.f.V; }
template <> __device__ __forceinline__ const float* pl_v<float>(const MapDesc& M) { return M.h.V; }
template <typename T>
__device__ __forceinline__ const T* pl_di(const MapDesc& M);
template <> __device__ __forceinline__ const double* pl_di<double>(const MapDesc& M) { return M.f.Dinv; }
template <> __device__ __forceinline__ const float* pl_di<float>(const MapDesc& M) { return M.h.Dinv; }
template <typename T>
__device__ __forceinline__ T* pl_r(const MapDesc& M);
template <> __device__ __forceinline__ double* pl_r<double>(const MapDesc& M) { return M.f.r; }
template <> __device__ __forceinline__ float* pl_r<float>(const MapDesc& M) { return M.h.r; }
template <typename T>
__device__ __forceinline__ T* pl_s(const MapDesc& M);
template <> __device__ __forceinline__ double* pl_s<double>(const MapDesc& M) { return M.f.s; }
template <> __device__ __forceinline__ float* pl_s<float>(const MapDesc& M) { return M.h.s; }

// Sum of products: FP64 FMAs, or the double-float accumulation of the mixed solver.
struct Sum64 {
  double v = 0.0;
  __device__ __forceinline__ void add(double a, double b) { v = fma(a, b, v); }
  __device__ __forceinline__ double value() const { return v; }
};
struct Sum32 {
  DF v;
  __device__ __forceinline__ void add(float a, float b) { v.add_prod(a, b); }
  __device__ __forceinline__ double value() const { return v.value(); }
};

// One pixel of A d: FP64 as stencil_tile, FP32 as stencil_tile32 (see there for the form).
__device__ __forceinline__ double ax_px(double dd, double xc, double ue, double xe, double uw, double xw, double vs,
                                        double xs, double vn, double xn) {
  double ax = dd * xc;
  ax = fma(-ue, xe, ax);
  ax = fma(-uw, xw, ax);
  ax = fma(-vs, xs, ax);
  return fma(-vn, xn, ax);
}
__device__ __forceinline__ float ax_px(float, float xc, float ue, float xe, float uw, float xw, float vs, float xs,
                                       float vn, float xn) {
  float ax = __fmul_rn(ue, __fsub_rn(xc, xe));
  ax = __fmaf_rn(uw, __fsub_rn(xc, xw), ax);
  ax = __fmaf_rn(vn, __fsub_rn(xc, xn), ax);
  return __fmaf_rn(vs, __fsub_rn(xc, xs), ax);
}
__device__ __forceinline__ double fma_t(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float fma_t(float a, float b, float c) { return __fmaf_rn(a, b, c); }

// One tile in a warp's keeping.  RT: rows the registers hold (R <= RT).
template <typename T, int KIND, int RT>
struct ResTile {
  using V2 = Vec2<T>;
  using V = typename V2::V;
  static constexpr bool F64 = sizeof(T) == 8;
  // shared memory
  V *U, *Vv, *D, *Di, *X, *Rr, *S;  // [row][lane]; Vv has the row above first; X: phi or the correction
  T *uw, *dw, *de;                  // edge columns: U left of the tile, d left and right of it
  // registers
  V d[RT], q[RT];
  V dn, ds;  // d in the rows above and below the tile
  T dh;      // d at an edge column: lane r < R the left one of row r, lane 16 + r the right one
  bool pend; // phi (the correction) has yet to move by the last iteration's alpha d
  TileGeo g;
  int R, nrow;

  __device__ __forceinline__ void place(unsigned char* sm, int R_) {
    R = R_;
    V* p = reinterpret_cast<V*>(sm);
    auto take = [&](int rows) {
      V* r = p;
      p += rows * 32;
      return r;
    };
    U = take(R);
    Vv = take(R + 1);
    if (F64) D = take(R);
    Di = take(R);
    X = take(R);
    Rr = take(R);
    S = take(R);
    uw = reinterpret_cast<T*>(p);
    dw = uw + R;
    de = dw + R;
  }

  // The loops that run once a solve or on refresh iterations only are not unrolled: the code of
  // an iteration runs once per warp and pass, and what lies between its parts costs instruction
  // fetches.  Unrolled, builds of the same arithmetic differed by up to 9 % with the address
  // arithmetic elsewhere (600x500 FP64, 400 iterations: 5.97 to 6.51 ms; here 5.97).

  // weights, D, D^-1 (and phi) into shared memory; rows past the map are 0
  __device__ __forceinline__ void load(const MapDesc& M, int t, int lane) {
    g = tile_geo(M, t, R);
    nrow = g.i1 - g.i0;
    const int j = g.j0 + 2 * lane;
    const size_t P = M.pitch;
    const V z = V2::make(0, 0);
#pragma unroll 1
    for (int r = -1; r < R; ++r) {
      const int i = g.i0 + r;
      const bool in = i >= 0 && r < nrow;
      const size_t o = (size_t)i * P + j;
      Vv[(r + 1) * 32 + lane] = in ? V2::ld(pl_v<T>(M), o) : z;
      if (r < 0) continue;
      U[r * 32 + lane] = in ? V2::ld(pl_u<T>(M), o) : z;
      if constexpr (F64) D[r * 32 + lane] = in ? ld2(M.f.D, o) : z;
      if (KIND == kJacobi) Di[r * 32 + lane] = in ? V2::ld(pl_di<T>(M), o) : z;
      if constexpr (F64) X[r * 32 + lane] = in ? ld2(M.f.phi, o) : z;
      else X[r * 32 + lane] = z;
    }
    if (lane < R) uw[lane] = (lane < nrow && g.j0 > 0) ? __ldcg(pl_u<T>(M) + (size_t)(g.i0 + lane) * P + g.j0 - 1) : (T)0;
#pragma unroll
    for (int r = 0; r < RT; ++r) d[r] = q[r] = z;
    dn = ds = z;
    dh = (T)0;
    pend = false;
  }
  __device__ __forceinline__ void move(double alpha_, int lane) {
    const T alpha = (T)alpha_;
#pragma unroll
    for (int r = 0; r < RT; ++r) {
      if (r >= nrow) break;
      V x = X[r * 32 + lane];
      x.x = fma_t(alpha, d[r].x, x.x);
      x.y = fma_t(alpha, d[r].y, x.y);
      X[r * 32 + lane] = x;
    }
  }
  // r (and s) as the residual step left them in the planes
  __device__ __forceinline__ void load_rs(const MapDesc& M, int lane) {
    const V z = V2::make(0, 0);
#pragma unroll 1
    for (int r = 0; r < R; ++r) {
      const size_t o = (size_t)(g.i0 + r) * M.pitch + g.j0 + 2 * lane;
      Rr[r * 32 + lane] = r < nrow ? V2::ld(pl_r<T>(M), o) : z;
      if (KIND == kJacobi) S[r * 32 + lane] = r < nrow ? V2::ld(pl_s<T>(M), o) : z;
    }
  }

  __device__ __forceinline__ static V dir(T beta, bool first, V d, V s) {
    return first ? s : V2::make(fma_t(beta, d.x, s.x), fma_t(beta, d.y, s.y));
  }

  // phase A: d = s + beta d (d = s at the first iteration), q = A d; the lane's share of d^T q
  __device__ __forceinline__ double phase_a(const MapDesc& M, bool first, double beta_, double alpha, int lane) {
    const T beta = (T)beta_;
    const T* sp = KIND == kIdentity ? pl_r<T>(M) : pl_s<T>(M);
    const size_t P = M.pitch;
    const int j = g.j0 + 2 * lane;
    // the neighbours' rim of s: one round of loads
    const V z = V2::make(0, 0);
    const V sn = g.i0 > 0 ? V2::ld(sp, (size_t)(g.i0 - 1) * P + j) : z;
    const V ss = g.i1 < M.H ? V2::ld(sp, (size_t)g.i1 * P + j) : z;
    const int hr = lane & 15;
    const bool left = lane < 16;
    T sh = (T)0;
    if (hr < nrow && (left ? g.j0 > 0 : g.j0 + kStrip < M.pitch))
      sh = __ldcg(sp + (size_t)(g.i0 + hr) * P + (left ? g.j0 - 1 : g.j0 + kStrip));
    if (pend) move(alpha, lane);
    pend = false;
#pragma unroll
    for (int r = 0; r < RT; ++r)
      if (r < nrow) d[r] = dir(beta, first, d[r], (KIND == kIdentity ? Rr : S)[r * 32 + lane]);
    dn = dir(beta, first, dn, sn);
    ds = dir(beta, first, ds, ss);
    dh = first ? sh : fma_t(beta, dh, sh);
    if (hr < R) (left ? dw : de)[hr] = dh;
    __syncwarp();
    using Sum = typename std::conditional<F64, Sum64, Sum32>::type;
    Sum dq;
#pragma unroll
    for (int r = 0; r < RT; ++r) {
      if (r >= nrow) break;
      const V xc = d[r];
      const V xn = r == 0 ? dn : d[r > 0 ? r - 1 : 0];
      const V xs = r + 1 < nrow ? d[r + 1 < RT ? r + 1 : r] : ds;
      const V u = U[r * 32 + lane], v = Vv[(r + 1) * 32 + lane], vn = Vv[r * 32 + lane];
      V dd = z;
      if constexpr (F64) dd = D[r * 32 + lane];
      T west = __shfl_up_sync(kFull, xc.y, 1);
      T east = __shfl_down_sync(kFull, xc.x, 1);
      T ul = __shfl_up_sync(kFull, u.y, 1);
      if (lane == 0) {
        west = dw[r];
        ul = uw[r];
      }
      if (lane == 31) east = de[r];
      V ax;
      ax.x = ax_px(dd.x, xc.x, u.x, xc.y, ul, west, v.x, xs.x, vn.x, xn.x);
      ax.y = ax_px(dd.y, xc.y, u.y, east, u.x, xc.x, v.y, xs.y, vn.y, xn.y);
      q[r] = ax;
      dq.add(xc.x, ax.x);
      dq.add(xc.y, ax.y);
    }
    __syncwarp();  // dw, de are rewritten in the next phase A
    return dq.value();
  }

  // phase B: r -= alpha q, s = D^-1 r, the rim, then the dots; phi (the correction) follows in
  // the next phase A.  On a refresh iteration phi alone, into the map's plane, for the
  // residual that follows.
  __device__ __forceinline__ void phase_b(const MapDesc& M, double alpha_, bool refresh, int lane, double& rs,
                                          double& rr) {
    const size_t P = M.pitch;
    const int j = g.j0 + 2 * lane;
    rs = rr = 0.0;
    if (refresh) {
      move(alpha_, lane);
      finish(M, lane);
      if (!F64)
#pragma unroll 1
        for (int r = 0; r < nrow; ++r) X[r * 32 + lane] = V2::make(0, 0);
      return;
    }
    const T alpha = (T)alpha_;
    T* sp = KIND == kIdentity ? pl_r<T>(M) : pl_s<T>(M);
    V rv[RT], sv[RT];
#pragma unroll
    for (int r = 0; r < RT; ++r) {
      if (r >= nrow) break;
      V x = Rr[r * 32 + lane];
      x.x = fma_t(-alpha, q[r].x, x.x);
      x.y = fma_t(-alpha, q[r].y, x.y);
      Rr[r * 32 + lane] = rv[r] = x;
      if (KIND == kJacobi) {
        const V di = Di[r * 32 + lane];
        S[r * 32 + lane] = sv[r] = V2::make(di.x * x.x, di.y * x.y);
      }
      if (r == 0 || r == nrow - 1 || lane == 0 || lane == 31)
        V2::st(sp, (size_t)(g.i0 + r) * P + j, KIND == kIdentity ? rv[r] : sv[r]);
    }
    using Sum = typename std::conditional<F64, Sum64, Sum32>::type;
    Sum ars, arr;
#pragma unroll
    for (int r = 0; r < RT; ++r) {
      if (r >= nrow) break;
      if (KIND == kJacobi) {
        ars.add(rv[r].x, sv[r].x);
        ars.add(rv[r].y, sv[r].y);
      }
      arr.add(rv[r].x, rv[r].x);
      arr.add(rv[r].y, rv[r].y);
    }
    rr = arr.value();
    rs = KIND == kIdentity ? rr : ars.value();
    pend = true;
  }

  // end of the solve: phi from the chip (or the correction added to it)
  __device__ __forceinline__ void finish(const MapDesc& M, int lane) {
#pragma unroll 1
    for (int r = 0; r < nrow; ++r) {
      const size_t o = (size_t)(g.i0 + r) * M.pitch + g.j0 + 2 * lane;
      const V x = X[r * 32 + lane];
      if constexpr (F64) {
        st2(M.f.phi, o, x);
      } else {
        double2 ph = ld2(M.f.phi, o);
        ph.x += (double)x.x;
        ph.y += (double)x.y;
        st2(M.f.phi, o, ph);
      }
    }
  }
};

// A block's copy of one map's scalars, and the warps and blocks that share the map.
struct ResMap {
  double delta, delta0, rr, bb, alpha, beta;
  long long iter, lmax;
  int m, phase, set, done, stop_after, status, fresh;
  int refresh, left;     // true-residual period; iterations until the next one (0: this one)
  int w0, w1;            // the block's warps on the map
  int slot, nslot;       // first slot of the map's partials, how many blocks publish
};

struct ResShared {
  ResMap loc[kResMaxWarps];             // a block's tiles lie in at most that many maps
  MapDesc map[kResMaxWarps];
  double red[3][kResMaxWarps][32];      // lane sums of each warp's tile
  double part[kPartSlots][4];           // each map's and sum's own slot (ulp_parts.h)
  double sum[3];
  int n, alive, fail;
};

// The maps of the block's tiles [first, first + count) and their start state.
__device__ __forceinline__ void res_begin(const PcgArgs& a, ResShared& sh, int per_block) {
  if (threadIdx.x == 0) {
    const int first = blockIdx.x * per_block, last = min(first + per_block, a.ntiles);
    int n = 0, alive = 0;
    for (int m = 0; m < a.nmaps; ++m) {
      const int b0 = a.maps[m].tile_base, b1 = b0 + a.maps[m].ntiles;
      if (b1 <= first || b0 >= last) continue;
      ResMap& L = sh.loc[n];
      L = ResMap{};
      sh.map[n] = a.maps[m];
      L.m = m;
      L.phase = kPhResInit;
      L.done = a.st[m].done;
      L.refresh = sh.map[n].refresh;
      L.lmax = a.lmax > 0 ? a.lmax : 2LL * sh.map[n].H * sh.map[n].W;
      L.w0 = max(b0 - first, 0);
      L.w1 = min(b1, last) - first;
      // block b's partial of map m has slot b + m: consecutive for the blocks of a map
      L.slot = b0 / per_block + m;
      L.nslot = (b1 - 1) / per_block - b0 / per_block + 1;
      ++n;
      if (!L.done) ++alive;
    }
    sh.n = n;
    sh.alive = alive;
    sh.fail = 0;
  }
  __syncthreads();
}

// The block's sum q over its tiles of the map at place i (128 threads, r = 0 .. 127: warp k
// adds tiles k, k + 4, ... lane by lane and its lanes as a tree), published.
__device__ __forceinline__ void res_publish(const PcgArgs& a, ResShared& sh, const ResMap& L, int i, int q, int r,
                                            double* slots, double* clear) {
  const int lane = r & 31, k = r >> 5;
  double s = 0.0;
  for (int w = L.w0 + k; w < L.w1; w += 4) s += sh.red[q][w][lane];
  s = warp_sum(s);
  double* p = sh.part[part_slot(i, q)];
  if (lane == 0) p[k] = s;
  asm volatile("bar.sync %0, 128;" ::"r"((q & 1) + 1) : "memory");
  if (r == 0) {
    s = (p[0] + p[1]) + (p[2] + p[3]);
    if (clear) st_relaxed(clear + blockIdx.x + L.m, sentinel());
    if (L.phase != kPhA) __threadfence();  // the rim (or the planes) of the block's tiles first
    st_relaxed(slots + blockIdx.x + L.m, s);
  }
}

// One warp: waits for every block's partial and adds them (lane l: l, l + 32, ..., then a tree).
__device__ __forceinline__ bool res_collect(const PcgArgs& a, const ResMap& L, const double* slots, int lane,
                                            double* sum) {
  constexpr int K = 5;  // 160 slots in one round of loads
  double s = 0.0;
  bool ok = true;
  const unsigned long long t_in = globaltimer();
  for (int k0 = 0; k0 < L.nslot; k0 += 32 * K) {
    double v[K];
#pragma unroll
    for (int u = 0; u < K; ++u) {
      const int k = k0 + 32 * u + lane;
      v[u] = k < L.nslot ? ld_relaxed(slots + L.slot + k) : 0.0;
    }
    for (;;) {
      bool again = false;
#pragma unroll
      for (int u = 0; u < K; ++u) {
        if (is_sentinel(v[u])) {
          v[u] = ld_relaxed(slots + L.slot + k0 + 32 * u + lane);
          again |= is_sentinel(v[u]);
        }
      }
      if (!again) break;
      if (globaltimer() - t_in > a.timeout_ns) atomicExch(&a.bar->err, 1);
      if (*(volatile int*)&a.bar->err) {
        ok = false;
        break;
      }
    }
#pragma unroll
    for (int u = 0; u < K; ++u) s += v[u];
  }
  // the bound is on the whole wait, so values that were there at the first look count too
  if (lane == 31 && globaltimer() - t_in > a.timeout_ns) {
    atomicExch(&a.bar->err, 1);
    ok = false;
  }
  s = warp_sum(s);
  if (lane == 0) *sum = s;
  return ok;
}

// Algorithm 1's scalars of one map after a phase (one thread).
__device__ __forceinline__ void res_advance(const PcgArgs& a, ResMap& L, const double* sum) {
  const int ph = L.phase;
  L.set = (L.set + 1) & 3;
  L.fresh = ph == kPhResInit || ph == kPhRes;
  if (ph == kPhA) {
    const double dq = sum[0];
    L.phase = kPhB;
    if (!(dq > 0.0) || !isfinite(dq)) {  // breakdown: stop after this iteration
      L.status = -3;
      L.alpha = 0.0;
      L.stop_after = 1;
    } else {
      L.alpha = L.delta / dq;
    }
    return;
  }
  if (ph == kPhB && L.left == 0) {
    L.phase = kPhRes;  // phi is complete: the true residual follows
    return;
  }
  if (ph == kPhResInit) {
    L.delta = L.delta0 = sum[0];
    L.bb = sum[2];
  } else {
    const double dold = L.delta;
    L.delta = sum[0];
    L.beta = sum[0] / dold;
    L.iter += 1;
    L.left = (L.left == 0 ? L.refresh : L.left) - 1;
  }
  L.rr = sum[1];
  L.phase = kPhA;
  const bool conv = (a.stop_mode == 1) ? !(L.delta > a.tol2 * L.delta0) : !(L.rr > a.tol2 * L.bb);
  if (L.stop_after) {
    L.done = 1;
  } else if (L.bb == 0.0 || conv) {
    L.done = 1;
    L.status = 0;
  } else if (L.iter >= L.lmax) {
    L.done = 1;
    L.status = 1;
  }
}

// Ends a phase of every map of the block: publishes, waits, advances.  False (in every
// thread) if a wait ran out.
__device__ __forceinline__ bool res_step(const PcgArgs& a, ResShared& sh) {
  const int q = threadIdx.x >> 7, r = threadIdx.x & 127, lane = threadIdx.x & 31;
  const size_t N = a.nflow;
  auto slots = [&](int set, int qq) { return a.flow + (size_t)(2 * set + qq) * N; };
  __syncthreads();
  // every map's partials go out before the block waits for any map
  for (int i = 0; i < sh.n; ++i) {
    const ResMap& L = sh.loc[i];
    const int cnt = L.phase == kPhA ? 1 : 2;
    if (L.done) continue;
    // the set of the phase after next gets its sentinels back: its values are those of two
    // phases ago, which every block has read; they are behind this phase's fence or, in
    // phase A, the next one's
    const int clear = (L.set + 2) & 3;
    if (q < cnt) res_publish(a, sh, L, i, q, r, slots(L.set, q), slots(clear, q));
    if (q == 0 && L.phase == kPhResInit) res_publish(a, sh, L, i, 2, r, a.flow + 8 * N, nullptr);
    if (q == 1 && cnt == 1 && r == 0) st_relaxed(slots(clear, 1) + blockIdx.x + L.m, sentinel());
  }
  for (int i = 0; i < sh.n; ++i) {
    ResMap& L = sh.loc[i];
    if (L.done) continue;
    const int cnt = L.phase == kPhA ? 1 : 2;
    bool ok = true;
    if (q < cnt && r < 32) {
      ok = res_collect(a, L, slots(L.set, q), lane, &sh.sum[q]);
      if (q == 0 && L.phase == kPhResInit) ok &= res_collect(a, L, a.flow + 8 * N, lane, &sh.sum[2]);
      __threadfence();  // the phase's stores behind the partials just read
    }
    if (!ok) sh.fail = 1;
    __syncthreads();
    if (sh.fail) return false;
    if (threadIdx.x == 0) {
      res_advance(a, L, sh.sum);
      if (L.done) {
        sh.alive -= 1;
        if (L.slot == (int)blockIdx.x + L.m) {  // the block of the map's first tile reports its end
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
    __syncthreads();
  }
  return true;
}

// The true residual of a tile, out of line: it is rare and its registers are not the loop's.
template <typename T, int KIND>
__device__ __noinline__ void res_residual(const PcgArgs& a, const MapDesc& M, bool init, int t, int lane, double* v) {
  if constexpr (sizeof(T) == 8) {
    res_tile<KIND>(a, M, init, t, lane, v[0], v[1], v[2]);
  } else {
    if (init) conv_tile<KIND>(a, M, t, lane);  // (the residual reads only its own pixels of these planes)
    res64_tile<KIND>(a, M, init, t, lane, v[0], v[1], v[2]);
  }
}

// MAXW: warps per block, 8 (up to 255 registers a thread) or 16.
template <typename T, int KIND, int RT, int MAXW>
__global__ void __launch_bounds__(MAXW * 32, 1) k_pcg_res(PcgArgs a, int per_block) {
  extern __shared__ __align__(16) unsigned char res_dsm[];
  __shared__ ResShared sh;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  res_begin(a, sh, per_block);
  const int t = blockIdx.x * per_block + warp;
  int i = 0;
  while (i + 1 < sh.n && warp >= sh.loc[i].w1) ++i;
  ResMap& L = sh.loc[i];
  const MapDesc& M = sh.map[i];
  const bool active = warp < sh.loc[sh.n - 1].w1 && !L.done;
  ResTile<T, KIND, RT> tile;
  if (active) tile.place(res_dsm + (size_t)warp * res_warp_bytes(sizeof(T) == 8, a.R), a.R);
  bool loaded = false;
  while (sh.alive > 0) {
    if (active && !L.done) {
      double v[3] = {0.0, 0.0, 0.0};
      if (L.phase == kPhA) {
        if (!loaded) tile.load(M, t, lane);  // every tile's planes are there: the start has been published
        loaded = true;
        if (L.fresh) tile.load_rs(M, lane);
        v[0] = tile.phase_a(M, L.iter == 0, L.beta, L.alpha, lane);
      } else if (L.phase == kPhB) {
        tile.phase_b(M, L.alpha, L.left == 0, lane, v[0], v[1]);
      } else {
        res_residual<T, KIND>(a, M, L.phase == kPhResInit, t, lane, v);
      }
      sh.red[0][warp][lane] = v[0];
      if (L.phase != kPhA) sh.red[1][warp][lane] = v[1];
      if (L.phase == kPhResInit) sh.red[2][warp][lane] = v[2];
    }
    if (!res_step(a, sh)) return;
  }
  if (active && loaded) {
    if (tile.pend) tile.move(L.alpha, lane);
    tile.finish(M, lane);
  }
}

// ------------------------------------------------------------------ host side
template <typename T, int KIND>
static const void* res_kernel(int R, int warps) {
  const bool small = warps <= kWarps;
  if (R <= 4)
    return small ? (const void*)k_pcg_res<T, KIND, 4, kWarps> : (const void*)k_pcg_res<T, KIND, 4, kResMaxWarps>;
  if constexpr (sizeof(T) == 4) {
    if (R <= 6) return (const void*)k_pcg_res<T, KIND, 6, kResMaxWarps>;
    if (R <= 8) return (const void*)k_pcg_res<T, KIND, 8, kResMaxWarps>;
  }
  return nullptr;
}
static const void* res_kernel(bool f64, int kind, int R, int warps) {
  if (f64) return kind == kIdentity ? res_kernel<double, kIdentity>(R, warps) : res_kernel<double, kJacobi>(R, warps);
  return kind == kIdentity ? res_kernel<float, kIdentity>(R, warps) : res_kernel<float, kJacobi>(R, warps);
}

// Shared memory a block may ask for beside its ResShared (227 KB per block on sm_103a).
constexpr size_t kResSmem = 232448 - (sizeof(ResShared) + 1024);

void resident_attrs() {
  for (int f64 = 0; f64 < 2; ++f64)
    for (int kind : {(int)kIdentity, (int)kJacobi})
      for (int R : {4, 6, 8})
        for (int warps : {kWarps, kResMaxWarps})
          if (const void* k = res_kernel(f64, kind, R, warps))
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kResSmem);
}

// One tile per warp, spread over all SMs: the resident form runs wherever the tiles fit
// (see the head of the file for both sides' times).
bool resident_fits(const Plan& pl, bool f64, int kind) {
  if (kind != kIdentity && kind != kJacobi) return false;
  if (!res_kernel(f64, kind, pl.R, kResMaxWarps)) return false;
  const int per_block = (pl.ntiles + pl.nsm - 1) / pl.nsm;
  return per_block <= kResMaxWarps && (size_t)per_block * res_warp_bytes(f64, pl.R) <= kResSmem;
}

cudaError_t launch_resident(const Plan& pl, bool f64, int kind, const PcgArgs& a, cudaStream_t st) {
  int per_block = (pl.ntiles + pl.nsm - 1) / pl.nsm;
  const int blocks = (pl.ntiles + per_block - 1) / per_block;
  // (the kernels of more than four rows a tile are built for 16 warps only)
  const int threads = per_block <= kWarps && pl.R <= 4 ? kThreads : kResMaxWarps * 32;
  void* args[] = {(void*)&a, (void*)&per_block};
  return cudaLaunchCooperativeKernel(res_kernel(f64, kind, pl.R, threads / 32), blocks, threads, args,
                                     (size_t)per_block * res_warp_bytes(f64, pl.R), st);
}

}  // namespace ulp
