// ulp_sweep.cuh -- wavefront triangular sweeps for the no-fill preconditioners
// (Sec. 2 list items 3-5: ILU(0), IC(0), SOR read as SSOR) in natural
// row-major order.
//
// For the symmetric 5-point A with strict lower part L (entries -U_{i,j-1},
// -V_{i-1,j}) all three have the form M = c (P + L) P^-1 (P + L^T):
//   ILU(0) = IC(0): P = pivots p_k = a_kk - U_{i,j-1}^2/p_{k-1} - V_{i-1,j}^2/p_{k-W}, c = 1
//   SSOR(omega):     P = D / omega,                                      c = omega/(2-omega)
// so s = M^-1 r is a forward sweep z_k = (r_k/c + U_{i,j-1} z_{k-1} + V_{i-1,j} z_{k-W}) / P_k
// and a backward sweep s_k = z_k + (U_{i,j} s_{k+1} + V_{i,j} s_{k+W}) / P_k.
// With pinv = 1/P and the coefficient planes cw = U_{i,j-1} pinv, cn = V_{i-1,j} pinv,
// ce = U_{i,j} pinv, cs = V_{i,j} pinv precomputed, each sweep step is two
// dependent FMAs: out = fma(c2, v_nb, fma(c1, v_prev, a)).
//
// Work decomposition: a band is 32 rows, one row per lane of its computing warp; lane i
// runs one column behind lane i-1 (forward) or lane i+1 (backward), so the
// neighbour row's value for the same column arrives by a shuffle of the
// previous step.  Band b needs the last row of band b-1 (forward) or the first
// row of band b+1 (backward).  The producing band writes that row a second
// time into an exchange row that holds a signalling-NaN sentinel until the
// value lands, so the value itself is the flag: the consuming band re-reads
// values that still hold the sentinel (with a time limit) and puts the sentinel
// back after use.
//
// What bounds it: the serial chain of W + H steps or so, each two dependent FP64 FMAs
// (64 cycles each on GB300, the pipe's issue rate for a whole warp) and a shuffle.  Lane
// i works on column t - i, so loads straight from the planes touch 32 rows for 8 bytes
// each and sit between the steps of the in-order warp.  Here the computing warp does
// nothing but the chain, on operands in shared memory, and a helper warp beside it moves
// the data: rows stream through a ring of kSweepCols columns, filled by cp.async in
// aligned chunks of 8 columns x 32 rows (16-byte copies) three chunks ahead; a step
// writes its result over the operand it consumed, and finished chunks leave the ring as
// 16-byte stores; the helper also waits on the exchange row, a block of 8 steps ahead.
// A ring row is kSweepCols + 2 doubles: 16-byte rows, conflict-free along the diagonal.
// Measured on a band of its own: 223 cycles per step (305 when the computing warp also runs
// the copies), and 48 steps from a band's start to the next one's.  Against one warp per
// band with every lane loading and storing the planes itself, an SSOR iteration on 320x240
// went from 437 to 176 us and an ILU(0) iteration on 480x360 from 690 to 257 us, the same
// values bit for bit.  Four bands run on an SM at a time instead of up to sixteen, and batches
// of more bands than that gain all the same, ms a call: 64 maps of 256x256 (512 bands) 20.4 ->
// 11.9, 64 of 512x512 (1024) 31.5 -> 21.6, 64 of 1024x1024 (2048) 56.9 -> 44.7; one map of 20011
// rows (626 bands) 240 -> 61.
#pragma once
#include <type_traits>

#include "ulp_internal.cuh"

namespace ulp {

constexpr unsigned long long kSentinelBits = 0x7ff4dead5eed0001ull;  // a NaN no arithmetic produces

__device__ __forceinline__ double sentinel() { return __longlong_as_double((long long)kSentinelBits); }
__device__ __forceinline__ bool is_sentinel(double v) {
  return (unsigned long long)__double_as_longlong(v) == kSentinelBits;
}
__device__ __forceinline__ double ld_relaxed(const double* p) {
  double v;
  asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed(double* p, double v) {
  asm volatile("st.relaxed.gpu.global.f64 [%0], %1;" ::"l"(p), "d"(v) : "memory");
}

enum SweepMode { kSweepFwd = 0, kSweepBwd = 1, kSweepPiv = 2 };

struct SweepIO {
  const double* a;   // FWD: r pinv / c    BWD: z      PIV: D
  const double* b;   // FWD: cw            BWD: ce     PIV: U (read at j-1)
  const double* c;   // FWD: cn            BWD: cs     PIV: V (read at i-1)
  double* out;       // FWD: z             BWD: s      PIV: pinv
  double* xin;       // exchange row of the neighbour band (read, then reset), or null
  double* xout;      // this band's exchange row for its neighbour (written), or null
};

constexpr int kSweepCols = 64;                 // ring columns (a power of two)
constexpr int kSweepLd = kSweepCols + 2;       // row stride in doubles
constexpr int kSweepChunk = 8;                 // columns per chunk, steps per block
constexpr int kSweepLead = 3;                  // chunks in flight ahead of the leading lane
constexpr int kSweepPlane = 32 * kSweepLd;     // doubles of one operand's ring
constexpr int kSweepPairs = kWarps / 2;        // (computing, helper) warps per block, one computing warp per SM partition

// A pair's shared memory: the rings of the three operands (the first one's columns turn
// into the results), the exchange values of two blocks of steps, and the helper's verdict.
struct SweepSmem {
  double a[kSweepPlane], b[kSweepPlane], c[kSweepPlane];
  double x[2][kSweepChunk];
  int fail, pad_[3];
};
constexpr size_t kSweepSmem = kSweepPairs * sizeof(SweepSmem);  // 203,328 bytes

// Geometry of one band, shared by the two roles.
template <int MODE>
struct SweepBand {
  static constexpr bool FWD = (MODE != kSweepBwd);
  static constexpr int PB = kSweepChunk;
  int W, row0, nrows, nch, Wt, nb;
  __device__ __forceinline__ SweepBand(const MapDesc& M, int band) {
    W = M.W;
    row0 = band * 32;
    nrows = min(32, M.H - row0);
    nch = (W + PB - 1) / PB;              // chunks, in the order of travel
    // backward the travel starts at the last column of the last chunk, so that blocks of
    // steps and chunks of columns coincide; the planes are 0 beyond column W - 1
    Wt = FWD ? W : nch * PB;
    nb = (Wt + nrows - 1 + PB - 1) / PB;  // blocks of steps
  }
};

__device__ __forceinline__ void sweep_pair_sync(int pair) {
  asm volatile("bar.sync %0, 64;" ::"r"(pair + 1) : "memory");
}
__device__ __forceinline__ void sweep_cpa16(void* sdst, const void* gsrc, int bytes) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(sdst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sa), "l"(gsrc), "r"(bytes) : "memory");
}

// The pair's barrier number b (0 .. nb) separates block b - 1 of the steps from block b:
// before it the helper has landed chunks up to b + 1 and the exchange values of block b.
// Lane l is at column index t - skew in the order of travel, so before block b every row
// is past index 8 b - 32: chunk b - 5 is complete and leaves, and its ring columns take
// chunk b + 3.
template <int MODE>
__device__ bool sweep_helper(const MapDesc& M, int band, int lane, const SweepIO& io, SweepSmem& sm, int pair,
                             unsigned long long timeout_ns, int* err) {
  const SweepBand<MODE> g(M, band);
  constexpr bool FWD = SweepBand<MODE>::FWD;
  constexpr int PB = kSweepChunk;
  const size_t P = (size_t)M.pitch;
  // a chunk's copies: 4 lanes per row (two columns each), 8 rows per instruction
  const int lr = lane >> 2, lc = 2 * (lane & 3);
  auto chunk_col = [&](int n) { return PB * (FWD ? n : g.nch - 1 - n) + lc; };
  auto issue = [&](int n) {
    if (n < g.nch) {
      const int j = chunk_col(n);  // j + 1 < pitch: the planes are padded to 64 columns
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int r = lr + 8 * q;
        const bool in = r < g.nrows;
        const int row = in ? g.row0 + r : g.row0;
        const size_t off = (size_t)row * P + j;
        const int so = r * kSweepLd + (j & (kSweepCols - 1));
        sweep_cpa16(sm.a + so, io.a + off, in ? 16 : 0);
        sweep_cpa16(sm.b + so, io.b + off, in ? 16 : 0);
        // the pivots read V of the row above (none above row 0)
        const bool inc = MODE == kSweepPiv ? in && row > 0 : in;
        sweep_cpa16(sm.c + so, io.c + (inc ? (MODE == kSweepPiv ? off - P : off) : 0), inc ? 16 : 0);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // results of chunk n (complete in every row) from the ring to the plane
  auto flush = [&](int n) {
    if (n < 0 || n >= g.nch) return;
    const int j = chunk_col(n);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int r = lr + 8 * q;
      if (r < g.nrows && j < g.W) {
        const double2 v = *reinterpret_cast<const double2*>(sm.a + r * kSweepLd + (j & (kSweepCols - 1)));
        double* o = io.out + (size_t)(g.row0 + r) * P + j;
        if (j + 1 < g.W) __stcg(reinterpret_cast<double2*>(o), v);
        else __stcg(o, v.x);
      }
    }
  };
  // the exchange values of block b (lane l < 8: the edge row's column of step 8 b + l)
  auto exchange = [&](int b) -> bool {
    bool ok = true;
    if (lane < PB) {
      const int j = FWD ? b * PB + lane : g.Wt - 1 - (b * PB + lane);
      double v = 0.0;
      if (io.xin && j >= 0 && j < g.W) {
        v = ld_relaxed(io.xin + j);
        if (is_sentinel(v)) {
          const unsigned long long t_start = globaltimer();
          do {
            if (*(volatile int*)err) { ok = false; break; }
            if (globaltimer() - t_start > timeout_ns) {
              atomicExch(err, 1);
              ok = false;
              break;
            }
            v = ld_relaxed(io.xin + j);
          } while (is_sentinel(v));
        }
        st_relaxed(io.xin + j, sentinel());
      }
      sm.x[b & 1][lane] = v;
    }
    return __all_sync(kFull, ok);
  };

  if (lane == 0) sm.fail = 0;
#pragma unroll
  for (int n = 0; n < kSweepLead; ++n) issue(n);
  bool ok = exchange(0);
  for (int b = 0;; ++b) {
    if (!ok && lane == 0) sm.fail = 1;
    // all but the newest chunk have landed: up to b + 1
    asm volatile("cp.async.wait_group %0;" ::"n"(kSweepLead - 2) : "memory");
    __syncwarp();
    sweep_pair_sync(pair);  // barrier b
    if (!ok || b == g.nb) break;
    flush(b - 5);
    __syncwarp();
    issue(b + kSweepLead);
    if (b + 1 < g.nb) ok = exchange(b + 1);
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  if (!ok) return false;
  for (int n = g.nb > 5 ? g.nb - 5 : 0; n < g.nch; ++n) flush(n);
  __syncwarp();  // every lane is done with the rings before the pair's next band refills them
  return true;
}

template <int MODE>
__device__ bool sweep_compute(const MapDesc& M, int band, int lane, const SweepIO& io, SweepSmem& sm, int pair) {
  const SweepBand<MODE> g(M, band);
  constexpr bool FWD = SweepBand<MODE>::FWD;
  constexpr int PB = kSweepChunk;
  constexpr int PF = PB / 2;                             // steps whose operands are fetched together
  const int edge = FWD ? 0 : g.nrows - 1;                // lane that consumes the neighbour's row
  const int pub = FWD ? g.nrows - 1 : 0;                 // lane whose row the neighbour consumes
  const bool publish = io.xout != nullptr && lane == pub;
  const int skew = FWD ? lane : (lane < g.nrows ? g.nrows - 1 - lane : 0);  // steps behind the leading lane
  double* sa = sm.a + lane * kSweepLd;
  const double* sb = sm.b + lane * kSweepLd;
  const double* sc = sm.c + lane * kSweepLd;
  // column of step t, before the check that it lies in the grid
  auto col = [&](int t) { return FWD ? t - skew : g.Wt - 1 - (t - skew); };
  // operands of the PF steps from t0 (columns outside the grid: whatever the ring holds)
  auto fetch = [&](int t0, double* va, double* vb, double* vc) {
#pragma unroll
    for (int k = 0; k < PF; ++k) {
      const int j = col(t0 + k) & (kSweepCols - 1);
      va[k] = sa[j];
      vb[k] = sb[MODE == kSweepPiv ? (j - 1) & (kSweepCols - 1) : j];
      vc[k] = sc[j];
    }
  };
  double prev = 0.0, carry = 0.0;
  double fa[2][PF], fb[2][PF], fc[2][PF];
  auto block = [&](int b, auto ramp) {
    constexpr bool RAMP = decltype(ramp)::value;
    const int t0 = b * PB;
    double xv[PB];
#pragma unroll
    for (int k = 0; k < PB; k += 2) {
      const double2 x = *reinterpret_cast<const double2*>(&sm.x[b & 1][k]);
      xv[k] = x.x;
      xv[k + 1] = x.y;
    }
#pragma unroll
    for (int k = 0; k < PB; ++k) {
      const int t = t0 + k;
      const int Q = k / PF;
      if (k % PF == 0) fetch(t + PF, fa[Q ^ 1], fb[Q ^ 1], fc[Q ^ 1]);
      double nbv = FWD ? __shfl_up_sync(kFull, carry, 1) : __shfl_down_sync(kFull, carry, 1);
      if (lane == edge) nbv = xv[k];
      const double va = fa[Q][k % PF], vb = fb[Q][k % PF], vc = fc[Q][k % PF];
      const int j = col(t);
      double v;
      if (MODE == kSweepPiv) {
        // p = a_kk - U_{i,j-1}^2 pinv_{k-1} - V_{i-1,j}^2 pinv_{k-W}, guarded, then 1/p
        const double u = j > 0 ? vb : 0.0;
        double p = fma(-(vc * vc), nbv, fma(-(u * u), prev, va));
        if (!(p > 1e-12 * va && p > 0.0)) p = (va > 0.0) ? va : 1.0;
        v = 1.0 / p;
      } else {
        v = fma(vc, nbv, fma(vb, prev, va));
      }
      // a lane that has not reached its first column contributes nothing; past its last
      // one its values reach no stored row
      if (RAMP && t < skew) v = 0.0;
      else sa[j & (kSweepCols - 1)] = v;
      if (publish && j >= 0 && j < g.W) st_relaxed(io.xout + j, v);
      prev = v;
      carry = v;
    }
  };
  for (int b = 0;; ++b) {
    sweep_pair_sync(pair);  // barrier b
    if (sm.fail) return false;
    if (b == g.nb) return true;
    if (b == 0) fetch(0, fa[0], fb[0], fc[0]);
    if (b < 32 / PB) block(b, std::true_type{});
    else block(b, std::false_type{});
  }
}

}  // namespace ulp
