// ulp_flow32.cuh -- tile steps of the mixed-precision persistent solvers that run off the
// FP64 planes: the FP32 copies at the start of a solve and the true residual.
#pragma once
#include "ulp_flow.cuh"
#include "ulp_mixed.cuh"

namespace ulp {

// FP32 copies of the weights and the Jacobi inverse; the correction starts at 0.
template <int KIND>
__device__ __forceinline__ void conv_tile(const PcgArgs& a, const MapDesc& M, int t, int lane) {
  const TileGeo g = tile_geo(M, t, a.R);
  const size_t P = M.pitch;
  const int j = g.j0 + 2 * lane;
  for (int i = g.i0; i < g.i1; ++i) {
    const size_t off = (size_t)i * P + j;
    const double2 u = ld2(M.f.U, off), v = ld2(M.f.V, off);
    stf2(M.h.U, off, make_float2((float)u.x, (float)u.y));
    stf2(M.h.V, off, make_float2((float)v.x, (float)v.y));
    if (KIND == kJacobi) {
      const double2 di = ld2(M.f.Dinv, off);
      stf2(M.h.Dinv, off, make_float2((float)di.x, (float)di.y));
    }
    stf2(M.h.x, off, make_float2(0.f, 0.f));
  }
}

// True residual in FP64: r = b - A phi (FP64 weights, FP64 phi), rounded to
// FP32 for the recurrence; s = M^-1 r; the lane's shares of r^T s, r^T r (and b^T b).
template <int KIND>
__device__ __forceinline__ void res64_tile(const PcgArgs& a, const MapDesc& M, bool init, int t, int lane, double& vrs,
                                           double& vrr, double& bb) {
  const TileGeo g = tile_geo(M, t, a.R);
  XPlane x{M.f.phi, (size_t)M.pitch};
  DF rs, rr;
  bb = 0.0;
  auto epi = [&](size_t off, double2, double2 ax) {
    const double2 bv = ld2(M.f.b, off);
    const float2 r = make_float2((float)(bv.x - ax.x), (float)(bv.y - ax.y));
    stf2(M.h.r, off, r);
    if (KIND == kJacobi) {
      const float2 di = ldf2(M.h.Dinv, off);
      const float2 s = make_float2(di.x * r.x, di.y * r.y);
      stf2(M.h.s, off, s);
      rs.add_prod(r.x, s.x);
      rs.add_prod(r.y, s.y);
    }
    rr.add_prod(r.x, r.x);
    rr.add_prod(r.y, r.y);
    if (init) {
      bb = fma(bv.x, bv.x, bb);
      bb = fma(bv.y, bv.y, bb);
    }
  };
  stencil_tile(M, g.i0, g.i1, g.j0, lane, M.f.U, M.f.V, M.f.D, x, epi);
  vrr = rr.value();
  vrs = (KIND == kIdentity) ? vrr : rs.value();
}

}  // namespace ulp
