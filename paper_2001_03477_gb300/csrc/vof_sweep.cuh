// vof_sweep.cuh -- the pieces of a sweep that its kernels share: the no-op
// test, the face energy flux, the cell update and the PLIC plane and donor
// volume of a mixed cell (Malan et al., arXiv:2001.03477, Sec. 3.3.1 and
// 3.4.1).  vof_sweep.cu (stand-alone sweeps) and vof_fused.cu (the sweeps of
// a time step) call the same functions, so both give the same bits.
#pragma once
#include "vof_launch.h"

namespace vofgb {

// ---------------------------------------------------------------------------
// No-op cells.  A cell's c and e come out bit-identical when the 7 cells
// around it along the sweep axis have the same (c, e) bits, c is exactly 0 or
// 1 and the cell has not changed earlier in the step: both donors are then
// pure with the same c, F = c a, both face temperatures equal T, and
// (G - Theta a) vanishes exactly on both faces.
// ---------------------------------------------------------------------------

constexpr unsigned kFull = 0xffffffffu;
constexpr long long kOneBits = 0x3FF0000000000000LL;

__device__ __forceinline__ bool same_bits(double a, double b) { return dbits(a) == dbits(b); }
__device__ __forceinline__ bool is01(double c) { long long b = dbits(c); return b == 0 || b == kOneBits; }

__device__ __forceinline__ size_t cell_at(const GridDev& g, int x, int y, int z) {
  return ((size_t)z * g.n[1] + y) * g.n[0] + x;
}

template <int AX>
__device__ __forceinline__ size_t face_of(const GridDev& g, int f, int x, int y, int z) {
  if (AX == 0) return ((size_t)z * g.n[1] + y) * (g.n[0] + 1) + f;
  if (AX == 1) return ((size_t)z * (g.n[1] + 1) + f) * g.n[0] + x;
  return ((size_t)f * g.n[1] + y) * g.n[0] + x;
}

// An FP64 instruction occupies its SM partition's FP64 unit for ~76 cycles
// whatever its active lanes, predicated ones included, so the forms that few
// lanes need are calls under a warp vote: a warp without such a lane issues
// none of their FP64 instructions.

// Face temperature: WENO5 from the donor value and the four differences in
// upwind order, the weights in pairs or, in the precision form, in FP32.
__device__ __forceinline__ double face_temperature(bool f32, double v0, double D0, double D1, double D2, double D3) {
  return f32 ? weno5_add(v0, weno5_corr_f(D0, D1, D2, D3)) : weno5_add6(v0, weno5_corr6_df(D0, D1, D2, D3));
}

// VOF flux c a of a donor that is not mixed: 0 a and 1 a exactly for c = 0, 1
// (no multiply); a c within eps of them is multiplied.
static __device__ __noinline__ double flux_mul(double c, double a) { return c * a; }
__device__ __forceinline__ double flux01(double cd, double a) {  // cd exactly 0 or 1
  return dbits(cd) == kOneBits ? a : __longlong_as_double(dbits(a) & (long long)0x8000000000000000ull);
}
__device__ __forceinline__ double pure_flux(double cd, double a) {
  const long long b = dbits(cd);
  double F = flux01(cd, a);
  const bool other = b != 0 && b != kOneBits;
  if (__any_sync(__activemask(), other)) {
    const double Fm = flux_mul(cd, a);
    if (other) F = Fm;
  }
  return F;
}

// Energy flux G = T_f (C_pl F + C_pg (a - F)): with F = a (cd = 1) or 0 (cd
// = 0) it is (T_f C_pl) a or (T_f C_pg) a, the same rounding as the general
// form's one fused multiply-add (the other term is an exact zero): two FP64
// instructions instead of five.
static __device__ __noinline__ double energy_mix(double Tf, double Cp_l, double Cp_g, double F, double a) {
  return fma(Tf * Cp_l, F, (Tf * Cp_g) * (a - F));
}
__device__ __forceinline__ double energy_flux01(const GridDev& g, double Tf, double cd, double a) {
  return (Tf * (dbits(cd) == kOneBits ? g.Cp_l : g.Cp_g)) * a;
}
__device__ __forceinline__ double energy_flux(const GridDev& g, double Tf, double cd, double F, double a) {
  const bool pure = is01(cd);
  double G = energy_flux01(g, Tf, cd, a);
  if (__any_sync(__activemask(), !pure)) {
    const double Gm = energy_mix(Tf, g.Cp_l, g.Cp_g, F, a);
    if (!pure) G = Gm;
  }
  return G;
}

// c of one cell from its two faces: {new c, clipped volume}.  Weymouth-Yue
// (lag = 0): cc is 0 or 1, so cc a is a or 0 exactly; Lagrangian explicit:
// the cell's own c.
static __device__ __noinline__ double2 update_c_general(double c, double Fl, double al, double Fr, double ar, int cc,
                                                        int lag) {
  const double lf = lag ? Fl - c * al : (cc ? Fl - al : Fl);
  const double rf = lag ? Fr - c * ar : (cc ? Fr - ar : Fr);
  const double cn = (c + lf) - rf;
  double2 r = make_double2(cn, 0.0);
  if (dlt0(cn)) r = make_double2(0.0, cn);
  else if (dgt1(cn)) r = make_double2(1.0, cn - 1.0);
  return r;
}
// A cell with c = cc exactly 0 or 1 between faces that carry its own phase
// (F = c a on both, by their bits) keeps c without arithmetic.
__device__ __forceinline__ double2 update_c(double c, double Fl, double al, double Fr, double ar, bool cc, bool lag) {
  const bool own = cc ? dbits(c) == kOneBits && same_bits(Fl, al) && same_bits(Fr, ar)
                      : dbits(c) == 0 && !dnz(Fl) && !dnz(Fr);
  double2 r = make_double2(c, 0.0);
  if (__any_sync(__activemask(), !own)) {
    const double2 q = update_c_general(c, Fl, al, Fr, ar, cc ? 1 : 0, lag ? 1 : 0);
    if (!own) r = q;
  }
  return r;
}

// Theta of the Lagrangian-explicit form (the cell's own c); C_p(c) T exactly
// as for cc when c is 0 or 1
static __device__ __noinline__ double theta_mix(double T, double c, double Cp_l, double Cp_g) {
  return (T * Cp_l) * c + (T * Cp_g) * (1.0 - c);
}
__device__ __forceinline__ double theta_now(const GridDev& g, double T, double c, bool cc, bool lag) {
  double th = (cc ? g.Cp_l : g.Cp_g) * T;
  const bool mix = lag && !is01(c);
  if (__any_sync(__activemask(), mix)) {
    const double m = theta_mix(T, c, g.Cp_l, g.Cp_g);
    if (mix) th = m;
  }
  return th;
}

// c of a word that carries a step's two tag bits above the value (vof_fused.cu)
__device__ __forceinline__ double c_value(double w) {
  return __hiloint2double((int)((unsigned)__double2hiint(w) & 0x3FFFFFFFu), __double2loint(w));
}

// PLIC plane (MYC normal, plane constant) of the 3x3x3 stencil centred on
// position (qx, qy, qz), each index mapped by the boundary conditions.
// tagged: the words carry a step's tag bits.
// F32: the precision form's FP32 MYC normal (its own instance, so that the
// FP64 form keeps its register budget); YOUNGS: Youngs' normal instead
template <bool F32, bool YOUNGS = false>
__device__ __forceinline__ double4 stencil_plane(const GridDev& g, const double* __restrict__ c_in, int qx, int qy,
                                                 int qz, bool tagged = false) {
  double s[27];
#pragma unroll
  for (int oz = 0; oz < 3; ++oz) {
    const int zz = map_idx(qz + oz - 1, g.n[2], g.bc[2]);
#pragma unroll
    for (int oy = 0; oy < 3; ++oy) {
      const int yy = map_idx(qy + oy - 1, g.n[1], g.bc[1]);
#pragma unroll
      for (int ox = 0; ox < 3; ++ox) {
        const int xx = map_idx(qx + ox - 1, g.n[0], g.bc[0]);
        s[(oz * 3 + oy) * 3 + ox] = __ldg(c_in + cell_at(g, xx, yy, zz));
      }
    }
  }
  if (tagged) {
#pragma unroll
    for (int i = 0; i < 27; ++i) s[i] = c_value(s[i]);
  }
  double m[3];
  if (YOUNGS) youngs_normal(s, m);
  else if (F32) myc_normal_f(s, m);
  else myc_normal(s, m);
  double4 pl;
  pl.x = m[0]; pl.y = m[1]; pl.z = m[2];
  pl.w = plane_alpha(m[0], m[1], m[2], s[13]);
  return pl;
}

// Volume a mixed donor of plane pl sends through one of its faces (pos: the
// face on its right; da = |a| > 0).  Weymouth-Yue: the donor slab of width
// |a|; Lagrangian explicit: the preimage of width |a| / J, J = 1 + (a_r - a_l)
// of the donor (adl, adr), its liquid stretched by J (the width capped at 1).
__device__ __forceinline__ double donor_volume(const GridDev& g, int ax, const double4& pl, double cd, double da,
                                               bool pos, double adl, double adr, int* __restrict__ status) {
  if (da > 1.0 && status) atomicOr(status, DEV_CFL);
  double w = da, J = 1.0;
  if (g.le) {
    J = 1.0 + (adr - adl);
    if (J > da) {
      w = da / J;
    } else {
      w = 1.0;
      if (status) atomicOr(status, DEV_CFL);
    }
  }
  const double mv[3] = {pl.x, pl.y, pl.z};
  double vol = g.f32 ? slab_volume_f(mv, pl.w, ax, pos ? 1.0 - w : 0.0, w, cd)
                     : slab_volume_nn(mv, pl.w, ax, pos ? 1.0 - w : 0.0, w);
  if (g.le) vol = J * vol;
  return vol;
}

}  // namespace vofgb
