// vof_diffuse.cu -- implicit heat diffusion with the interface as a
// Dirichlet boundary (Malan et al., arXiv:2001.03477, Sec. 3.4.2: Eqs.
// T_diff_disc and mod_branchesT, after Sato and Niceno).
//
// A node is liquid when c >= 1/2, else gas; each phase diffuses with its own
// conductivity and T_Gamma = T_sat on the interface.  Along each axis the
// gradient towards a same-phase neighbour is the plain difference over h;
// towards the other phase it is (T_Gamma - T) / theta, theta the distance
// from the node to the interface along that axis, and the axis' second
// difference is divided by (d_- + d_+) / 2 (d = h or theta).  theta is the
// height function of the 7 cells centred on the node along the axis when
// the column ends in pure cells of the node's phase behind and the other
// phase beyond (the interface H - 3.5 cells ahead of a liquid node, 3.5 - H
// of a gas node), else the distance along the axis to the PLIC plane of the
// pair's mixed cell (the node's own if mixed, else the neighbour's), half a
// cell when both are pure or the plane is parallel to the axis; capped to
// [1e-3 h, h].  Zero-gradient walls carry no flux unless the caller fixes
// their temperature T_w: the node then sees the wall half a cell away,
// gradient (T_w - T) / (h / 2), d = h / 2 (the heated wall of Sec. 4.3).
// Periodic axes wrap.  Backward Euler with the heat capacity of the
// reading chosen:
//   phase (the default): every node diffuses with the constant C_p of its
//     phase, C_p,node (T' - T) / dt = k_p sum L(T'), and the cell's energy
//     changes by the heat conducted into it, e' = e + C_p,node (T' - T)
//     (Sec. 3.4.2 solves phase by phase with constant properties);
//   mixture: C_p(c) (T' - T) / dt = k_p sum L(T'), e' = C_p(c) T'.
// T = e / C_p(c) in both.
//
// Kernels: k_dif_mlist (list of the mixed cells), k_dif_planes (MYC normal
// and plane constant of each listed cell), k_dif_classify (per cell: its
// class and T at the start), k_dif_irregular (the listed cells next to the
// interface or a heated wall: their couplings), the Jacobi sweeps -- the
// system is strictly diagonally dominant (C_p / dt sits on the diagonal alone),
// so the iteration converges; on every fourth sweep the largest change is
// reduced -- and the store of e'.
//
// Phase heat capacity: the sweeps iterate on the change d = T - T0 of each node,
//   d' = B sum d_nb + s,  B = k_p / h^2 / diagonal,  s = B sum (T0_nb - T0),
// (the same iterates T, since C_p / dt and the couplings add up to the
// diagonal), s formed once in FP64 (k_dif_first: it is also the first sweep),
// d, B and s held as pairs of FP32 numbers (48 bits of the change itself), over
// the power of two next to the largest T.  What bounds a sweep on this part is the
// FP64 unit: 8 FP64 instructions per cell took 45 us at 128^3 (76 cycles of an
// SM partition each); the pairs' FP32 instructions take 20.6 us (two cells of a row in one 16-byte
// block; 22 us with high and low parts in arrays of their own).
// A pair of the change is as accurate as an FP64 T only while the change is small
// beside T.  Every iterate lies between the smallest and the largest of the T0,
// of T_Gamma where a cell sees an interface and of the walls' T, so |d| is at most
// their range R, and the rule is 16 R <= the smallest of them (all positive): the
// energies' errors against long double are then 0.2 to 0.4 of the FP64 sweeps'
// (14^3 box, diffusion numbers 0.05 to 20; R = T / 8: up to 0.65 in the mean and as
// large at most; R = T: 1.4 to 24 times).  Other calls sweep T itself in FP64 (128^3,
// a hot wall on gas at 0: 42.7 us a sweep all in all, 20.4 in pairs).  The
// kernels decide on the device: the first batch's sweeps in pairs return at once
// where the rule says FP64, and the host reads it with that batch's checks.
// The sweeps are queued in batches without waiting: each starts by reading the last
// check's result and leaves its buffers alone once that was within tol.
// Mixture heat capacity: the FP64 form, every cell's diagonal stored.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "../../include/vofgb.h"
#include "vof_launch.h"

namespace vofgb {

namespace {

constexpr int kDifThreads = 256;
constexpr int kDifCTAs = 152 * 8;
constexpr int kDifPlaneThreads = 64;  // few cells, long FP64 chains: spread over the SMs
constexpr double kThetaEps = 1e-3;

__device__ __forceinline__ size_t dcid(const GridDev& g, int x, int y, int z) {
  return ((size_t)z * g.n[1] + y) * g.n[0] + x;
}

// coordinate p + k along an axis of n cells: wrapped (periodic) or -1 off a
// zero-gradient wall
__device__ __forceinline__ int step_coord(int p, int k, int n, int bc) {
  int q = p + k;
  if (q < 0 || q >= n) {
    if (bc != 0) return -1;
    q %= n;
    if (q < 0) q += n;
  }
  return q;
}

// the same, clamped to the boundary cell on a zero-gradient axis (the
// height function's column extends by its boundary values)
__device__ __forceinline__ int clamp_coord(int p, int k, int n, int bc) {
  int q = p + k;
  if (bc != 0) return q < 0 ? 0 : (q >= n ? n - 1 : q);
  q %= n;
  return q < 0 ? q + n : q;
}

// the mixed cells of the grid, appended to a list (one atomic per warp);
// the list's order varies from run to run, and nothing depends on it
__global__ void __launch_bounds__(kDifThreads)
k_dif_mlist(GridDev g, const double* __restrict__ c, uint32_t* __restrict__ mlist, int* __restrict__ count,
            size_t N) {
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  const size_t n_iter = (N + stride - 1) / stride;  // whole warps iterate together
  const int lane = threadIdx.x & 31;
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (size_t it = 0; it < n_iter; ++it, i += stride) {
    const bool mx = i < N && is_mixed_b(__ldg(c + i), g);
    const unsigned mask = __ballot_sync(0xffffffffu, mx);
    if (!mask) continue;
    int base = 0;
    if (lane == __ffs(mask) - 1) base = atomicAdd(count, __popc(mask));
    base = __shfl_sync(0xffffffffu, base, __ffs(mask) - 1);
    if (mx) mlist[base + __popc(mask & ((1u << lane) - 1u))] = (uint32_t)i;
  }
}

// MYC normal and plane constant of each listed mixed cell (lanes dense over
// the list: the FP64 work of a warp serves 32 cells)
__global__ void __launch_bounds__(kDifPlaneThreads)
k_dif_planes(GridDev g, const double* __restrict__ c, const uint32_t* __restrict__ mlist,
             const int* __restrict__ count, double4* __restrict__ plane) {
  const int nm = *count;
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < nm; k += gridDim.x * blockDim.x) {
    const size_t i = mlist[k];
    const double cv = __ldg(c + i);
    int x, y, z;
    cell_xyz(g, i, x, y, z);
    double s[27];
#pragma unroll
    for (int oz = 0; oz < 3; ++oz)
#pragma unroll
      for (int oy = 0; oy < 3; ++oy)
#pragma unroll
        for (int ox = 0; ox < 3; ++ox)
          s[(oz * 3 + oy) * 3 + ox] = __ldg(c + dcid(g, map_idx(x + ox - 1, g.n[0], g.bc[0]),
                                                      map_idx(y + oy - 1, g.n[1], g.bc[1]),
                                                      map_idx(z + oz - 1, g.n[2], g.bc[2])));
    double m[3];
    myc_normal(s, m);
    double4 p;
    p.x = m[0]; p.y = m[1]; p.z = m[2];
    p.w = plane_alpha(m[0], m[1], m[2], cv);
    plane[i] = p;
  }
}

// theta (cell units) from node (x, y, z) towards its neighbour in direction
// s along axis, the two being of different phases
__device__ double interface_theta(const GridDev& g, const double* __restrict__ c, const double4* __restrict__ plane,
                                  int x, int y, int z, int axis, int s, bool liquid_p) {
  const int pc[3] = {x, y, z};
  const int n = g.n[axis], bc = g.bc[axis];
  double col[7];
  for (int k = -3; k <= 3; ++k) {
    int q[3] = {x, y, z};
    q[axis] = clamp_coord(pc[axis], s * k, n, bc);
    col[k + 3] = __ldg(c + dcid(g, q[0], q[1], q[2]));
  }
  const double back = col[0], front = col[6];
  const double one_m_eps = 1.0 - g.eps;
  const bool ok = liquid_p ? (back >= one_m_eps && front <= g.eps) : (back <= g.eps && front >= one_m_eps);
  double theta;
  if (ok) {
    double H = 0.0;
    for (int k = 0; k < 7; ++k) H += col[k];
    theta = liquid_p ? H - 3.5 : 3.5 - H;
  } else {
    theta = 0.5;
    const size_t pid = dcid(g, x, y, z);
    int q[3] = {x, y, z};
    q[axis] = step_coord(pc[axis], s, n, bc);
    int mcell = -1;  // 0: the node's own cell, 1: the neighbour
    if (is_mixed_b(__ldg(c + pid), g)) mcell = 0;
    else if (q[axis] >= 0 && is_mixed_b(__ldg(c + dcid(g, q[0], q[1], q[2])), g)) mcell = 1;
    if (mcell >= 0) {
      const double4 p = plane[mcell == 0 ? pid : dcid(g, q[0], q[1], q[2])];
      // the node in the mixed cell's local coordinates
      double x0[3] = {0.5, 0.5, 0.5};
      if (mcell == 1) x0[axis] = 0.5 - (double)s;
      const double mm[3] = {p.x, p.y, p.z};
      const double ma = mm[axis] * (double)s;
      if (ma != 0.0) {
        const double t = (p.w - ((mm[0] * x0[0] + mm[1] * x0[1]) + mm[2] * x0[2])) / ma;
        theta = fabs(t);
      }
    }
  }
  return fmin(fmax(theta, kThetaEps), 1.0);
}

// walls at fixed temperature, per face x-, x+, y-, y+, z-, z+
struct DifWalls {
  double T[6];
  int on[6];
};

// Per-phase constants of the assembled system (index 0 gas, 1 liquid),
// computed on the host in the order the per-cell assembly would use:
// k_p / h^2, C_p / dt (phase heat capacity), and the reciprocal of the
// diagonal C_p / dt + n k_p / h^2 of a cell with n same-phase sides.
struct DifConst {
  double kq[2];
  double cdt[2];
  double rdiag[2][7];
  double B[2][7];    // kq * rdiag
  float2 Bf[2][7];   // the same as pairs of FP32 numbers
  int wlo, whi;      // smallest and largest high word of the heated walls' T
};

// Cell classes: bits 0..5 the sides (-x, +x, -y, +y, -z, +z) with a
// neighbour in the grid; kDifLiq the node is liquid (c >= 1/2); kDifIrr
// the cell has an interface or heated-wall side, so its couplings and
// diagonal are stored.  Every other cell couples by k_p / h^2 to each
// neighbour and, with the phase heat capacity, takes its diagonal from the
// table: the sweeps then read no coupling for it.
constexpr uint8_t kDifLiq = 0x40, kDifIrr = 0x80;

struct DifVec {
  double* off;    // [6 N]: coupling to the neighbour (face order -x, +x, -y, +y, -z, +z), kDifIrr cells
                  // only; in pairs over the diagonal, as a pair of FP32 numbers
  double* diag;   // [N] reciprocal of the diagonal; kDifIrr cells (all cells with the mixture heat capacity)
  double* rhs;    // [N] right side; likewise
  double* T0;     // [N] T at the start (the first iterate in FP64)
  double* Ta;     // [N] the two later Jacobi iterates
  double* Tb;
  unsigned long long* part;  // [kDifChecks] the largest change of each checked sweep of a batch (bits),
                             // [kDifChecks]: infinity where the sweeps run in pairs, else 0
  uint8_t* cls;   // [N] cell class
  // in pairs: two cells of a row (x even, x + 1) in 16 bytes, {hi, hi, lo, lo},
  // a row of px such blocks
  float4* s;      // [px ny nz]: s, also the first iterate d
  float4* d[2];   // the two later iterates
  int px;
  int* range;     // [0] the largest high word of a T, [1] 0x7FFFFFFF minus the smallest (unsigned maximum)
};
// high words (as signed integers: positive values in order, any negative one
// below them) of the smallest and the largest T of the system
__device__ __forceinline__ int dif_lo(const DifVec& v, const DifConst& K) { 
  return min((int)(0x7FFFFFFFu - (unsigned)v.range[1]), K.wlo);
}
__device__ __forceinline__ int dif_hi(const DifVec& v, const DifConst& K) { return max(v.range[0], K.whi); }
// the rule for pairs (an infinite or NaN T fails it: hi is its high word, or lo
// is negative)
__device__ __forceinline__ bool dif_pairs(const DifVec& v, const DifConst& K) {
  const int lo = dif_lo(v, K), hi = dif_hi(v, K);
  if (lo < 0x00100000 || hi >= 0x7FE00000) return false;
  const double a = __hiloint2double(lo, 0), b = __hiloint2double(hi + 1, 0);  // around all of them
  return 16.0 * (b - a) <= a;
}
// the pairs hold d / 2^k
__device__ __forceinline__ int dif_scale(const DifVec& v, const DifConst& K) { return (dif_hi(v, K) >> 20) - 1023; }
// the high part of cell (x, y, z) in array a; the low part is two floats on
__device__ __forceinline__ float* part_of(const GridDev& g, const DifVec& v, float4* a, int x, int y, int z) {
  return reinterpret_cast<float*>(a + ((size_t)z * g.n[1] + y) * v.px + (x >> 1)) + (x & 1);
}

constexpr long long kHalfBits = 0x3FE0000000000000LL;  // 0.5: c >= 1/2 on the integer pipe (c >= +0)

// The six sides of node (x, y, z): in the grid (inm), with a node of the
// same phase (same), and whether a side is a wall at fixed temperature.
__device__ __forceinline__ void dif_sides(const GridDev& g, const double* __restrict__ c, const DifWalls& walls,
                                          int x, int y, int z, bool liq, unsigned& inm, unsigned& same,
                                          bool& hot_wall) {
  const int pc[3] = {x, y, z};
  inm = 0u;
  same = 0u;
  hot_wall = false;
#pragma unroll
  for (int f = 0; f < 6; ++f) {
    const int axis = f >> 1, s = (f & 1) ? 1 : -1;
    int q[3] = {x, y, z};
    q[axis] = step_coord(pc[axis], s, g.n[axis], g.bc[axis]);
    if (q[axis] < 0) {
      hot_wall = hot_wall || walls.on[f] != 0;
      continue;
    }
    inm |= 1u << f;
    if ((dbits(__ldg(c + dcid(g, q[0], q[1], q[2]))) >= kHalfBits) == liq) same |= 1u << f;
  }
}

// the sweep's CTAs: 32 x 8 cells of every plane each, enough z shares for
// a few waves
static dim3 dif_sweep_grid(const GridDev& g) {
  const unsigned gx = (unsigned)((g.n[0] + 31) / 32), gy = (unsigned)((g.n[1] + 7) / 8);
  unsigned gz = (unsigned)std::max(1, std::min(g.n[2], (int)(152u * 16u / std::max(1u, gx * gy))));
  return dim3(gx, gy, gz);
}

// Per cell: its class and T; with the mixture heat capacity every cell that
// couples by k_p / h^2 on all sides also gets its right side and diagonal; the
// others -- next to the interface or a heated wall -- are listed for
// k_dif_irregular (one atomic per warp; the list's order varies from run to
// run, and nothing depends on it).
template <bool PHASE>
__global__ void __launch_bounds__(kDifThreads)
k_dif_classify(GridDev g, const double* __restrict__ c, const double* __restrict__ e, DifVec v, DifWalls walls,
               double inv_dt, DifConst K, uint32_t* __restrict__ ilist, int* __restrict__ icount) {
  const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 8 + threadIdx.y;
  if (y >= g.n[1]) return;  // whole warps (a warp is one row segment)
  const bool in_x = x < g.n[0];
  const int lane = threadIdx.x;
  int thi = 0;
  unsigned tlo = 0u;
  auto in_range = [&](double T) {
    thi = max(thi, __double2hiint(T));
    tlo = max(tlo, 0x7FFFFFFFu - (unsigned)__double2hiint(T));
  };
  for (int z = blockIdx.z; z < g.n[2]; z += gridDim.z) {
    const size_t i = ((size_t)z * g.n[1] + y) * g.n[0] + x;
    bool irr = false;
    if (in_x) {
      const double cv = __ldg(c + i);
      const bool liq = dbits(cv) >= kHalfBits;
      const double T0 = temp_of(g, __ldg(e + i), cv);
      unsigned inm, same;
      bool hot_wall;
      dif_sides(g, c, walls, x, y, z, liq, inm, same, hot_wall);
      const int li = liq ? 1 : 0;
      v.T0[i] = T0;
      in_range(T0);
      if (same != inm) in_range(g.T_sat);
      irr = hot_wall || same != inm;
      v.cls[i] = (uint8_t)(inm | (liq ? kDifLiq : 0) | (irr ? kDifIrr : 0));
      if (!irr && !PHASE) {
        // every side in the grid couples by k_p / h^2 (walls without flux:
        // 0); with the phase heat capacity the sweeps form the right side
        // C_p / dt T0 and take the diagonal from the table themselves
        const double cdt = (g.Cp_l * cv + g.Cp_g * (1.0 - cv)) * inv_dt;
        v.rhs[i] = cdt * T0;
        const double kq = li ? K.kq[1] : K.kq[0];
        double diag = cdt;
#pragma unroll
        for (int f = 0; f < 6; ++f)
          if (inm & (1u << f)) diag += kq;
        v.diag[i] = 1.0 / diag;
      }
    }
    const unsigned mask = __ballot_sync(0xffffffffu, irr);
    if (!mask) continue;
    int base = 0;
    if (lane == __ffs(mask) - 1) base = atomicAdd(icount, __popc(mask));
    base = __shfl_sync(0xffffffffu, base, __ffs(mask) - 1);
    if (irr) ilist[base + __popc(mask & ((1u << lane) - 1u))] = (uint32_t)i;
  }
  if constexpr (PHASE) {
    thi = __reduce_max_sync(0xffffffffu, thi);
    tlo = __reduce_max_sync(0xffffffffu, tlo);
    if (lane < 2) {  // (few warps find either larger)
      const unsigned key = lane ? tlo : (unsigned)thi;
      if (key > *(volatile unsigned*)(v.range + lane)) atomicMax(reinterpret_cast<unsigned*>(v.range) + lane, key);
    }
  }
}

// x / 2^k as a pair of FP32 numbers (48 bits)
__device__ __forceinline__ float2 pair_of(double x, int k) {
  const df::f2 p = df::split_scaled(df::words_of(x), k);
  return make_float2(p.hi, p.lo);
}
// f 2^k (0 below the FP64 normal range; infinities and NaN kept)
__device__ __forceinline__ double wide_of(float f, int k) {
  const unsigned b = __float_as_uint(f), ef = (b >> 23) & 0xFFu;
  int ex = ef == 255u ? 2047 : (int)ef + 896 + k;
  unsigned long long m = (unsigned long long)(b & 0x7FFFFFu) << 29;
  if (ex > 2046 && ef != 255u) { ex = 2047; m = 0; }
  if (ef == 0u || ex <= 0) { ex = 0; m = 0; }
  return __longlong_as_double((long long)(((unsigned long long)(b & 0x80000000u) << 32) | ((unsigned long long)ex << 52) | m));
}
__device__ __forceinline__ df::f2 f2_of(float2 p) { return df::f2{p.x, p.y}; }

// Checks of a batch of sweeps: at most kDifChecks; a sweep reads the slot of
// the check before it (the first ones of a call, in pairs, whether the rule
// lets them run).
constexpr int kDifChecks = 31;

// A check's result within tol (both non-negative: compared as integers).
__device__ __forceinline__ bool dif_done(const unsigned long long* __restrict__ prev, double tol) {
  return prev && *prev <= (unsigned long long)dbits(tol);
}

// Per listed cell (lanes dense over the list): the six couplings (heights
// or plane distances on the interface sides), the diagonal and the right
// side.
__global__ void __launch_bounds__(kDifPlaneThreads)
k_dif_irregular(GridDev g, double h, double inv_h, double inv_dt, double k_l, double k_g,
                const double* __restrict__ c, const double* __restrict__ e, const double4* __restrict__ plane,
                DifVec v, DifWalls walls, int phase_cp, DifConst K, const uint32_t* __restrict__ ilist,
                const int* __restrict__ icount) {
  const int ni = *icount;
  const bool pairs = phase_cp && dif_pairs(v, K);
  const int ks = dif_scale(v, K);
  if (blockIdx.x == 0 && threadIdx.x == 0) v.part[kDifChecks] = pairs ? 0x7FF0000000000000ull : 0ull;
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < ni; k += gridDim.x * blockDim.x) {
    const size_t i = ilist[k];
    int x, y, z;
    cell_xyz(g, i, x, y, z);
    const double cv = __ldg(c + i);
    const bool liq = dbits(cv) >= kHalfBits;
    const double T0 = temp_of(g, __ldg(e + i), cv);
    unsigned inm, same;
    bool hot_wall;
    dif_sides(g, c, walls, x, y, z, liq, inm, same, hot_wall);
    const int li = liq ? 1 : 0;
    const double cdt = phase_cp ? K.cdt[li] : (g.Cp_l * cv + g.Cp_g * (1.0 - cv)) * inv_dt;
    double diag = cdt, rhs = cdt * T0;
    double off[6], gain = 0.0;  // gain: the heat conducted at T0 over its own unit (pairs)
    auto nb_T = [&](int f) {     // T0 of the neighbour across side f
      int q[3] = {x, y, z};
      q[f >> 1] = step_coord(q[f >> 1], (f & 1) ? 1 : -1, g.n[f >> 1], g.bc[f >> 1]);
      return v.T0[dcid(g, q[0], q[1], q[2])];
    };
    const double kp = liq ? k_l : k_g;
    // a same-phase neighbour couples by k_p / h^2 (no division); only the
    // interface and heated-wall sides need their own distances
    const double kq = kp * (inv_h * inv_h);
#pragma unroll
    for (int axis = 0; axis < 3; ++axis) {
      double cs[2], cq[2], cst[2], d[2], Tfix[2] = {0.0, 0.0};
      bool reg[2];  // the side's distance is h (same phase or a wall without flux)
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        const int f = 2 * axis + side;
        reg[side] = true;
        if (!(inm & (1u << f)) && walls.on[f]) {  // a wall at fixed T, half a cell away
          const double Tw = walls.T[f];
          cs[side] = 2.0 * inv_h; cq[side] = 0.0; cst[side] = Tw * 2.0 * inv_h; d[side] = 0.5 * h;
          Tfix[side] = Tw;
          reg[side] = false;
        } else if (!(inm & (1u << f))) {  // a wall: no flux
          cs[side] = 0.0; cq[side] = 0.0; cst[side] = 0.0; d[side] = h;
        } else if (same & (1u << f)) {
          cs[side] = inv_h; cq[side] = inv_h; cst[side] = 0.0; d[side] = h;
        } else {
          const double th = interface_theta(g, c, plane, x, y, z, axis, side ? 1 : -1, liq) * h;
          cs[side] = 1.0 / th; cq[side] = 0.0; cst[side] = g.T_sat / th; d[side] = th;
          Tfix[side] = g.T_sat;
          reg[side] = false;
        }
      }
      if (reg[0] && reg[1]) {
        // both sides h: k_p / h^2 each (walls without flux contribute 0)
#pragma unroll
        for (int side = 0; side < 2; ++side) {
          const double o = dnz(cq[side]) ? kq : 0.0;
          diag += o;
          off[2 * axis + side] = o;
          if (pairs && dnz(o)) gain += o * (nb_T(2 * axis + side) - T0);
        }
      } else {
        const double kd = kp / (0.5 * (d[0] + d[1]));
#pragma unroll
        for (int side = 0; side < 2; ++side) {
          diag += kd * cs[side];
          off[2 * axis + side] = kd * cq[side];
          rhs += kd * cst[side];
          if (pairs) {
            // towards a fixed temperature (T_Gamma, T_w) or the neighbour's
            if (dnz(cq[side])) gain += kd * cq[side] * (nb_T(2 * axis + side) - T0);
            else if (dnz(cs[side])) gain += kd * cs[side] * (Tfix[side] - T0);
          }
        }
      }
    }
    const double rd = 1.0 / diag;  // stored as its reciprocal: the sweeps multiply
    if (pairs) {
#pragma unroll
      for (int f = 0; f < 6; ++f) reinterpret_cast<float2*>(v.off)[6 * i + f] = pair_of(off[f] * rd, 0);
      const float2 sp = pair_of(gain * rd, ks);
      float* const at = part_of(g, v, v.s, x, y, z);
      at[0] = sp.x;
      at[2] = sp.y;
    } else {
#pragma unroll
      for (int f = 0; f < 6; ++f) v.off[6 * i + f] = off[f];
      v.diag[i] = rd;
      v.rhs[i] = rhs;
    }
  }
}

// The Jacobi update of one cell in FP64 from its neighbours' values t0..t5
// (sides not in the grid skipped): (rhs + sum off T_nb) / diag, the right side
// C_p / dt T0 and the couplings k_p / h^2 unless the cell's are stored.  Not
// inlined, and called only by warps with a cell that needs it, so that the
// other warps issue none of its FP64 instructions.
template <bool PHASE>
static __device__ __noinline__ double dif_row(unsigned cls, const double* __restrict__ off6,
                                              const double* __restrict__ rhs_i, const double* __restrict__ diag_i,
                                              double kq, double cdt, double rdt, double T0, double t0, double t1,
                                              double t2, double t3, double t4, double t5) {
  const bool irr = (cls & kDifIrr) != 0, stored = irr || !PHASE;
  double acc = stored ? __ldg(rhs_i) : cdt * T0;
  const double tn[6] = {t0, t1, t2, t3, t4, t5};
#pragma unroll
  for (int f = 0; f < 6; ++f)
    if (cls & (1u << f)) acc = fma(irr ? __ldg(off6 + f) : kq, tn[f], acc);
  return acc * (stored ? __ldg(diag_i) : rdt);
}

// Neighbour index of cell i at (x, y, z) across side f (its class bit set):
// the next cell along the axis, or across a periodic boundary the first or
// last of the line.
__device__ __forceinline__ size_t dif_nb(const GridDev& g, size_t i, int x, int y, int z, int f) {
  const size_t sx = 1, sy = (size_t)g.n[0], sz = (size_t)g.n[0] * g.n[1];
  switch (f) {
    case 0: return x > 0 ? i - sx : i + (size_t)(g.n[0] - 1) * sx;
    case 1: return x < g.n[0] - 1 ? i + sx : i - (size_t)(g.n[0] - 1) * sx;
    case 2: return y > 0 ? i - sy : i + (size_t)(g.n[1] - 1) * sy;
    case 3: return y < g.n[1] - 1 ? i + sy : i - (size_t)(g.n[1] - 1) * sy;
    case 4: return z > 0 ? i - sz : i + (size_t)(g.n[2] - 1) * sz;
    default: return z < g.n[2] - 1 ? i + sz : i - (size_t)(g.n[2] - 1) * sz;
  }
}

// One Jacobi sweep in FP64, Tout = (rhs + sum off T_nb(in)) / diag; with CHECK
// the largest |Tout - Tin| into *change (non-negative doubles order like their
// bits: an integer atomic max, the same whatever the order).  A cell
// coupled by k_p / h^2 whose own and neighbours' values all equal its T0 is
// the sweep's fixed point, (C_p/dt T0 + n k_p/h^2 T0) / (C_p/dt + n k_p/h^2)
// = T0, and keeps T0 without arithmetic.  CTAs of 32 x 8 threads over x and
// y, each walking its share of the z planes (no index division).
template <bool CHECK, bool PHASE>
__global__ void __launch_bounds__(kDifThreads)
k_dif_jacobi(GridDev g, DifVec v, DifConst K, const double* __restrict__ Tin, double* __restrict__ Tout,
             const unsigned long long* __restrict__ prev, double tol, unsigned long long* __restrict__ change) {
  if (dif_done(prev, tol)) return;
  const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 8 + threadIdx.y;
  double dmax = 0.0;
  if (x < g.n[0] && y < g.n[1]) {
    for (int z = blockIdx.z; z < g.n[2]; z += gridDim.z) {
      const size_t i = ((size_t)z * g.n[1] + y) * g.n[0] + x;
      const unsigned cls = __ldg(v.cls + i);
      const double T0 = __ldg(v.T0 + i), tin = Tin[i];
      const long long b0 = dbits(T0);
      double tn[6];
      bool fixed = (cls & kDifIrr) == 0 && dbits(tin) == b0;
#pragma unroll
      for (int f = 0; f < 6; ++f) {
        tn[f] = 0.0;
        if (!(cls & (1u << f))) continue;  // a wall: its coupling is 0
        tn[f] = Tin[dif_nb(g, i, x, y, z, f)];
        fixed = fixed && dbits(tn[f]) == b0;
      }
      double t = T0;
      if (__any_sync(__activemask(), !fixed)) {
        const int li = (cls & kDifLiq) ? 1 : 0;
        const double r = dif_row<PHASE>(cls, v.off + 6 * i, v.rhs + i, v.diag + i, li ? K.kq[1] : K.kq[0],
                                        li ? K.cdt[1] : K.cdt[0], K.rdiag[li][__popc(cls & 63u)], T0, tn[0], tn[1],
                                        tn[2], tn[3], tn[4], tn[5]);
        if (!fixed) t = r;
      }
      Tout[i] = t;
      if (CHECK) dmax = fmax(dmax, fabs(t - tin));
    }
  }
  if constexpr (CHECK) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dmax = fmax(dmax, __shfl_down_sync(0xffffffffu, dmax, o));
    if ((threadIdx.x & 31) == 0 && dnz(dmax)) atomicMax(change, (unsigned long long)dbits(dmax));
  }
}


// The larger of two non-negative pairs (each its high part rounded, so that they
// order by high part, then low part); a NaN is left out.
__device__ __forceinline__ void dif_larger(df::f2& m, df::f2 d) {
  if (d.hi > m.hi || (d.hi == m.hi && d.lo > m.lo)) m = d;
}
// |a - b| of two pairs
__device__ __forceinline__ df::f2 dif_apart(df::f2 a, df::f2 b) {
  df::f2 d = df::two_sum(a.hi, -b.hi);
  d = df::fast_two_sum(d.hi, d.lo + (a.lo - b.lo));
  return d.hi < 0.f ? df::neg(d) : d;
}
// largest change of the warp's lanes (over 2^k) into *change: FP64 bits
__device__ __forceinline__ void dif_change(df::f2 m, int k, unsigned long long* change) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    dif_larger(m, df::f2{__shfl_down_sync(0xffffffffu, m.hi, o), __shfl_down_sync(0xffffffffu, m.lo, o)});
  if ((threadIdx.x & 31) != 0 || !(m.hi > 0.f)) return;
  // (a change near the ends of FP64's range is put together by an addition)
  const double x = k > -800 && k < 800 ? df::widen_pair(m, k) : wide_of(m.hi, k) + wide_of(m.lo, k);
  atomicMax(change, (unsigned long long)dbits(x));
}

// Offsets to a cell's neighbours across the sides in the grid (wrapped across a
// periodic boundary); has: bit f set where side f is in the grid.
struct DifSides {
  long long o[6];
  unsigned has;
};
__device__ __forceinline__ void dif_lateral(const GridDev& g, int x, int y, long long row, DifSides& d) {
  const int nx = g.n[0], ny = g.n[1];
  d.o[0] = x > 0 ? -1 : nx - 1;
  d.o[1] = x < nx - 1 ? 1 : 1 - nx;
  d.o[2] = y > 0 ? -row : (ny - 1) * row;
  d.o[3] = y < ny - 1 ? row : (1 - ny) * row;
  d.has = (x > 0 || g.bc[0] == 0 ? 1u : 0u) | (x < nx - 1 || g.bc[0] == 0 ? 2u : 0u) |
          (y > 0 || g.bc[1] == 0 ? 4u : 0u) | (y < ny - 1 || g.bc[1] == 0 ? 8u : 0u);
}
__device__ __forceinline__ unsigned dif_vertical(const GridDev& g, int z, long long plane, long long (&o)[6]) {
  const int nz = g.n[2];
  o[4] = z > 0 ? -plane : (nz - 1) * plane;
  o[5] = z < nz - 1 ? plane : (1 - nz) * plane;
  return (z > 0 || g.bc[2] == 0 ? 16u : 0u) | (z < nz - 1 || g.bc[2] == 0 ? 32u : 0u);
}

// First sweep in pairs: d = s = B sum (T0_nb - T0) in FP64 (an irregular cell's
// is k_dif_irregular's).  Cells of uniform T take no FP64.
template <bool CHECK>
__global__ void __launch_bounds__(kDifThreads)
k_dif_first(GridDev g, DifVec v, DifConst K, unsigned long long* __restrict__ change) {
  if (v.part[kDifChecks] == 0ull) return;  // not in pairs: s has no place of its own then
  const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 8 + threadIdx.y;
  const bool in = x < g.n[0] && y < g.n[1];
  const long long plane = (long long)g.n[0] * g.n[1];
  const int ks = dif_scale(v, K);
  DifSides sd;
  dif_lateral(g, x, y, g.n[0], sd);
  df::f2 dmax = {0.f, 0.f};
  for (int z = blockIdx.z; z < g.n[2]; z += gridDim.z) {
    const unsigned has = sd.has | dif_vertical(g, z, plane, sd.o);
    const size_t i = in ? ((size_t)z * g.n[1] + y) * g.n[0] + x : 0;
    const unsigned cls = in ? __ldg(v.cls + i) : kDifIrr;
    const bool irr = (cls & kDifIrr) != 0;
    float2 r = make_float2(0.f, 0.f);
    bool vary = false;
    double T0 = 0.0, tn[6];
    if (!irr) T0 = __ldg(v.T0 + i);
#pragma unroll
    for (int f = 0; f < 6; ++f) {
      tn[f] = T0;
      if (!irr && (has & (1u << f))) tn[f] = __ldg(v.T0 + (long long)i + sd.o[f]);
      vary = vary || dbits(tn[f]) != dbits(T0);
    }
    if (__any_sync(0xffffffffu, vary)) {
      double a = tn[0] - T0;
#pragma unroll
      for (int f = 1; f < 6; ++f) a += tn[f] - T0;
      const double sv = a * K.B[(cls & kDifLiq) ? 1 : 0][__popc(cls & 63u)];
      if (vary) r = pair_of(sv, ks);
    }
    if (in) {
      float* const at = part_of(g, v, v.s, x, y, z);
      if (!irr) {
        at[0] = r.x;
        at[2] = r.y;
      } else if (CHECK) {
        r = make_float2(at[0], at[2]);
      }
    }
    if (CHECK) dif_larger(dmax, dif_apart(f2_of(r), df::f2{0.f, 0.f}));
  }
  if constexpr (CHECK) dif_change(dmax, ks, change);
}

// One later sweep in pairs, d' = sum B_nb d_nb + s, two cells of a row
// per thread: every packed instruction serves both.  A cell whose own s and
// neighbours' d are all 0 keeps 0 without arithmetic.  (z walked in consecutive
// planes held in registers, for a third of the reads of d, took 25 us at 128^3
// against 22: the loads' latency bounds it, and that form keeps fewer warps.)
template <bool CHECK>
__global__ void __launch_bounds__(kDifThreads)
k_dif_sweep(GridDev g, DifVec v, DifConst K, const float4* __restrict__ din, float4* __restrict__ dout,
            const unsigned long long* __restrict__ prev, double tol, unsigned long long* __restrict__ change) {
  pdl_wait();
  using namespace df;
  din = after_wait(din);
  v.s = after_wait(v.s);
  if (dif_done(after_wait(prev), tol)) return;
  const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
  const int xb = blockIdx.x * 32 + threadIdx.x, x = 2 * xb, y = blockIdx.y * 8 + threadIdx.y;
  const bool in = x < nx && y < ny, in1 = x + 1 < nx && y < ny;
  const int row = v.px;
  const long long plane = (long long)row * ny;
  // sides of the pair: the outer x neighbours, y and z (those two cells share)
  const bool wrap = g.bc[0] == 0;
  const bool hasL = x > 0 || wrap, hasR = (in1 ? x + 1 : x) < nx - 1 || wrap;
  const int oL = x > 0 ? -1 : (nx - 1) >> 1, oR = x + 2 < nx ? 1 : -xb;  // blocks of the outer neighbours
  const bool oddL = x > 0 || (nx & 1) == 0;                             // and L's place in its block (R's is the first)
  const bool hasS = y > 0 || g.bc[1] == 0, hasN = y < ny - 1 || g.bc[1] == 0;
  const long long oS = y > 0 ? -row : (ny - 1) * (long long)row, oN = y < ny - 1 ? row : (1 - ny) * (long long)row;
  f2 dmax = {0.f, 0.f};
  for (int z = blockIdx.z; z < nz; z += gridDim.z) {
    const bool hasB = z > 0 || g.bc[2] == 0, hasT = z < nz - 1 || g.bc[2] == 0;
    const long long oB = z > 0 ? -plane : (nz - 1) * plane, oT = z < nz - 1 ? plane : (1 - nz) * plane;
    const long long ip = in ? z * plane + (long long)y * row + xb : 0;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    auto at = [&](const float4* a, bool ok, long long o) { return ok ? __ldg(a + ip + o) : zero; };
    const float4 s4 = at(v.s, in, 0);
    float4 c4 = at(din, in, 0);
    if (!in1) c4.y = c4.w = 0.f;  // (the padding)
    const float4 S4 = at(din, in && hasS, oS), N4 = at(din, in && hasN, oN);
    const float4 B4 = at(din, in && hasB, oB), T4 = at(din, in && hasT, oT);
    const float4 L4 = at(din, in && hasL, oL), R4 = at(din, in && hasR, oR);
    const float2 sh = make_float2(s4.x, s4.y), sl = make_float2(s4.z, s4.w);
    const float2 ch = make_float2(c4.x, c4.y), cl = make_float2(c4.z, c4.w);
    const float2 Sh = make_float2(S4.x, S4.y), Sl = make_float2(S4.z, S4.w);
    const float2 Nh = make_float2(N4.x, N4.y), Nl = make_float2(N4.z, N4.w);
    const float2 Bh = make_float2(B4.x, B4.y), Bl = make_float2(B4.z, B4.w);
    const float2 Th = make_float2(T4.x, T4.y), Tl = make_float2(T4.z, T4.w);
    const float Lh = oddL ? L4.y : L4.x, Ll = oddL ? L4.w : L4.z;
    const float Rh = R4.x, Rl = R4.z;
    const size_t ic = ((size_t)z * ny + y) * nx + x;
    const unsigned c0 = in ? __ldg(v.cls + ic) : 0u;
    const unsigned c1 = in1 ? __ldg(v.cls + ic + 1) : 0u;
    auto fb = [](float f) { return __float_as_uint(f); };
    // (a pair's high part is 0 exactly where the pair is; the padding's values
    // reach no cell)
    const unsigned any = (fb(sh.x) | fb(ch.x) | fb(Sh.x) | fb(Nh.x) | fb(Bh.x) | fb(Th.x) | fb(Lh) | fb(Rh) |
                          (in1 ? fb(sh.y) | fb(ch.y) | fb(Sh.y) | fb(Nh.y) | fb(Bh.y) | fb(Th.y) : 0u)) & 0x7FFFFFFFu;
    float2 rh = make_float2(0.f, 0.f), rl = rh;
    const bool work = __any_sync(0xffffffffu, any != 0u);
    if (work) {
      // left and right neighbours of both cells: (L, c0), (c1, R); a lone last
      // cell's right neighbour is R
      const f2x2 W = {vset(Lh, ch.x), vset(Ll, cl.x)};
      const f2x2 E = {vset(in1 ? ch.y : Rh, Rh), vset(in1 ? cl.y : Rl, Rl)};
      f2x2 t = two_sum(W.hi, E.hi);
      v2 lo = vadd(vadd(W.lo, E.lo), t.lo);
      auto more = [&](float2 h, float2 l) {
        t = two_sum(t.hi, vset(h.x, h.y));
        lo = vadd(lo, vadd(vset(l.x, l.y), t.lo));
      };
      more(Sh, Sl);
      more(Nh, Nl);
      more(Bh, Bl);
      more(Th, Tl);
      const float2 B0 = K.Bf[(c0 & kDifLiq) ? 1 : 0][__popc(c0 & 63u)], B1 = K.Bf[(c1 & kDifLiq) ? 1 : 0][__popc(c1 & 63u)];
      const f2x2 r = add_c(mul(fast_two_sum(t.hi, lo), f2x2{vset(B0.x, B1.x), vset(B0.y, B1.y)}),
                           f2x2{vset(sh.x, sh.y), vset(sl.x, sl.y)});
      vget(r.hi, rh.x, rh.y);
      vget(r.lo, rl.x, rl.y);
      if (__any_sync(0xffffffffu, ((c0 | c1) & kDifIrr) != 0u)) {
        // cells next to the interface or a heated wall: their own couplings
        const float2 n0[6] = {make_float2(Lh, Ll), in1 ? make_float2(ch.y, cl.y) : make_float2(Rh, Rl),
                              make_float2(Sh.x, Sl.x), make_float2(Nh.x, Nl.x), make_float2(Bh.x, Bl.x), make_float2(Th.x, Tl.x)};
        const float2 n1[6] = {make_float2(ch.x, cl.x), make_float2(Rh, Rl), make_float2(Sh.y, Sl.y),
                              make_float2(Nh.y, Nl.y), make_float2(Bh.y, Bl.y), make_float2(Th.y, Tl.y)};
        f2 e0 = f2{sh.x, sl.x}, e1 = f2{sh.y, sl.y};
        const float2* off = reinterpret_cast<const float2*>(v.off) + 6 * ic;
#pragma unroll
        for (int f = 0; f < 6; ++f) {
          if ((c0 & kDifIrr) && (c0 & (1u << f))) e0 = add_c(mul(f2_of(__ldg(off + f)), f2_of(n0[f])), e0);
          if ((c1 & kDifIrr) && (c1 & (1u << f))) e1 = add_c(mul(f2_of(__ldg(off + 6 + f)), f2_of(n1[f])), e1);
        }
        if (c0 & kDifIrr) { rh.x = e0.hi; rl.x = e0.lo; }
        if (c1 & kDifIrr) { rh.y = e1.hi; rl.y = e1.lo; }
      }
    }
    if (in) dout[ip] = make_float4(rh.x, rh.y, rl.x, rl.y);
    if (CHECK && work) {
      dif_larger(dmax, dif_apart(f2{rh.x, rl.x}, f2{ch.x, cl.x}));
      if (in1) dif_larger(dmax, dif_apart(f2{rh.y, rl.y}, f2{ch.y, cl.y}));
    }
  }
  if constexpr (CHECK) dif_change(dmax, dif_scale(v, K), change);
}

// e' = e + C_p,node d; a node without change keeps its e
__global__ void __launch_bounds__(kDifThreads)
k_dif_store_pairs(GridDev g, const DifVec v, DifConst K, float4* d, double* __restrict__ e) {
  const int ks = dif_scale(v, K);
  const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 8 + threadIdx.y;
  if (x >= g.n[0] || y >= g.n[1]) return;
  for (int z = blockIdx.z; z < g.n[2]; z += gridDim.z) {
    const size_t i = ((size_t)z * g.n[1] + y) * g.n[0] + x;
    const float* const at = part_of(g, v, d, x, y, z);
    const float hi = at[0], lo = at[2];
    if (hi == 0.f && lo == 0.f) continue;
    const double Cd = (__ldg(v.cls + i) & kDifLiq) ? g.Cp_l : g.Cp_g;
    e[i] = e[i] + Cd * (wide_of(hi, ks) + wide_of(lo, ks));
  }
}

// From an iterate in FP64: e' = e + C_p,node (T' - T0) (phase; a node whose T came
// back unchanged keeps its e), e' = C_p(c) T' (mixture)
template <bool PHASE>
__global__ void k_dif_store(GridDev g, const double* __restrict__ c, const DifVec v, const double* __restrict__ T,
                            double* __restrict__ e, size_t N) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x) {
    if constexpr (PHASE) {
      const double Tn = T[i], T0 = __ldg(v.T0 + i);
      if (dbits(Tn) == dbits(T0)) continue;
      e[i] = e[i] + ((__ldg(v.cls + i) & kDifLiq) ? g.Cp_l : g.Cp_g) * (Tn - T0);
      continue;
    }
    const double cv = __ldg(c + i);
    const double Cp = g.Cp_l * cv + g.Cp_g * (1.0 - cv);
    e[i] = Cp * T[i];
  }
}

struct DifLayout {
  size_t plane, off, diag, rhs, T0, Ta, Tb, part, cls, mlist, count, total;
};

DifLayout dif_layout(size_t N) {
  auto a = [](size_t b) { return (b + 255) & ~(size_t)255; };
  DifLayout L;
  size_t o = 0;
  L.plane = o; o += a(N * 32);
  L.off = o; o += a(N * 6 * 8);
  L.diag = o; o += a(N * 8);
  L.rhs = o; o += a(N * 8);
  L.T0 = o; o += a(N * 8);
  L.Ta = o; o += a(N * 8);
  L.Tb = o; o += a(N * 8);
  L.part = o; o += a((kDifChecks + 1) * 8);  // the checks' largest changes (bits of non-negative doubles)
  L.cls = o; o += a(N);
  L.mlist = o; o += a(N * 4);
  L.count = o; o += 256;
  L.total = o;
  return L;
}

}  // namespace

size_t dif_scratch_bytes(size_t N) { return dif_layout(N).total; }

cudaError_t launch_heat_diffusion(const GridDev& g, double h, const double* c, double* e, double k_l, double k_g,
                                  double dt, double tol, int max_iter, int phase_cp, const double* wall_T,
                                  void* workspace, cudaStream_t st, int* iters_out, double* change_out,
                                  int* status) {
  const size_t N = (size_t)g.n[0] * g.n[1] * g.n[2];
  const DifLayout L = dif_layout(N);
  char* ws = static_cast<char*>(workspace);
  double4* plane = reinterpret_cast<double4*>(ws + L.plane);
  DifVec v;
  v.off = reinterpret_cast<double*>(ws + L.off);
  v.diag = reinterpret_cast<double*>(ws + L.diag);
  v.rhs = reinterpret_cast<double*>(ws + L.rhs);
  v.T0 = reinterpret_cast<double*>(ws + L.T0);
  v.Ta = reinterpret_cast<double*>(ws + L.Ta);
  v.Tb = reinterpret_cast<double*>(ws + L.Tb);
  v.part = reinterpret_cast<unsigned long long*>(ws + L.part);
  v.cls = reinterpret_cast<uint8_t*>(ws + L.cls);
  // the pairs' blocks (up to two cell arrays each): s in diag's and rhs's
  // place, the iterates in the planes' (not read any more when they are written)
  v.px = (g.n[0] + 1) / 2;
  const size_t pn = (size_t)v.px * g.n[1] * g.n[2];
  v.s = reinterpret_cast<float4*>(ws + L.diag);
  v.d[0] = reinterpret_cast<float4*>(ws + L.plane);
  v.d[1] = v.d[0] + pn;
  uint32_t* mlist = reinterpret_cast<uint32_t*>(ws + L.mlist);
  int* count = reinterpret_cast<int*>(ws + L.count);
  v.range = count + 2;
  *status = 0;
  const int grid = (int)std::min<size_t>((N + kDifThreads - 1) / kDifThreads, (size_t)kDifCTAs);
  cudaError_t err = cudaMemsetAsync(count, 0, 4 * sizeof(int), st);
  if (err != cudaSuccess) return err;
  k_dif_mlist<<<grid, kDifThreads, 0, st>>>(g, c, mlist, count, N);
  k_dif_planes<<<kDifCTAs, kDifPlaneThreads, 0, st>>>(g, c, mlist, count, plane);
  prof_mark("diffuse.planes", st);
  DifWalls walls;
  for (int f = 0; f < 6; ++f) {
    walls.on[f] = wall_T && wall_T[f] == wall_T[f] ? 1 : 0;  // NaN: no wall temperature
    walls.T[f] = walls.on[f] ? wall_T[f] : 0.0;
  }
  // the per-phase constants, in the order of the per-cell assembly
  const double inv_h = 1.0 / h, inv_dt = 1.0 / dt;
  DifConst K;
  const double kp[2] = {k_g, k_l}, Cph[2] = {g.Cp_g, g.Cp_l};
  for (int p = 0; p < 2; ++p) {
    K.kq[p] = kp[p] * (inv_h * inv_h);
    K.cdt[p] = Cph[p] * inv_dt;
    double d = K.cdt[p];
    for (int n = 0; n <= 6; ++n) {
      K.rdiag[p][n] = 1.0 / d;
      K.B[p][n] = K.kq[p] * K.rdiag[p][n];
      K.Bf[p][n].x = (float)K.B[p][n];
      K.Bf[p][n].y = (float)(K.B[p][n] - (double)K.Bf[p][n].x);
      d += K.kq[p];
    }
  }
  K.wlo = 0x7FFFFFFF;
  K.whi = 0;
  for (int f = 0; f < 6; ++f) {
    if (!walls.on[f]) continue;
    long long b;
    std::memcpy(&b, &walls.T[f], sizeof(b));
    K.wlo = std::min(K.wlo, (int)(b >> 32));
    K.whi = std::max(K.whi, (int)(b >> 32));
  }
  // the cells next to the interface or a heated wall are listed in the
  // mixed-cell list's storage (k_dif_planes is done with it)
  uint32_t* ilist = mlist;
  const dim3 sgrid = dif_sweep_grid(g);
  if (phase_cp) k_dif_classify<true><<<sgrid, dim3(32, 8), 0, st>>>(g, c, e, v, walls, inv_dt, K, ilist, count + 1);
  else k_dif_classify<false><<<sgrid, dim3(32, 8), 0, st>>>(g, c, e, v, walls, inv_dt, K, ilist, count + 1);
  k_dif_irregular<<<kDifCTAs, kDifPlaneThreads, 0, st>>>(g, h, inv_h, inv_dt, k_l, k_g, c, e, plane, v, walls, phase_cp, K,
                                                 ilist, count + 1);
  prof_mark("diffuse.assemble", st);
  // Sweeps in batches, each with its checks' slots cleared first: a sweep
  // queued behind a check that was within tol returns at once (its slot stays
  // 0, so the ones behind it do too), and the host reads a batch's slots
  // together.  The batches grow, cut short where the last checks' rate says
  // when tol will be met.
  unsigned long long* slot = v.part;
  // the iterates: T0, then Ta and Tb in turn (in pairs: s, the first sweep's
  // result, then d[0] and d[1])
  double* buf[2] = {v.Ta, v.Tb};
  int it = 0, batch = 2;
  bool pairs = phase_cp != 0;  // until the first batch's results say otherwise
  double change = 0.0, before = 0.0;
  bool done = false;
  auto iterate = [&](int n) -> double* { return n == 0 ? v.T0 : buf[n & 1]; };  // the n-th sweep's result
  auto iterate_d = [&](int n) -> float4* { return n <= 1 ? v.s : v.d[n & 1]; };
  // two cells of a row per thread
  const dim3 pgrid((unsigned)((g.n[0] + 63) / 64), sgrid.y,
                   (unsigned)std::max(1, std::min(g.n[2], (int)(152u * 16u / std::max(1u, (unsigned)((g.n[0] + 63) / 64) * sgrid.y)))));
  while (!done && it < max_iter) {
    err = cudaMemsetAsync(slot, 0, kDifChecks * sizeof(unsigned long long), st);
    if (err != cudaSuccess) return err;
    int nc = 0;
    const unsigned long long* prev = pairs && it == 0 ? slot + kDifChecks : nullptr;
    int at[kDifChecks];
    while (it < max_iter && nc < batch) {
      const bool check = (it + 1) % 4 == 0 || it + 1 == max_iter;
      unsigned long long* chg = check ? slot + nc : nullptr;
      const double* in = iterate(it);
      double* out = iterate(it + 1);
      if (pairs && it == 0) {
        if (check) k_dif_first<true><<<sgrid, dim3(32, 8), 0, st>>>(g, v, K, chg);
        else k_dif_first<false><<<sgrid, dim3(32, 8), 0, st>>>(g, v, K, chg);
      } else if (pairs) {
        const float4* di = iterate_d(it);
        float4* dd = iterate_d(it + 1);
        if (check) launch_pdl(k_dif_sweep<true>, pgrid, dim3(32, 8), st, g, v, K, di, dd, prev, tol, chg);
        else launch_pdl(k_dif_sweep<false>, pgrid, dim3(32, 8), st, g, v, K, di, dd, prev, tol, chg);
      } else {
        auto sweep = phase_cp ? (check ? k_dif_jacobi<true, true> : k_dif_jacobi<false, true>)
                              : (check ? k_dif_jacobi<true, false> : k_dif_jacobi<false, false>);
        sweep<<<sgrid, dim3(32, 8), 0, st>>>(g, v, K, in, out, prev, tol, chg);
      }
      ++it;
      if (check) {
        at[nc] = it;
        prev = slot + nc++;
      }
    }
    unsigned long long hb[kDifChecks + 1];
    err = cudaMemcpyAsync(hb, slot, sizeof(hb), cudaMemcpyDeviceToHost, st);
    if (err == cudaSuccess) err = cudaStreamSynchronize(st);
    if (err != cudaSuccess) return err;
    if (pairs && hb[kDifChecks] == 0ull) {  // nothing has run: from the start, in FP64
      pairs = false;
      it = 0;
      continue;
    }
    for (int k = 0; k < nc && !done; ++k) {
      before = change;
      std::memcpy(&change, &hb[k], sizeof(change));
      done = change <= tol;
      if (done) it = at[k];
    }
    batch = batch * 2 < kDifChecks ? batch * 2 : kDifChecks;
    if (!done && change > 0.0 && before > change) {
      // checks until tol at the last pair's rate
      const double more = std::log(change / tol) / std::log(before / change);
      if (more + 1.0 < (double)batch) batch = (int)more + 1;
    }
  }
  prof_mark("diffuse.jacobi", st);
  if (!done) *status = 2;
  if (pairs) k_dif_store_pairs<<<sgrid, dim3(32, 8), 0, st>>>(g, v, K, iterate_d(it), e);
  else if (phase_cp) k_dif_store<true><<<grid, kDifThreads, 0, st>>>(g, c, v, iterate(it), e, N);
  else k_dif_store<false><<<grid, kDifThreads, 0, st>>>(g, c, v, iterate(it), e, N);
  prof_mark("diffuse.store", st);
  if (iters_out) *iters_out = it;
  if (change_out) *change_out = change;
  return cudaGetLastError();
}

}  // namespace vofgb
