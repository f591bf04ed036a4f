// vof_mdot.cu -- mass transfer rate from PLIC interface distances (Malan et
// al., arXiv:2001.03477, Sec. 3.2 "Calculating the mass transfer rate":
// Eqs. mdot_calc, grad_n_T, plane_m, cell_d, dint_trans, the collinearity
// xi, normTgrad and the weights chi, gamma).
//
// For every mixed cell M the plane is put in Hessian form: unit normal
// n = m / |m| (m the MYC normal, pointing from liquid into gas) and distance
// d = alpha / |m| from M's low corner (Eq. cell_d).  Every pure cell P within
// two cells of a mixed cell (Chebyshev distance <= 2, the 3D reading of the
// 5 x 5 stencil) takes, among its mixed neighbours, the one of largest
// collinearity xi = |n . dx| (dx from that neighbour's low corner to P's
// centre; the first in z-, y-, x-order on ties) and the normal distance
// |d_Gamma| = |d - n . dx| h (Eq. dint_trans); its temperature gradient
// along n is (T_Gamma - T) / |d_Gamma| on the liquid side and
// (T - T_Gamma) / |d_Gamma| on the gas side (Eq. grad_n_T with n pointing
// into the gas).  Each mixed cell averages its pure neighbours' gradients
// per phase with weights gamma = |n . dx| / |dx|^2, dx the offset between
// the two centres (Eq. normTgrad), and mdot = (k_g grad_g - k_l grad_l) /
// h_fg (Eq. mdot_calc).  On a zero-gradient axis, offsets that leave the
// grid are not cells; periodic axes wrap.
//
// Five kernels, all over compact lists except the first:
//   k_md_list    stream c once: zero the outputs, list the mixed cells;
//   k_md_planes  a thread per mixed cell: MYC normal, plane constant (FP64),
//                Hessian plane;
//   k_md_band    a warp per mixed cell, its lanes over the 124 offsets: the
//                pure neighbours join the band (an atomic OR on one bit per
//                cell; the lane that sets the bit lists the cell);
//   k_md_grad    a warp per band cell: the most collinear mixed neighbour's
//                plane (warp argmax), |d_Gamma|, grad_n T;
//   k_md_avg     a warp per mixed cell: the weighted averages (lane sums and
//                a shuffle tree) and mdot.
// A warp per stencil spreads the 124 dependent neighbour loads over 32
// lanes: the lists are short (1e4-1e5 cells) and a thread per cell walking
// its 124 neighbours leaves the GPU waiting on load latency.  What the warps issue
// besides is kept short: a lane's four offsets (and their values as FP64 numbers,
// from shared memory: a constant array read at 32 different indices is read
// once per index) are formed once per warp, a neighbour of a cell away from the
// boundary is one addition, the argmax reduces 32-bit words, and the averages'
// four sums fold into 6 additions instead of 20 (an FP64 instruction takes 76
// cycles of an SM partition).  At 256^3 with 10,709 mixed and 46,885 band cells:
// band 24 -> 19 us, grad 60 -> 47 us, avg 69 -> 43 us.
#include <algorithm>

#include "../../include/vofgb.h"
#include "vof_launch.h"

namespace vofgb {

namespace {

constexpr int kMdThreads = 128;
constexpr int kMdCTAs = 152 * 8;
constexpr int kListThreads = 256;

// a gradient that does not exist (a node on its plane): a quiet NaN pattern,
// tested on the integer pipe
constexpr long long kNoGrad = 0x7FF8DEAD00000000LL;

// small FP64 tables, copied to shared memory by each CTA: 0.5 - d for the
// offsets d = -2 .. 2 (the node of a cell at offset -d from a mixed cell, from
// that cell's low corner), the offsets themselves, and 1 / |dx|^2 for the squared
// offsets 0 .. 12 of the 5 x 5 x 5 stencil
__constant__ double c_half_minus[5] = {2.5, 1.5, 0.5, -0.5, -1.5};
__constant__ double c_off[5] = {-2.0, -1.0, 0.0, 1.0, 2.0};
__constant__ double c_rinv[13] = {0.0, 1.0, 0.5, 1.0 / 3.0, 0.25, 0.2, 1.0 / 6.0, 0.0, 0.125, 1.0 / 9.0, 0.0, 0.0,
                                  1.0 / 12.0};

// per axis: the neighbour coordinate of offset o in [-2, 2], or -1 where a
// zero-gradient axis has no cell
__device__ __forceinline__ int nb_coord(int x, int o, int n, int bc) {
  const int p = x + o;
  if (bc == 0) {
    int r = p % n;
    return r < 0 ? r + n : r;
  }
  return (p < 0 || p >= n) ? -1 : p;
}

__device__ __forceinline__ size_t nb_id(const GridDev& g, int x, int y, int z) {
  return ((size_t)z * g.n[1] + y) * g.n[0] + x;
}

// grid-wide list append, one atomic per warp
__device__ __forceinline__ void warp_append(bool take, uint32_t v, uint32_t* list, int* counter) {
  const unsigned mask = __ballot_sync(0xffffffffu, take);
  if (!mask) return;
  const int lane = threadIdx.x & 31;
  int base = 0;
  if (lane == __ffs(mask) - 1) base = atomicAdd(counter, __popc(mask));
  base = __shfl_sync(0xffffffffu, base, __ffs(mask) - 1);
  if (take) list[base + __popc(mask & ((1u << lane) - 1u))] = v;
}

__global__ void __launch_bounds__(kListThreads)
k_md_list(GridDev g, const double* __restrict__ c, double* __restrict__ mdot, double* __restrict__ d_gamma,
          double* __restrict__ grad_n, double* __restrict__ dd, uint32_t* __restrict__ mlist,
          int* __restrict__ counters, size_t N) {
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  // whole warps iterate together (the append is warp-collective)
  const size_t n_iter = (N + stride - 1) / stride;
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (size_t it = 0; it < n_iter; ++it, i += stride) {
    const bool in = i < N;
    bool mx = false;
    if (in) {
      mx = is_mixed_b(__ldg(c + i), g);
      mdot[i] = 0.0;
      if (d_gamma) d_gamma[i] = -1.0;
      if (grad_n) grad_n[i] = 0.0;
      if (dd) dd[i] = 0.0;
    }
    warp_append(mx, (uint32_t)i, mlist, counters);
  }
}

__global__ void __launch_bounds__(kMdThreads)
k_md_planes(GridDev g, const double* __restrict__ c, const uint32_t* __restrict__ mlist,
            const int* __restrict__ counters, double4* __restrict__ plane) {
  pdl_wait();
  mlist = after_wait(mlist);
  const int nm = *after_wait(counters);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nm; i += gridDim.x * blockDim.x) {
    const uint32_t id = mlist[i];
    int x, y, z;
    cell_xyz(g, id, x, y, z);
    double s[27];
#pragma unroll
    for (int oz = 0; oz < 3; ++oz) {
      const int zz = map_idx(z + oz - 1, g.n[2], g.bc[2]);
#pragma unroll
      for (int oy = 0; oy < 3; ++oy) {
        const int yy = map_idx(y + oy - 1, g.n[1], g.bc[1]);
#pragma unroll
        for (int ox = 0; ox < 3; ++ox) {
          const int xx = map_idx(x + ox - 1, g.n[0], g.bc[0]);
          s[(oz * 3 + oy) * 3 + ox] = __ldg(c + nb_id(g, xx, yy, zz));
        }
      }
    }
    double m[3];
    myc_normal(s, m);
    const double al = plane_alpha(m[0], m[1], m[2], s[13]);
    const double len = sqrt(m[0] * m[0] + m[1] * m[1] + m[2] * m[2]);
    double4 p;
    p.x = m[0] / len;
    p.y = m[1] / len;
    p.z = m[2] / len;
    p.w = al / len;
    plane[id] = p;
  }
}

// The 124 offsets of the 5 x 5 x 5 stencil (all but the centre, index 62)
// are spread over a warp's lanes: lane l takes the indices l, l + 32, l + 64
// and l + 96 below 125, in increasing order; index o is the offset
// (o % 5 - 2, o / 5 % 5 - 2, o / 25 - 2), so increasing indices visit z
// outer, then y, then x.
constexpr int kOffRounds = 4;

// the neighbour of (x, y, z) at offset (dx, dy, dz), or -1 (off a zero-gradient
// axis)
__device__ __forceinline__ long long stencil_nb(const GridDev& g, int x, int y, int z, int dx, int dy, int dz) {
  const int xx = nb_coord(x, dx, g.n[0], g.bc[0]);
  const int yy = nb_coord(y, dy, g.n[1], g.bc[1]);
  const int zz = nb_coord(z, dz, g.n[2], g.bc[2]);
  if (xx < 0 || yy < 0 || zz < 0) return -1;
  return (long long)nb_id(g, xx, yy, zz);
}

// A lane's offsets, one per round: dx + 2, dy + 2, dz + 2 in bytes 0..2 of at (a
// round without an offset -- the centre, or past 124: byte 3 set), and the
// cell's distance in the arrays.
struct LaneOffsets {
  unsigned at[kOffRounds];
  int step[kOffRounds];
};
__device__ __forceinline__ LaneOffsets lane_offsets(const GridDev& g, int lane) {
  LaneOffsets L;
#pragma unroll
  for (int r = 0; r < kOffRounds; ++r) {
    const int o = lane + 32 * r, ox = o % 5, oy = (o / 5) % 5, oz = o / 25;
    L.at[r] = (unsigned)(ox | (oy << 8) | (oz << 16)) | (o >= 125 || o == 62 ? 1u << 24 : 0u);
    L.step[r] = ((oz - 2) * g.n[1] + (oy - 2)) * g.n[0] + (ox - 2);
  }
  return L;
}
// The neighbour of cell id at the lane's offset of round r, or -1.  inner: the
// cell is two or more cells from every side of the grid (the same for the whole
// warp).
__device__ __forceinline__ bool inner_cell(const GridDev& g, int x, int y, int z) {
  return x >= 2 && y >= 2 && z >= 2 && x < g.n[0] - 2 && y < g.n[1] - 2 && z < g.n[2] - 2;
}
__device__ __forceinline__ long long lane_nb(const GridDev& g, const LaneOffsets& L, int r, uint32_t id, bool inner,
                                             int x, int y, int z) {
  if (L.at[r] >> 24) return -1;
  if (inner) return (long long)id + L.step[r];
  return stencil_nb(g, x, y, z, (int)(L.at[r] & 0xFFu) - 2, (int)((L.at[r] >> 8) & 0xFFu) - 2,
                    (int)((L.at[r] >> 16) & 0xFFu) - 2);
}

// one warp per mixed cell: its pure neighbours join the band; the lane that
// sets a cell's bit lists it
__global__ void __launch_bounds__(kMdThreads)
k_md_band(GridDev g, const double* __restrict__ c, const uint32_t* __restrict__ mlist, uint32_t* __restrict__ blist,
          int* __restrict__ counters, uint32_t* __restrict__ bits) {
  pdl_wait();
  mlist = after_wait(mlist);
  const int nm = *after_wait(counters);
  const int lane = threadIdx.x & 31;
  const int nwarps = (gridDim.x * blockDim.x) >> 5;
  const LaneOffsets L = lane_offsets(g, lane);
  for (int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < nm; i += nwarps) {
    int x, y, z;
    const uint32_t id = mlist[i];
    cell_xyz(g, id, x, y, z);
    const bool inner = inner_cell(g, x, y, z);
    // all rounds' loads, then their atomics, then one append (its lists' order
    // is free)
    long long q[kOffRounds];
    bool pure[kOffRounds];
#pragma unroll
    for (int r = 0; r < kOffRounds; ++r) {
      q[r] = lane_nb(g, L, r, id, inner, x, y, z);
      pure[r] = q[r] >= 0 && !is_mixed_b(__ldg(c + (q[r] < 0 ? 0 : q[r])), g);
    }
    unsigned mine = 0u;
#pragma unroll
    for (int r = 0; r < kOffRounds; ++r) {
      if (!pure[r]) continue;
      // (most cells were listed by a neighbour: a plain read spares the atomic)
      const uint32_t bit = 1u << ((uint32_t)q[r] & 31u);
      uint32_t* w = bits + (q[r] >> 5);
      if ((__ldcg(w) & bit) == 0u && (atomicOr(w, bit) & bit) == 0u) mine |= 1u << r;
    }
    const int k = __popc(mine);
    int pre = k;  // inclusive prefix over the lanes
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, pre, o);
      if (lane >= o) pre += t;
    }
    const int total = __shfl_sync(0xffffffffu, pre, 31);
    if (total == 0) continue;
    int base = 0;
    if (lane == 0) base = atomicAdd(counters + 1, total);
    int at = __shfl_sync(0xffffffffu, base, 0) + pre - k;
#pragma unroll
    for (int r = 0; r < kOffRounds; ++r)
      if ((mine >> r) & 1u) blist[at++] = (uint32_t)q[r];
  }
}

// A warp takes kBatch consecutive list entries at a time and treats them
// one after the other, all lanes on one stencil; lane j keeps the result of
// entry j, and the per-cell tail (FP64 divisions) then runs on kBatch lanes
// at once.  Band cells 8 and mixed cells 4 at a time: enough lanes to share the
// divisions, enough warps to hide the neighbour loads (1e4 mixed cells are 2700
// warps, 4 per SM partition).
constexpr int kMdWarps = kMdThreads / 32;
constexpr int kBatchGrad = 8, kBatchAvg = 4;

// one warp per band cell: the mixed neighbour of largest xi (the lowest
// stencil index on ties), |d_Gamma| and grad_n T.  The mixed neighbours are
// first compacted in stencil-index order into the warp's slots, so the FP64
// evaluation of xi runs lane-dense (one round for up to 32 of them).
__global__ void __launch_bounds__(kMdThreads)
k_md_grad(GridDev g, double h, const double* __restrict__ c, const double* __restrict__ e,
          const uint32_t* __restrict__ blist, const int* __restrict__ counters, const double4* __restrict__ plane,
          double* __restrict__ grad, double* __restrict__ d_gamma, double* __restrict__ grad_n) {
  __shared__ uint32_t s_q[kMdWarps][kOffRounds * 32];
  __shared__ unsigned char s_o[kMdWarps][kOffRounds * 32];
  __shared__ double s_half[5];
  pdl_wait();
  blist = after_wait(blist);
  counters = after_wait(counters);
  plane = after_wait(plane);
  if (threadIdx.x < 5) s_half[threadIdx.x] = c_half_minus[threadIdx.x];
  __syncthreads();
  const int nb_count = counters[1];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int nwarps = (gridDim.x * blockDim.x) >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const LaneOffsets L = lane_offsets(g, lane);
  // n . dx, dx from the mixed cell's low corner to the centre of the cell at
  // stencil index o from it
  auto along = [&](const double4& p, int o) {
    return (p.x * s_half[o % 5] + p.y * s_half[(o / 5) % 5]) + p.z * s_half[o / 25];
  };
  for (int b0 = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * kBatchGrad; b0 < nb_count; b0 += nwarps * kBatchGrad) {
    const int nj = min(kBatchGrad, nb_count - b0);
    const uint32_t my_id = lane < nj ? blist[b0 + lane] : 0u;
    uint32_t my_q = 0u;  // the most collinear mixed neighbour
    int my_o = 0;
    for (int j = 0; j < nj; ++j) {
      const uint32_t id = __shfl_sync(0xffffffffu, my_id, j);
      int x, y, z;
      cell_xyz(g, id, x, y, z);
      const bool inner = inner_cell(g, x, y, z);
      long long q[kOffRounds];
      bool mx[kOffRounds];
#pragma unroll
      for (int r = 0; r < kOffRounds; ++r) {
        q[r] = lane_nb(g, L, r, id, inner, x, y, z);
        mx[r] = q[r] >= 0 && is_mixed_b(__ldg(c + (q[r] < 0 ? 0 : q[r])), g);
      }
      // compact the mixed neighbours, in increasing stencil index
      int n = 0;
#pragma unroll
      for (int r = 0; r < kOffRounds; ++r) {
        const unsigned bm = __ballot_sync(0xffffffffu, mx[r]);
        if (mx[r]) {
          s_q[wib][n + __popc(bm & lt)] = (uint32_t)q[r];
          s_o[wib][n + __popc(bm & lt)] = (unsigned char)(lane + 32 * r);
        }
        n += __popc(bm);
      }
      __syncwarp();
      // this lane's best over its slots (increasing index: the first wins
      // ties): xi bits (non-negative doubles order as integers), stencil index
      long long bxi = -1;
      int bo = 255;
      uint32_t bq = 0u;
      for (int k = lane; k < n; k += 32) {
        const int o = s_o[wib][k];
        const uint32_t qk = s_q[wib][k];
        const long long xb = dbits(along(plane[qk], o)) & 0x7FFFFFFFFFFFFFFFll;
        if (xb > bxi) {
          bxi = xb;
          bo = o;
          bq = qk;
        }
      }
      __syncwarp();
      // warp argmax: largest xi (high word, then low word), then lowest stencil
      // index (band cells have a mixed neighbour, so some lane holds one)
      const int hi = (int)(bxi >> 32);
      // (every lane takes part in each reduction)
      const int hi1 = __reduce_max_sync(0xffffffffu, hi);
      const unsigned lo = hi == hi1 ? (unsigned)bxi : 0u;
      const unsigned lo1 = __reduce_max_sync(0xffffffffu, lo);
      const bool best = hi == hi1 && lo == lo1;
      const int o1 = __reduce_min_sync(0xffffffffu, best ? bo : 256);
      const unsigned who = __ballot_sync(0xffffffffu, best && bo == o1);
      const uint32_t q1 = __shfl_sync(0xffffffffu, bq, __ffs(who) - 1);
      if (lane == j) {
        my_q = q1;
        my_o = o1;
      }
    }
    if (lane >= nj) continue;
    const double4 p = plane[my_q];
    const double dist = dabs_i(p.w - along(p, my_o)) * h;  // Eq. dint_trans
    if (d_gamma) d_gamma[my_id] = dist;
    if (!dnz(dist)) {
      grad[my_id] = __longlong_as_double(kNoGrad);
      continue;
    }
    const double cv = __ldg(c + my_id);
    const double T = div_by(__ldg(e + my_id), rcp_of(heat_cap(g.Cp_l, g.Cp_g, cv)));
    const double gr = div_by(dgthalf(cv) ? g.T_sat - T : T - g.T_sat, rcp_of(dist));
    grad[my_id] = gr;
    if (grad_n) grad_n[my_id] = gr;
  }
}

// one warp per mixed cell: per-phase weighted averages of the pure
// neighbours' gradients (lane partial sums in increasing stencil index,
// then a fixed shuffle tree) and mdot
__global__ void __launch_bounds__(kMdThreads)
k_md_avg(GridDev g, double k_l, double k_g, double h_fg, double dd_per_mdot, const double* __restrict__ c,
         const uint32_t* __restrict__ mlist, const int* __restrict__ counters, const double4* __restrict__ plane,
         const double* __restrict__ grad, double* __restrict__ mdot, double* __restrict__ dd) {
  __shared__ double s_off[5], s_rinv[13];
  pdl_wait();
  mlist = after_wait(mlist);
  counters = after_wait(counters);
  plane = after_wait(plane);
  grad = after_wait(grad);
  if (threadIdx.x < 5) s_off[threadIdx.x] = c_off[threadIdx.x];
  if (threadIdx.x < 13) s_rinv[threadIdx.x] = c_rinv[threadIdx.x];
  __syncthreads();
  const int nm = counters[0];
  const int lane = threadIdx.x & 31;
  const int nwarps = (gridDim.x * blockDim.x) >> 5;
  const LaneOffsets L = lane_offsets(g, lane);
  for (int b0 = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * kBatchAvg; b0 < nm; b0 += nwarps * kBatchAvg) {
    const int nj = min(kBatchAvg, nm - b0);
    const uint32_t my_id = lane < nj ? mlist[b0 + lane] : 0u;
    double s_al = 0.0, s_wl = 0.0, s_ag = 0.0, s_wg = 0.0;
    for (int j = 0; j < nj; ++j) {
      const uint32_t id = __shfl_sync(0xffffffffu, my_id, j);
      int x, y, z;
      cell_xyz(g, id, x, y, z);
      const bool inner = inner_cell(g, x, y, z);
      const double4 p = plane[id];
      double gq[kOffRounds];
      bool use[kOffRounds], liq[kOffRounds];
#pragma unroll
      for (int r = 0; r < kOffRounds; ++r) {
        const long long q = lane_nb(g, L, r, id, inner, x, y, z);
        const double cq = __ldg(c + (q < 0 ? 0 : q));
        use[r] = q >= 0 && !is_mixed_b(cq, g);
        liq[r] = dgthalf(cq);
        gq[r] = use[r] ? grad[q] : 0.0;
      }
      double acc_l = 0.0, w_l = 0.0, acc_g = 0.0, w_g = 0.0;
#pragma unroll
      for (int r = 0; r < kOffRounds; ++r) {
        const unsigned a = L.at[r], ox = a & 0xFFu, oy = (a >> 8) & 0xFFu, oz = (a >> 16) & 0xFFu;
        const int dx = (int)ox - 2, dy = (int)oy - 2, dz = (int)oz - 2;
        const double xi = dabs_i((p.x * s_off[ox] + p.y * s_off[oy]) + p.z * s_off[oz < 5u ? oz : 0u]);
        const double gam = xi * s_rinv[min(dx * dx + dy * dy + dz * dz, 12)];
        // one phase's sums at a time (no divergent paths)
        const double na = fma(gam, gq[r], liq[r] ? acc_l : acc_g), nw = (liq[r] ? w_l : w_g) + gam;
        if (use[r] && dbits(gq[r]) != kNoGrad) {
          if (liq[r]) {
            acc_l = na;
            w_l = nw;
          } else {
            acc_g = na;
            w_g = nw;
          }
        }
      }
      // the four sums folded: a lane of the upper half keeps the gas's, one with
      // bit 3 set the weights'; the additions are those of each sum's own tree
      const bool gas = (lane & 16) != 0, wgt = (lane & 8) != 0;
      double a = gas ? acc_g : acc_l, w = gas ? w_g : w_l;
      a += __shfl_xor_sync(0xffffffffu, gas ? acc_l : acc_g, 16);
      w += __shfl_xor_sync(0xffffffffu, gas ? w_l : w_g, 16);
      double v = wgt ? w : a;
      v += __shfl_xor_sync(0xffffffffu, wgt ? a : w, 8);
#pragma unroll
      for (int off = 4; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
      const double al = __shfl_sync(0xffffffffu, v, 0), wl = __shfl_sync(0xffffffffu, v, 8),
                   ag = __shfl_sync(0xffffffffu, v, 16), wg = __shfl_sync(0xffffffffu, v, 24);
      if (lane == j) {
        s_al = al;
        s_wl = wl;
        s_ag = ag;
        s_wg = wg;
      }
    }
    if (lane >= nj) continue;
    const double gl = dgt0(s_wl) ? s_al / s_wl : 0.0;
    const double gg = dgt0(s_wg) ? s_ag / s_wg : 0.0;
    const double md = (k_g * gg - k_l * gl) / h_fg;
    mdot[my_id] = md;
    if (dd) dd[my_id] = dd_per_mdot * md;
  }
}

}  // namespace

size_t mdot_scratch_bytes(size_t N) {
  auto a = [](size_t b) { return (b + 255) & ~(size_t)255; };
  return a(N * sizeof(double4)) + a(N * sizeof(double)) + 2 * a(N * sizeof(uint32_t)) + a(((N + 31) / 32) * 4) +
         a(4 * sizeof(int));
}

struct MdotScratch {
  double4* plane;     // [N]: unit normal and distance of each mixed cell's plane
  double* grad;       // [N]: grad_n T of each band cell
  uint32_t* mlist;    // mixed cells, grid-wide, no fixed order
  uint32_t* blist;    // band cells, grid-wide, no fixed order
  uint32_t* bits;     // [ceil(N / 32)]: band membership
  int* counters;      // [0] mixed cells, [1] band cells
  size_t zero_bytes;  // bits and counters, zeroed by each call
};

static MdotScratch carve_mdot(size_t N, void* workspace) {
  auto a = [](size_t b) { return (b + 255) & ~(size_t)255; };
  char* w = static_cast<char*>(workspace);
  MdotScratch s;
  s.plane = reinterpret_cast<double4*>(w);
  w += a(N * sizeof(double4));
  s.grad = reinterpret_cast<double*>(w);
  w += a(N * sizeof(double));
  s.mlist = reinterpret_cast<uint32_t*>(w);
  w += a(N * sizeof(uint32_t));
  s.blist = reinterpret_cast<uint32_t*>(w);
  w += a(N * sizeof(uint32_t));
  s.bits = reinterpret_cast<uint32_t*>(w);
  w += a(((N + 31) / 32) * 4);
  s.counters = reinterpret_cast<int*>(w);
  s.zero_bytes = a(((N + 31) / 32) * 4) + 4 * sizeof(int);
  return s;
}

int* mdot_counters(const GridDev& g, void* workspace) {
  return carve_mdot((size_t)g.n[0] * g.n[1] * g.n[2], workspace).counters;
}

cudaError_t launch_mass_transfer(const GridDev& g, double h, const double* c, const double* e, double k_l, double k_g,
                                 double h_fg, double dd_per_mdot, double* mdot, double* d_gamma, double* grad_n,
                                 double* dd, void* workspace, cudaStream_t st) {
  const size_t N = (size_t)g.n[0] * g.n[1] * g.n[2];
  const MdotScratch s = carve_mdot(N, workspace);
  cudaError_t err = cudaMemsetAsync(s.bits, 0, s.zero_bytes, st);
  if (err != cudaSuccess) return err;
  prof_mark("mdot.memset", st);
  const int list_ctas = (int)std::min<size_t>((N + kListThreads - 1) / kListThreads, (size_t)152 * 16);
  k_md_list<<<list_ctas, kListThreads, 0, st>>>(g, c, mdot, d_gamma, grad_n, dd, s.mlist, s.counters, N);
  prof_mark("mdot.list", st);
  launch_pdl(k_md_planes, dim3(kMdCTAs), dim3(kMdThreads), st, g, c, (const uint32_t*)s.mlist, (const int*)s.counters,
             s.plane);
  prof_mark("mdot.planes", st);
  launch_pdl(k_md_band, dim3(kMdCTAs), dim3(kMdThreads), st, g, c, (const uint32_t*)s.mlist, s.blist, s.counters, s.bits);
  prof_mark("mdot.band", st);
  launch_pdl(k_md_grad, dim3(kMdCTAs), dim3(kMdThreads), st, g, h, c, e, (const uint32_t*)s.blist,
             (const int*)s.counters, (const double4*)s.plane, s.grad, d_gamma, grad_n);
  prof_mark("mdot.grad", st);
  launch_pdl(k_md_avg, dim3(kMdCTAs), dim3(kMdThreads), st, g, k_l, k_g, h_fg, dd_per_mdot, c,
             (const uint32_t*)s.mlist, (const int*)s.counters, (const double4*)s.plane, (const double*)s.grad, mdot, dd);
  prof_mark("mdot.avg", st);
  return cudaGetLastError();
}

}  // namespace vofgb
