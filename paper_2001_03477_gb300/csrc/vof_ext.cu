// vof_ext.cu -- velocity extension across the interface (Malan et al.,
// arXiv:2001.03477, Sec. 3.3.1: Eq. press_inv, the correction u~ and
// u_l = u^{n+1} + u~).
//
// The sub-domain is the mixed cells and the pure gas cells of the first two
// layers around them (layers across cell faces).  Faces to pure liquid cells
// and zero-gradient walls are no-slip (no flux of p~, u~ = 0); faces to gas
// cells beyond the second layer are free flow (p~ = 0 there).  In every
// sub-domain cell
//     sum_faces beta_f (p~_Q - p~_P) = mdot (1/rho_g - 1/rho_l) A / h,
// beta_f = (dt / rho_f) / h^2, rho_f = rho_l c_f + rho_g (1 - c_f) with c_f
// the mean of the two cells' c, A the PLIC plane area of a mixed cell (cell
// units; gas cells have no source).  The negated system is symmetric
// positive definite and is solved by conjugate gradients with the diagonal
// as preconditioner; then u~ = -(dt / rho_f) (p~_R - p~_L) / h on every face
// with a sub-domain cell on one side and no liquid cell or wall.
//
// Kernels: k_ext_init (stream c: a code per cell, the mixed cells listed),
// k_ext_layer (the two gas layers, from the list of the layer before: the
// unknowns), k_ext_assemble (the six couplings and the source of each
// unknown), the CG iterations, and k_ext_faces (the correction on the faces of
// the unknowns).  Everything after the stream works on the list; whole-grid
// dilations, listing and face passes took 50 + 82 us at 160^3.
//
// The CG iterations run in one cooperative launch, k_ext_cg, one grid barrier
// each: the single-reduction form of Chronopoulos and Gear (1989) keeps s = M p
// by recurrence, so that both inner products belong to the same point of the
// iteration, and every thread forms its neighbours' new residuals again from
// their records {r, w, s, 1 / diag} (one 32-byte sector each; the owner's
// arithmetic) instead of waiting for them.  What bounds an iteration is the
// barrier and the chain of its sums (~15,000 unknowns are one per thread): the
// two-barrier form took 18.7 us per iteration at 160^3.  Where a cooperative
// launch of that size is refused, the standard iteration runs as the kernels
// k_ext_spmv, k_ext_update, k_ext_dir with a host test every 8 iterations.
// Inner products are per-CTA partial sums that every CTA adds up in the same
// fixed order, so all CTAs use the same scalars.
#include <algorithm>
#include <vector>

#include "../../include/vofgb.h"
#include "vof_launch.h"

namespace vofgb {

namespace {

constexpr uint8_t kOut = 255;  // pure liquid
constexpr uint8_t kGas = 254;  // pure gas beyond the layers reached so far
constexpr uint8_t kLayer = 2;  // pure gas of the two layers (unknowns, with the mixed cells' 0)
constexpr int kExtThreads = 256;    // grid-wide cell and face kernels
constexpr int kSolveThreads = 256;   // the CG kernels: one CTA per SM (few warps per FP64 sum tree)
constexpr int kExtCTAs = 152;
constexpr int kNoNb = -1;       // no-slip face (liquid cell or wall)
constexpr int kFreeNb = -2;     // free-flow face (p~ = 0 beyond)
// counters: [0] unknowns, [1] free-flow faces, [2], [3], [4] mixed cells, first
// and second layer
constexpr int kCntMixed = 2, kCnts = 5;

// face neighbour of (x, y, z) along `axis` in direction d (+-1): false
// across a zero-gradient wall
__device__ __forceinline__ bool face_nb(const GridDev& g, int x, int y, int z, int axis, int d, int& qx, int& qy,
                                        int& qz) {
  qx = x; qy = y; qz = z;
  int& p = axis == 0 ? qx : (axis == 1 ? qy : qz);
  const int n = g.n[axis];
  p += d;
  if (p < 0 || p >= n) {
    if (g.bc[axis] != 0) return false;
    p = p < 0 ? p + n : p - n;
  }
  return true;
}

__device__ __forceinline__ size_t cid(const GridDev& g, int x, int y, int z) {
  return ((size_t)z * g.n[1] + y) * g.n[0] + x;
}

__device__ __forceinline__ bool is_gas_b(double c, const GridDev& g) { return dbits(c) <= g.eps_bits; }

// entries appended to a list by a warp, one atomic
__device__ __forceinline__ int warp_append_ext(bool take, uint32_t v, uint32_t* list, int* counter) {
  const unsigned mask = __ballot_sync(0xffffffffu, take);
  if (!mask) return -1;
  const int lane = threadIdx.x & 31;
  int base = 0;
  if (lane == __ffs(mask) - 1) base = atomicAdd(counter, __popc(mask));
  base = __shfl_sync(0xffffffffu, base, __ffs(mask) - 1);
  if (!take) return -1;
  const int slot = base + __popc(mask & ((1u << lane) - 1u));
  list[slot] = v;
  return slot;
}

// code of every cell; the mixed cells are the first unknowns (list, map)
__global__ void __launch_bounds__(kExtThreads)
k_ext_init(GridDev g, const double* __restrict__ c, uint8_t* __restrict__ code, uint32_t* __restrict__ list,
           int* __restrict__ map, int* __restrict__ counters, size_t N) {
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  const size_t n_iter = (N + stride - 1) / stride;  // whole warps iterate together
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (size_t it = 0; it < n_iter; ++it, i += stride) {
    bool mx = false;
    if (i < N) {
      const double cv = __ldg(c + i);
      mx = is_mixed_b(cv, g);
      code[i] = mx ? (uint8_t)0 : (is_gas_b(cv, g) ? kGas : kOut);
    }
    const int slot = warp_append_ext(mx, (uint32_t)i, list, counters + kCntMixed);
    if (mx) map[i] = slot;
  }
}

// The gas cells next (across a face) to the unknowns of the layer before (the
// mixed cells; then the first layer) join the list behind them.  One bit mask
// per claim: kGas becomes kLayer, and the thread that sees kGas lists the cell.
__global__ void __launch_bounds__(kExtThreads)
k_ext_layer(GridDev g, uint8_t* __restrict__ code, uint32_t* __restrict__ list, int* __restrict__ map,
            int* __restrict__ counters, int layer) {
  const int nm = counters[kCntMixed], n1 = layer == 1 ? 0 : counters[kCntMixed + 1];
  const int b = layer == 1 ? 0 : nm, n = nm + n1;  // the sources; the new entries start at n
  // eight threads per source, six of them a face each
  const long long stride = (long long)gridDim.x * blockDim.x, total = 8ll * (n - b);
  for (long long j0 = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31); j0 < total; j0 += stride) {
    const long long j = j0 + (threadIdx.x & 31);
    const int f = (int)(j & 7);
    bool take = false;
    size_t q = 0;
    if (j < total && f < 6) {
      int x, y, z, qx, qy, qz;
      cell_xyz(g, list[b + (j >> 3)], x, y, z);
      if (face_nb(g, x, y, z, f >> 1, (f & 1) ? 1 : -1, qx, qy, qz)) {
        q = cid(g, qx, qy, qz);
        if (code[q] == kGas) {  // (it may have been claimed since: the mask keeps kLayer)
          const int sh = 8 * (int)(q & 3);
          const unsigned old = atomicAnd(reinterpret_cast<unsigned*>(code + (q & ~(size_t)3)), ~((unsigned)(kGas ^ kLayer) << sh));
          take = ((old >> sh) & 0xFFu) == kGas;
        }
      }
    }
    const int slot = warp_append_ext(take, (uint32_t)q, list + n, counters + kCntMixed + layer);
    if (take) map[q] = n + slot;
  }
}

// Fixed-order sums of the per-CTA partials (the same values in every CTA):
// warp 0 alone, each lane its partials lane, lane + 32, ... in order, then a
// shuffle tree; K sums at once (one barrier).  L2: the partials were written
// by other CTAs of the same launch, so the loads skip L1 (not coherent
// across SMs).
template <int K, bool L2>
__device__ __forceinline__ void sum_partials_k(const double* const (&part)[K], int n, double (&out)[K]) {
  __shared__ double res[K];
  __syncthreads();  // res may still be read from the previous call
  if (threadIdx.x < 32) {
    double v[K];
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] = 0.0;
    for (int i = threadIdx.x; i < n; i += 32)
#pragma unroll
      for (int k = 0; k < K; ++k) v[k] += L2 ? __ldcg(part[k] + i) : part[k][i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int k = 0; k < K; ++k) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
    if (threadIdx.x == 0)
#pragma unroll
      for (int k = 0; k < K; ++k) res[k] = v[k];
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < K; ++k) out[k] = res[k];
}
// A CTA's partial sums of K values in a fixed order (the threads' values
// staged in shared memory; warp 0 sums them, each lane its entries lane,
// lane + 32, ... in order, then a shuffle tree: few FP64 instructions per
// value), written to out[k][blockIdx.x].
template <int K>
__device__ __forceinline__ void block_partial_k(const double (&v)[K], double* const (&out)[K]) {
  __shared__ double red[K][kSolveThreads];
  __syncthreads();  // red may still be read from the previous call
#pragma unroll
  for (int k = 0; k < K; ++k) red[k][threadIdx.x] = v[k];
  __syncthreads();
  if (threadIdx.x < 32) {
    double x[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      x[k] = 0.0;
      for (int i = threadIdx.x; i < (int)blockDim.x; i += 32) x[k] += red[k][i];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int k = 0; k < K; ++k) x[k] += __shfl_down_sync(0xffffffffu, x[k], o);
    if (threadIdx.x == 0)
#pragma unroll
      for (int k = 0; k < K; ++k) out[k][blockIdx.x] = x[k];
  }
}
__device__ __forceinline__ void block_partial(double v, double* __restrict__ out) {
  const double vv[1] = {v};
  double* const o[1] = {out};
  block_partial_k<1>(vv, o);
}

// one unknown's state of the cooperative solver: a 32-byte sector
struct __align__(32) ExtRec {
  double r, w, s, rdiag;
};

struct ExtVec {
  int* nb;        // [6 n]: neighbour unknown, kNoNb, or kFreeNb
  double* beta;   // [6 n]
  double* diag;   // [n]
  double* rdiag;  // [n]: 1 / diag (0 where diag is 0), the Jacobi preconditioner
  double* x;      // p~
  double* r;
  double* d;
  double* q;
  ExtRec* rec[2]; // the cooperative solver's records, the two taking turns (in r, q and their
  int cap;        // spare's place, for up to cap unknowns)
  double* part;   // [6][kExtCTAs]: b.b, r.z (two, alternating), d.q, r.r; cooperative: two sets of three
  int* counters;  // [kCnts]
};

// area of the plane m . x = alpha inside the unit cube: |m|_2 dV/dalpha, the
// slope of the volume's branch form (a polygon's vertices sorted by angle took
// ~800 FP64 instructions)
__device__ __forceinline__ double cut_area(const double m[3], double alpha) {
  const Mirror r = mirror_normalise(m[0], m[1], m[2]);
  if (!dnz(r.l1)) return 0.0;
  const double a0 = div_by(alpha + r.sh, r.R);
  const double a = nn_lt(0.5, a0) ? 1.0 - a0 : a0;
  if (!dgt0(a)) return 0.0;
  double slope = 0.0;
  (void)vol_eval<true>(vol_form(r.mp[0], r.mp[1], r.mp[2]), a, slope);
  return div_by(slope, r.R) * sqrt(m[0] * m[0] + m[1] * m[1] + m[2] * m[2]);
}

constexpr int kAsmThreads = 64;  // few unknowns, long chains: spread over the SMs
__global__ void __launch_bounds__(kAsmThreads)  // (heavy per unknown: no register cap)
k_ext_assemble(GridDev g, double h, double dt, double rho_l, double rho_g, const double* __restrict__ c,
               const double* __restrict__ mdot, const uint8_t* __restrict__ code, const int* __restrict__ map,
               const uint32_t* __restrict__ list, ExtVec v, unsigned char* __restrict__ cg_state) {
  const int n = v.counters[kCntMixed] + v.counters[kCntMixed + 1] + v.counters[kCntMixed + 2];
  if (blockIdx.x == 0 && threadIdx.x < 32) reinterpret_cast<unsigned long long*>(cg_state)[threadIdx.x] = 0ull;
  if (blockIdx.x == 0 && threadIdx.x == 0) v.counters[0] = n;  // read by the kernels after this one
  int free_faces = 0;
  const Rcp rhh = rcp_of(h * h);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint32_t id = list[i];
    int x, y, z;
    cell_xyz(g, id, x, y, z);
    const double cp = __ldg(c + id);
    double dsum = 0.0;
    for (int f = 0; f < 6; ++f) {
      const int axis = f >> 1, dir = (f & 1) ? 1 : -1;
      int qx, qy, qz;
      int nb = kNoNb;
      double beta = 0.0;
      if (face_nb(g, x, y, z, axis, dir, qx, qy, qz)) {
        const size_t qid = cid(g, qx, qy, qz);
        const uint8_t qc = code[qid];
        if (qc != kOut) {
          const double cf = 0.5 * (cp + __ldg(c + qid));
          const double rho = rho_l * cf + rho_g * (1.0 - cf);
          beta = div_by(div_by(dt, rcp_of(rho)), rhh);
          nb = qc <= 2 ? map[qid] : kFreeNb;
          if (nb == kFreeNb) ++free_faces;
        }
      }
      v.nb[6 * (size_t)i + f] = nb;
      v.beta[6 * (size_t)i + f] = beta;
      dsum += beta;
    }
    double rhs = 0.0;
    if (code[id] == 0) {
      double s[27];
      for (int oz = 0; oz < 3; ++oz)
        for (int oy = 0; oy < 3; ++oy)
          for (int ox = 0; ox < 3; ++ox)
            s[(oz * 3 + oy) * 3 + ox] = __ldg(c + cid(g, map_idx(x + ox - 1, g.n[0], g.bc[0]),
                                                        map_idx(y + oy - 1, g.n[1], g.bc[1]),
                                                        map_idx(z + oz - 1, g.n[2], g.bc[2])));
      double m[3];
      myc_normal(s, m);
      const double al = plane_alpha(m[0], m[1], m[2], cp);
      rhs = __ldg(mdot + id) * (1.0 / rho_g - 1.0 / rho_l) * cut_area(m, al) / h;
    }
    // M = -A: diagonal sum beta, off-diagonal -beta; b = -rhs
    const double b = -rhs;
    const double rd = dsum > 0.0 ? 1.0 / dsum : 0.0;
    v.diag[i] = dsum;
    v.rdiag[i] = rd;
    v.x[i] = 0.0;
    if (n <= v.cap) {
      v.rec[0][i] = ExtRec{b, 0.0, 0.0, rd};
    } else {
      v.r[i] = b;
      v.d[i] = b * rd;
    }
  }
  if (free_faces) atomicAdd(v.counters + 1, free_faces);
}

// b . b and r . z of the start (the kernel-per-phase solver)
__global__ void __launch_bounds__(kSolveThreads) k_ext_start(ExtVec v) {
  const int n = v.counters[0];
  double bb = 0.0, rz = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const double b = v.r[i];
    bb = fma(b, b, bb);
    rz = fma(b, v.d[i], rz);
  }
  const double pv[2] = {bb, rz};
  double* const po[2] = {v.part, v.part + kExtCTAs};
  block_partial_k<2>(pv, po);
}

// The element arithmetic of one iteration of the kernel-per-phase solver: q = M d with its partial d . q; x += alpha d, r -= alpha q, z = r /
// diag with the partials r . z and r . r; d = z + beta d.
__device__ __forceinline__ double ext_spmv_elem(const ExtVec& v, int i) {
  double q = v.diag[i] * v.d[i];
#pragma unroll
  for (int f = 0; f < 6; ++f) {
    const int nb = v.nb[6 * (size_t)i + f];
    if (nb >= 0) q = fma(-v.beta[6 * (size_t)i + f], v.d[nb], q);
  }
  v.q[i] = q;
  return q;
}

// q = M d, partial d . q
__global__ void __launch_bounds__(kSolveThreads) k_ext_spmv(ExtVec v) {
  const int n = v.counters[0];
  double dq = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    dq = fma(v.d[i], ext_spmv_elem(v, i), dq);
  block_partial(dq, v.part + 3 * kExtCTAs);
}

// alpha = r.z / d.q; x += alpha d; r -= alpha q; partial r.z (new) and r.r
__device__ __forceinline__ void ext_update_elems(const ExtVec& v, int n, double alpha, double& rzn, double& rr) {
  rzn = 0.0;
  rr = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    v.x[i] = fma(alpha, v.d[i], v.x[i]);
    const double r = fma(-alpha, v.q[i], v.r[i]);
    v.r[i] = r;
    rzn = fma(r, r * v.rdiag[i], rzn);
    rr = fma(r, r, rr);
  }
}
__global__ void __launch_bounds__(kSolveThreads) k_ext_update(ExtVec v, int cur) {
  const double* pp[2] = {v.part + (1 + cur) * kExtCTAs, v.part + 3 * kExtCTAs};
  double s2[2];
  sum_partials_k<2, false>(pp, kExtCTAs, s2);
  const double alpha = s2[1] > 0.0 ? s2[0] / s2[1] : 0.0;
  double rzn, rr;
  ext_update_elems(v, v.counters[0], alpha, rzn, rr);
  const double pv[2] = {rzn, rr};
  double* const po[2] = {v.part + (2 - cur) * kExtCTAs, v.part + 4 * kExtCTAs};
  block_partial_k<2>(pv, po);
}

// d = z + (r.z new / r.z old) d
__device__ __forceinline__ void ext_dir_elems(const ExtVec& v, int n, double beta) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    v.d[i] = fma(beta, v.d[i], v.r[i] * v.rdiag[i]);
}
__global__ void __launch_bounds__(kSolveThreads) k_ext_dir(ExtVec v, int cur) {
  const double* pp[2] = {v.part + (1 + cur) * kExtCTAs, v.part + (2 - cur) * kExtCTAs};
  double s2[2];
  sum_partials_k<2, false>(pp, kExtCTAs, s2);
  const double beta = s2[0] > 0.0 ? s2[1] / s2[0] : 0.0;
  ext_dir_elems(v, v.counters[0], beta);
}

// Device state of the persistent solver (in the workspace; the assemble
// kernel clears it).
struct ExtCG {
  unsigned arrive;  // grid barrier: CTAs arrived at the current barrier
  unsigned gen;     // grid barrier: barriers completed
  int iters;        // iterations done
  int flag;         // 1 converged, 2 iteration limit, 3 a barrier wait gave up, 4 not solved here
  double res;       // |r| at the end
};
static_assert(sizeof(ExtCG) <= 256, "the solver state lives in 256 bytes of the workspace");

__device__ __forceinline__ unsigned long long ext_now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Grid barrier of a cooperative launch (all CTAs resident): the last of the
// CTAs to arrive starts the next generation, which the others poll (an atomic
// and a load from L2; a tree of counters and a sleeping poll took longer).  The
// wait is bounded (1 s): on expiry the CTA records DEV_WAIT and returns false,
// and the solver stops.
__device__ __forceinline__ bool ext_grid_barrier(ExtCG* cg, int* status) {
  __shared__ int ok_s;
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    volatile unsigned* vgen = &cg->gen;
    const unsigned g0 = *vgen;
    __threadfence();  // this CTA's writes, and g0, before its arrival
    if (atomicAdd(&cg->arrive, 1u) == gridDim.x - 1) {
      atomicExch(&cg->arrive, 0u);
      __threadfence();
      atomicAdd(&cg->gen, 1u);
    } else {
      const unsigned long long t0 = ext_now_ns();
      while (*vgen == g0) {
        if (ext_now_ns() - t0 > 1000000000ull) {
          ok = 0;
          if (status) atomicOr(status, DEV_WAIT);
          break;
        }
      }
    }
    __threadfence();  // the other CTAs' writes before this CTA reads them
    ok_s = ok;
  }
  __syncthreads();
  return ok_s != 0;
}

__device__ __forceinline__ ExtRec rec_l2(const ExtRec* p) {  // written by other CTAs of this launch: from L2
  const double2 a = __ldcg(reinterpret_cast<const double2*>(p)), b = __ldcg(reinterpret_cast<const double2*>(p) + 1);
  return ExtRec{a.x, a.y, b.x, b.y};
}

// One pass per iteration (the first, with alpha = beta = 0, only forms u = r /
// diag, w = M u and the inner products of the start):
//   s <- w + beta s, r <- r - alpha s, u = r / diag, w = M u,
//   p <- u_old + beta p, x <- x + alpha p;  gamma = r.u, delta = w.u, |r|^2
// then beta = gamma / gamma_old, alpha = gamma / (delta - beta gamma / alpha).
__global__ void __launch_bounds__(kSolveThreads)
k_ext_cg(ExtVec v, ExtCG* cg, double tol, int max_iter, int* status) {
  __shared__ double red[3][kSolveThreads];
  __shared__ double tot[3];
  const int n = v.counters[0];
  if (n == 0 || v.counters[1] == 0 || n > v.cap) {  // the same in every CTA
    if (blockIdx.x == 0 && threadIdx.x == 0) cg->flag = 4;
    return;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // unknown i is CTA i mod grid's: a few thousand of them reach every SM, and
  // its partitions' FP64 units share them; the first of a thread keeps its
  // couplings in registers
  const int i0 = blockIdx.x + gridDim.x * threadIdx.x, step = gridDim.x * blockDim.x;
  const int rows = min(kSolveThreads / 32, ((n - 1) / (int)gridDim.x) / 32 + 1);  // warps with unknowns
  int nb0[6];
  double be0[6], dg0 = 0.0;
#pragma unroll
  for (int f = 0; f < 6; ++f) {
    nb0[f] = i0 < n ? v.nb[6 * (size_t)i0 + f] : kNoNb;
    be0[f] = i0 < n ? v.beta[6 * (size_t)i0 + f] : 0.0;
  }
  if (i0 < n) dg0 = v.diag[i0];
  double alpha = 0.0, beta = 0.0, gamma = 0.0, rr = 0.0, limit = 0.0;
  int cur = 0, it = -1;
  bool ok = true;
  for (;;) {
    const ExtRec* __restrict__ in = v.rec[cur];
    ExtRec* __restrict__ out = v.rec[cur ^ 1];
    double gm = 0.0, dl = 0.0, r2 = 0.0;
    for (int i = i0; i < n; i += step) {
      ExtRec o = rec_l2(in + i), q[6];
      const bool kept = i == i0;
      int nb[6];
#pragma unroll
      for (int f = 0; f < 6; ++f) {
        nb[f] = kept ? nb0[f] : v.nb[6 * (size_t)i + f];
        q[f] = nb[f] >= 0 ? rec_l2(in + nb[f]) : ExtRec{0.0, 0.0, 0.0, 0.0};
      }
      if (it >= 0) {
        // (the direction: z of the iteration before, the owner's only)
        const double p = it == 0 ? o.r * o.rdiag : fma(beta, v.d[i], o.r * o.rdiag);
        v.d[i] = p;
        v.x[i] = fma(alpha, p, v.x[i]);
      }
      o.s = fma(beta, o.s, o.w);
      o.r = fma(-alpha, o.s, o.r);
      const double u = o.r * o.rdiag;
      double w = (kept ? dg0 : v.diag[i]) * u;
#pragma unroll
      for (int f = 0; f < 6; ++f) {
        if (__any_sync(__activemask(), nb[f] >= 0)) {
          const double un = fma(-alpha, fma(beta, q[f].s, q[f].w), q[f].r) * q[f].rdiag;
          const double be = kept ? be0[f] : v.beta[6 * (size_t)i + f];
          if (nb[f] >= 0) w = fma(-be, un, w);
        }
      }
      o.w = w;
      out[i] = o;
      gm = fma(o.r, u, gm);
      dl = fma(w, u, dl);
      r2 = fma(o.r, o.r, r2);
    }
    // the CTA's partial sums, one quantity per warp, in a fixed order
    red[0][threadIdx.x] = gm;
    red[1][threadIdx.x] = dl;
    red[2][threadIdx.x] = r2;
    // (the reciprocals of the scalars before, while others arrive)
    const Rcp Rg = rcp_of<true>(gamma), Ra = rcp_of<true>(alpha);
    __syncthreads();
    double* part = v.part + 3 * cur * kExtCTAs;  // the passes alternate: a slow CTA may still read the last
    if (warp < 3) {
      double t = red[warp][lane];
      for (int j = 1; j < rows; ++j) t += red[warp][lane + 32 * j];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
      if (lane == 0) part[warp * kExtCTAs + blockIdx.x] = t;
    }
    if (!(ok = ext_grid_barrier(cg, status))) break;
    if (warp < 3) {
      double t = 0.0;
#pragma unroll
      for (int j = 0; j < (kExtCTAs + 31) / 32; ++j) {
        const int b = lane + 32 * j;
        if (b < kExtCTAs) t += __ldcg(part + warp * kExtCTAs + b);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
      if (lane == 0) tot[warp] = t;
    }
    __syncthreads();
    const double g1 = tot[0], d1 = tot[1];
    rr = tot[2];
    cur ^= 1;
    ++it;
    if (it == 0) {
      limit = tol * tol * rr;  // (|r| against tol |b| without a square root)
      beta = 0.0;
      alpha = d1 > 0.0 ? div_by(g1, rcp_of<true>(d1)) : 0.0;
    } else {
      beta = gamma > 0.0 ? div_by(g1, Rg) : 0.0;
      const double den = alpha > 0.0 ? d1 - beta * div_by(g1, Ra) : 0.0;
      alpha = den > 0.0 ? div_by(g1, rcp_of<true>(den)) : 0.0;
    }
    gamma = g1;
    if (!(rr > limit) || it >= max_iter) break;  // the same values in every CTA
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    cg->iters = it;
    cg->res = sqrt(rr);
    cg->flag = !ok ? 3 : (rr > limit ? 2 : 1);
  }
}

// The face correction u~ = -(dt / rho_f) (p~_R - p~_L) / h on the faces of the
// unknowns, one (unknown, face) per thread: a face between two unknowns is its
// left cell's, any other face its unknown's; a face to a liquid cell or a wall
// has none.  Across a periodic boundary the face is stored twice.
struct ExtOut {
  double* u[3];
  double* ut[3];
};
// zeros in the arrays of u~ (three memsets one after the other took 45 us at
// 160^3)
__global__ void __launch_bounds__(kExtThreads) k_ext_zero(GridDev g, ExtOut out) {
  const size_t N = (size_t)g.n[0] * g.n[1] * g.n[2], stride = (size_t)gridDim.x * blockDim.x;
  for (int ax = 0; ax < 3; ++ax) {
    double* __restrict__ p = out.ut[ax];
    if (!p) continue;
    const size_t n = N / (size_t)g.n[ax] * (size_t)(g.n[ax] + 1);
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) p[i] = 0.0;
  }
}
__global__ void __launch_bounds__(kExtThreads)
k_ext_faces(GridDev g, double h, double dt, double rho_l, double rho_g, const double* __restrict__ c,
            const uint8_t* __restrict__ code, const int* __restrict__ map, const uint32_t* __restrict__ list,
            const int* __restrict__ counters, const double* __restrict__ xs, ExtOut out) {
  const long long total = 8ll * counters[0];  // (two of eight threads idle: no division by 6)
  for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < total; j += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(j >> 3), f = (int)(j & 7), axis = f >> 1;
    if (f >= 6) continue;
    const bool right = (f & 1) != 0;
    const size_t id = list[i];
    int x, y, z, qx, qy, qz;
    cell_xyz(g, id, x, y, z);
    if (!face_nb(g, x, y, z, axis, right ? 1 : -1, qx, qy, qz)) continue;  // a wall: no-slip
    const size_t q = cid(g, qx, qy, qz);
    const uint8_t cq = code[q];
    if (cq == kOut || (!right && cq <= kLayer)) continue;
    const double own = xs[i], oth = cq <= kLayer ? xs[map[q]] : 0.0;
    const double cf = 0.5 * (__ldg(c + (right ? id : q)) + __ldg(c + (right ? q : id)));
    const double rho = rho_l * cf + rho_g * (1.0 - cf);
    const double pl = right ? own : oth, pr = right ? oth : own;
    const double val = div_by(-div_by(dt, rcp_of(rho)) * (pr - pl), rcp_of(h));
    const int n = g.n[axis];
    int p[3] = {x, y, z};
    p[axis] += right ? 1 : 0;
    auto put = [&](int fp) {
      int s[3] = {p[0], p[1], p[2]};
      s[axis] = fp;
      const size_t at = axis == 0 ? ((size_t)s[2] * g.n[1] + s[1]) * (n + 1) + s[0]
                                  : (axis == 1 ? ((size_t)s[2] * (n + 1) + s[1]) * g.n[0] + s[0]
                                               : ((size_t)s[2] * g.n[1] + s[1]) * g.n[0] + s[0]);
      if (out.ut[axis]) out.ut[axis][at] = val;
      if (out.u[axis]) out.u[axis][at] += val;
    };
    put(p[axis]);
    if (g.bc[axis] == 0 && p[axis] == n) put(0);
    if (g.bc[axis] == 0 && p[axis] == 0) put(n);
  }
}

struct ExtLayout {
  size_t code, map, list, nb, beta, diag, rdiag, x, r, d, q, part, counters, cg, total;
};

ExtLayout ext_layout(size_t N) {
  auto a = [](size_t b) { return (b + 255) & ~(size_t)255; };
  ExtLayout L;
  size_t o = 0;
  L.code = o; o += a(N + 3);
  L.map = o; o += a(N * 4);
  L.list = o; o += a(N * 4);
  L.nb = o; o += a(N * 6 * 4);
  L.beta = o; o += a(N * 6 * 8);
  L.diag = o; o += a(N * 8);
  L.rdiag = o; o += a(N * 8);
  L.x = o; o += a(N * 8);
  L.d = o; o += a(N * 8);
  L.r = o; o += a(N * 8);
  L.q = o; o += 2 * a(N * 8);  // (and a spare: the cooperative solver's records take all three)
  L.part = o; o += a(6 * kExtCTAs * 8);
  L.counters = o; o += a(kCnts * 4);
  L.cg = o; o += 256;
  L.total = o;
  return L;
}

}  // namespace

size_t ext_scratch_bytes(size_t N) { return ext_layout(N).total; }

cudaError_t launch_velocity_extension(const GridDev& g, double h, const double* c, const double* mdot, double rho_l,
                                      double rho_g, double dt, double tol, int max_iter, double* u, double* v,
                                      double* w, double* ut, double* vt, double* wt, void* workspace,
                                      cudaStream_t st, int* iters_out, double* res_out, int* status) {
  const size_t N = (size_t)g.n[0] * g.n[1] * g.n[2];
  const ExtLayout L = ext_layout(N);
  char* ws = static_cast<char*>(workspace);
  uint8_t* code = reinterpret_cast<uint8_t*>(ws + L.code);
  int* map = reinterpret_cast<int*>(ws + L.map);
  uint32_t* list = reinterpret_cast<uint32_t*>(ws + L.list);
  ExtVec vec;
  vec.nb = reinterpret_cast<int*>(ws + L.nb);
  vec.beta = reinterpret_cast<double*>(ws + L.beta);
  vec.diag = reinterpret_cast<double*>(ws + L.diag);
  vec.rdiag = reinterpret_cast<double*>(ws + L.rdiag);
  vec.x = reinterpret_cast<double*>(ws + L.x);
  vec.r = reinterpret_cast<double*>(ws + L.r);
  vec.d = reinterpret_cast<double*>(ws + L.d);
  vec.q = reinterpret_cast<double*>(ws + L.q);
  vec.part = reinterpret_cast<double*>(ws + L.part);
  vec.counters = reinterpret_cast<int*>(ws + L.counters);
  *status = 0;
  cudaError_t err = cudaMemsetAsync(vec.counters, 0, kCnts * sizeof(int), st);
  if (err != cudaSuccess) return err;
  const int grid_cells = (int)std::min<size_t>((N + kExtThreads - 1) / kExtThreads, (size_t)152 * 16);
  k_ext_init<<<grid_cells, kExtThreads, 0, st>>>(g, c, code, list, map, vec.counters, N);
  k_ext_layer<<<kExtCTAs * 4, kExtThreads, 0, st>>>(g, code, list, map, vec.counters, 1);
  k_ext_layer<<<kExtCTAs * 4, kExtThreads, 0, st>>>(g, code, list, map, vec.counters, 2);
  prof_mark("ext.layers", st);
  // one cooperative launch when all kExtCTAs CTAs fit at once (the grid
  // barriers need them resident); else three kernels per iteration
  int dev = 0, nsm = 0, per_sm = 0, coop = 0;
  const bool one = cudaGetDevice(&dev) == cudaSuccess &&
                   cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess &&
                   cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
                   cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_ext_cg, kSolveThreads, 0) == cudaSuccess &&
                   coop && (long long)per_sm * nsm >= kExtCTAs;
  // the records of up to 3/8 N unknowns fit (interface layers hold far fewer
  // cells than that but on tiny grids); more go the other way
  vec.cap = one ? (int)(3 * N / 8) : 0;
  vec.rec[0] = reinterpret_cast<ExtRec*>(ws + L.r);
  vec.rec[1] = vec.rec[0] + vec.cap;
  unsigned char* cg_state = reinterpret_cast<unsigned char*>(ws + L.cg);
  k_ext_assemble<<<kExtCTAs * 8, kAsmThreads, 0, st>>>(g, h, dt, rho_l, rho_g, c, mdot, code, map, list, vec, cg_state);
  prof_mark("ext.assemble", st);
  ExtCG hcg{};
  if (one) {
    ExtCG* cg = reinterpret_cast<ExtCG*>(cg_state);
    int* dstat = device_status_ptr();
    void* args[] = {&vec, &cg, &tol, &max_iter, &dstat};
    err = cudaLaunchCooperativeKernel((const void*)k_ext_cg, dim3(kExtCTAs), dim3(kSolveThreads), args, 0, st);
    if (err != cudaSuccess) return err;
    prof_mark("ext.cg", st);
    err = cudaMemcpyAsync(&hcg, cg, sizeof(ExtCG), cudaMemcpyDeviceToHost, st);
    if (err != cudaSuccess) return err;
  }
  int host_counts[2] = {0, 0};
  err = cudaMemcpyAsync(host_counts, vec.counters, 2 * sizeof(int), cudaMemcpyDeviceToHost, st);
  if (err == cudaSuccess) err = cudaStreamSynchronize(st);
  if (err != cudaSuccess) return err;
  const int n = host_counts[0];
  std::vector<double> part(kExtCTAs);
  auto host_sum = [&](int slot, double* out) -> cudaError_t {
    cudaError_t e = cudaMemcpyAsync(part.data(), vec.part + slot * kExtCTAs, kExtCTAs * sizeof(double),
                                    cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    double s = 0.0;
    for (int i = 0; i < kExtCTAs; ++i) s += part[i];
    *out = s;
    return e;
  };
  int it = 0;
  double res = 0.0;
  if (n > 0 && host_counts[1] == 0) {
    *status = 1;  // nothing fixes p~
    return cudaSuccess;
  }
  const bool solved = one && n <= vec.cap;
  if (solved && n > 0) {
    it = hcg.iters;
    res = hcg.res;
    if (hcg.flag != 1) *status = 2;  // not converged (or a barrier wait gave up: DEV_WAIT is set)
  }
  if (n > 0 && !solved) {
    k_ext_start<<<kExtCTAs, kSolveThreads, 0, st>>>(vec);
    double bb = 0.0;
    err = host_sum(0, &bb);
    if (err != cudaSuccess) return err;
    const double target = tol * sqrt(bb);
    res = sqrt(bb);
    int cur = 0;
    while (res > target && it < max_iter) {
      k_ext_spmv<<<kExtCTAs, kSolveThreads, 0, st>>>(vec);
      k_ext_update<<<kExtCTAs, kSolveThreads, 0, st>>>(vec, cur);
      k_ext_dir<<<kExtCTAs, kSolveThreads, 0, st>>>(vec, cur);
      cur ^= 1;
      ++it;
      if (it % 8 == 0 || it == max_iter) {
        double rr = 0.0;
        err = host_sum(4, &rr);
        if (err != cudaSuccess) return err;
        res = sqrt(rr);
      }
    }
    prof_mark("ext.cg", st);
    if (res > target) *status = 2;  // not converged within max_iter
  }
  ExtOut out{{u, v, w}, {ut, vt, wt}};
  if (ut || vt || wt) k_ext_zero<<<152 * 8, kExtThreads, 0, st>>>(g, out);
  if (n > 0)
    k_ext_faces<<<kExtCTAs * 4, kExtThreads, 0, st>>>(g, h, dt, rho_l, rho_g, c, code, map, list, vec.counters, vec.x, out);
  prof_mark("ext.faces", st);
  if (iters_out) *iters_out = it;
  if (res_out) *res_out = res;
  return cudaGetLastError();
}

}  // namespace vofgb
