// vof_fused.cu -- the sweeps of an in-place time step (Malan et al.,
// arXiv:2001.03477, Sec. 3.3.1, 3.4.1), two kernels per sweep:
//   k_mix (donors): one mixed cell per thread over the stage's list: the PLIC
//     plane (MYC normal, plane constant) and the volume it sends through the
//     face or faces it is the donor of, stored per cell;
//   k_walk: a warp takes 32 lines (8 x 4 across a tile of 8^3 cells) and walks
//     them along the sweep axis with a register window: T = e / C_p(c) and its
//     difference to the previous cell once per cell, the face's VOF and energy
//     flux once per face, the update of the cell behind it, and the list of
//     the mixed cells it leaves for the next stage.
// The stages read one pair of (c, e) arrays and write the other (caller ->
// scratch -> caller -> scratch; the shift's last kernel brings the state back
// to the caller's), so no cell is read after it is written.  Only tiles that
// are not quiet (vof_tiles.cu) are visited and written; a quiet tile's cells
// are read from the caller's arrays at every stage.
//
// What bounds the walk is the FP64 unit: an FP64 instruction takes ~76 cycles
// of its SM partition per warp, and a face plus its cell now take 13 of them
// (T, its difference, u dt / h, the WENO5 correction's last addition, G's two
// products, Theta a on both sides and four additions of the update), where the
// list kernels of the stand-alone sweeps, which hold every value in memory
// between them, took 41.
#include <algorithm>

#include "vof_launch.h"
#include "vof_sums.cuh"
#include "vof_sweep.cuh"

namespace vofgb {

namespace {

constexpr int kMixThreads = 128;
constexpr int kWalkWarps = 2;           // warps per CTA of k_walk
constexpr int kWalkPerSM = 8;           // resident CTAs per SM (24 KB of rings, 128 registers a thread)
constexpr int kBatch = 4;               // positions loaded at a time
constexpr int kRing = 3 * kBatch;       // c, e: the batch before (updated cells), the current and the next one
constexpr int kRingF = 2 * kBatch;      // velocities, Theta: the current and the next batch
constexpr int kRow = 36;                // row stride in doubles: the x walk's transposed 8-byte
                                        // stores (4 rows x 4 positions per half warp) hit 16 banks
constexpr int kPend = 96;               // pending list entries per warp

__device__ __forceinline__ void cp8(double* dst, const double* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// Between the stages of a step the c words carry two bits above the value
// (c in [0, 1] leaves the sign and the exponent's top bit clear).  After the
// first two sweeps: bit 62 the cell has changed in this step, bit 63 its frozen
// cc.  After the third: 1 << 62 a moving mixed cell with dd < 0, 2 << 62 one
// with dd > 0, 3 << 62 a receiver of the shift.  (A byte per cell in an array of
// its own cost a load and a store per cell and stage.)
__device__ __forceinline__ unsigned c_tag(double w) { return (unsigned)__double2hiint(w) >> 30; }
__device__ __forceinline__ double c_with(double c, unsigned tag) {
  return __hiloint2double((int)((unsigned)__double2hiint(c) & 0x3FFFFFFFu | tag << 30), __double2loint(c));
}

// c within 1e-3 of 0 or 1: the shift takes its plane constant by bisection
__device__ __forceinline__ bool shift_edge(double c) {
  return dbits(c) < 0x3F50624DD2F1A9FCLL /* 1e-3 */ || dbits(c) > 0x3FEFF7CED916872BLL /* 0.999 */;
}

}  // namespace

// ---------------------------------------------------------------------------
// k_mix.  NRM 0: MYC; 1: the normals are already in A.plane (the learned
// normal, vof_mlp.cu); 2: Youngs.  A boundary cell on a zero-gradient sweep
// axis is also looked at as the ghost donor behind its wall, whose plane
// comes from the ghost's own stencil of the boundary-filled field (always
// MYC).  fl holds minus the volume sent to the left, fr the one to the right;
// gf the ghosts'.
// ---------------------------------------------------------------------------
template <int AX, bool F32, int NRM>
__device__ __forceinline__ void mix_body(const StepArgs& A, int stage, const VB vb) {
  const GridDev& g = A.g;
  const int n_ax = g.n[AX], bca = g.bc[AX];
  const int nm = A.cnt[4 * stage];
  const uint32_t* __restrict__ list = A.list[stage & 1];
  const double* __restrict__ c = (stage & 1) ? A.s_c : A.c;
  const double* __restrict__ uf = A.uf[AX];
  for (int i = vb.bx * blockDim.x + threadIdx.x; i < nm; i += vb.gx * blockDim.x) {
    const size_t id = list[i];
    int x, y, z;
    cell_xyz(g, id, x, y, z);
    const int k = AX == 0 ? x : (AX == 1 ? y : z);
    const int k1 = (bca == 0 && k + 1 == n_ax) ? 0 : k + 1;
    const double al = __ldg(uf + face_of<AX>(g, k, x, y, z)) * g.lam;
    const double ar = __ldg(uf + face_of<AX>(g, k1, x, y, z)) * g.lam;
    const double cd = stage ? c_value(c[id]) : c[id];
    // rep 0: the cell; 1: the ghost below it; 2: the ghost above it
    for (int rep = 0; rep < 3; ++rep) {
      const bool low = rep == 1 && bca != 0 && k == 0 && dgt0(al);
      const bool high = rep == 2 && bca != 0 && k == n_ax - 1 && dlt0(ar);
      const bool act = rep == 0 || low || high;
      if (!__any_sync(__activemask(), act)) continue;
      if (!act) continue;
      const int d = rep == 0 ? 0 : (rep == 1 ? -1 : 1);
      double4 pl;
      if (NRM == 1 && rep == 0) {
        pl = reinterpret_cast<const double4*>(A.plane)[id];
        pl.w = plane_alpha(pl.x, pl.y, pl.z, cd);
      } else if (NRM == 2 && rep == 0) {
        pl = stencil_plane<F32, true>(g, c, x, y, z, stage != 0);
      } else {
        pl = stencil_plane<F32>(g, c, x + (AX == 0 ? d : 0), y + (AX == 1 ? d : 0), z + (AX == 2 ? d : 0), stage != 0);
      }
      // the faces it feeds: right (a > 0) and left (a < 0) for the cell, the
      // wall's face for a ghost; the volumes of a cell that feeds one face
      // are evaluated once per warp
      bool right = rep == 0 ? dgt0(ar) : rep == 1;
      bool left = rep == 0 ? dlt0(al) : rep == 2;
      const size_t lines = (size_t)g.n[0] * g.n[1] * g.n[2] / (size_t)n_ax;
      const size_t li = AX == 0 ? (size_t)z * g.n[1] + y : (AX == 1 ? (size_t)z * g.n[0] + x : (size_t)y * g.n[0] + x);
      while (right || left) {
        const bool pos = right;
        const double a = rep == 0 ? (pos ? ar : al) : (rep == 1 ? al : ar);
        const double vol = donor_volume(g, AX, pl, cd, fabs(a), pos, al, ar, A.status);
        if (rep == 0) {
          if (pos) A.fr[id] = vol;
          else A.fl[id] = -vol;
        } else {
          A.gf[(pos ? 0 : lines) + li] = pos ? vol : -vol;
        }
        if (pos) right = false;
        else left = false;
      }
    }
  }
}

template <int AX, bool F32, int NRM>
__global__ void __launch_bounds__(kMixThreads) k_mix(StepArgs A, int stage) {
  pdl_wait();
  mix_body<AX, F32, NRM>(A, stage, vb_self());
}

// ---------------------------------------------------------------------------
// k_walk
// ---------------------------------------------------------------------------
struct WalkWarp {
  double c[kRing * kRow];    // c of cell p; after the update of cell q, its new c in q's place
  double e[kRing * kRow];
  double u[kRingF * kRow];   // place p: the velocity of face p - 3
  double th[kRingF * kRow];  // place p: Theta of cell p - 4 (x walk, first stage: the new one after the update)
  uint32_t pend[2][kPend];   // mixed cells for the next stage's list (shift: [1] the edge cells)
};

// Appends the warp's pending entries to the grid-wide list (front, or from
// the back); the order varies from run to run and nothing depends on it.
__device__ __forceinline__ void walk_flush(uint32_t* pend, int& n, uint32_t* list, int* counter, size_t back, int lane) {
  if (n == 0) return;
  int b = 0;
  if (lane == 0) b = atomicAdd(counter, n);
  b = __shfl_sync(kFull, b, 0);
  __syncwarp();
  for (int i = lane; i < n; i += 32) {
    if (back) list[back - 1 - (size_t)(b + i)] = pend[i];
    else list[b + i] = pend[i];
  }
  __syncwarp();
  n = 0;
}

template <int AX, bool F32>
__device__ __forceinline__ void walk_body(const StepArgs& A, int stage, const VB vb, WalkWarp& W) {
  const GridDev& g = A.g;
  const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
  const int n_ax = g.n[AX], bca = g.bc[AX];
  const size_t stride = AX == 0 ? 1 : (AX == 1 ? (size_t)nx : (size_t)nx * ny);
  const size_t N = (size_t)nx * ny * nz;
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const int ntx = A.nt[0], nty = A.nt[1], nt_ax = A.nt[AX];
  const int T_all = ntx * nty * A.nt[2];
  const bool first = stage == 0, last = stage == 2;
  const bool frozen = g.le == 0;              // Weymouth-Yue: frozen cc and Theta
  const bool keep = frozen && !last;          // they are needed by a later stage
  const bool old_th = frozen && !first;       // Theta from memory
  const double* src = (stage & 1) ? A.s_c : A.c;
  const double* src_e = (stage & 1) ? A.s_e : A.e;
  double* dst = (stage & 1) ? A.c : A.s_c;
  double* dst_e = (stage & 1) ? A.e : A.s_e;
  const double* uf = A.uf[AX];
  const size_t lines = N / (size_t)n_ax;
  uint32_t* nlist = A.list[(stage + 1) & 1];

  // Work items: the halves (32 lines) of the active tiles one by one; where
  // they are too few to give every resident warp one, the two quarters (4
  // positions) of each half; or, where more than half of the tiles are active,
  // chains of L tiles along the axis.  An item of n positions enters n + 7
  // cells and evaluates n + 1 faces, so a quarter does a third more than its
  // share but halves a lone warp's latency, and a chain does less twice; chains
  // are kept short enough for six items a resident warp, which evens out their
  // differences.  (Batches of boxes fill the machine together: A.chain gives
  // their chain length, and no quarters are made.)
  const int nact = A.cnt[14];
  const long long resident = 152ll * kWalkPerSM * kWalkWarps;
  const bool quarters = A.chain == 0 && 4ll * nact <= resident;
  int L = A.chain > 1 ? A.chain : 1;
  if (A.chain == 0 && 2ll * nact > T_all) {
    const long long l = 2ll * nact / (6 * resident);
    L = l < 1 ? 1 : (l > 8 ? 8 : (int)l);
  }
  L = L > nt_ax ? nt_ax : L;
  const int cross = T_all / nt_ax;
  const bool chains = L > 1;
  const long long items = chains ? 2ll * cross * ((nt_ax + L - 1) / L) : (quarters ? 4ll : 2ll) * nact;
  const long long nwarp = (long long)vb.gx * kWalkWarps;

  int npend = 0, npend_e = 0, nfaces = 0;
  for (long long item = (long long)vb.bx * kWalkWarps + (threadIdx.x >> 5); item < items; item += nwarp) {
    const int hf = (int)(item & 1);
    const int part = quarters ? (int)(item >> 1 & 1) : 0;
    int tc[3], t_beg, t_end;  // tile coordinates; the item's tiles along the axis
    if (chains) {
      const int ch = (int)(item >> 1), cr = ch % cross, seg = ch / cross;
      t_beg = seg * L;
      t_end = min(t_beg + L, nt_ax);
      if (AX == 0) { tc[1] = cr % nty; tc[2] = cr / nty; tc[0] = t_beg; }
      else if (AX == 1) { tc[0] = cr % ntx; tc[2] = cr / ntx; tc[1] = t_beg; }
      else { tc[0] = cr % ntx; tc[1] = cr / ntx; tc[2] = t_beg; }
    } else {
      const int t = (int)A.tlist[item >> (quarters ? 2 : 1)];
      tc[0] = t % ntx;
      tc[1] = (t / ntx) % nty;
      tc[2] = t / (ntx * nty);
      t_beg = tc[AX];
      t_end = t_beg + 1;
    }
    // line r of the item: its two cross coordinates (8 along the first, 4
    // along the second cross axis)
    const int p0 = (AX == 0 ? tc[1] : tc[0]) * kTile, q0 = (AX == 2 ? tc[1] : tc[2]) * kTile + 4 * hf;
    const int np = AX == 0 ? ny : nx, nq = AX == 2 ? ny : nz;
    auto line_ok = [&](int r) { return p0 + (r & 7) < np && q0 + (r >> 3) < nq; };
    auto line_base = [&](int r) -> size_t {  // cell index of position 0
      const size_t p = (size_t)(p0 + (r & 7)), q = (size_t)(q0 + (r >> 3));
      return AX == 0 ? (q * ny + p) * nx : (AX == 1 ? q * ny * nx + p : q * nx + p);
    };
    auto face_base = [&](int r) -> size_t {  // face index of face 0
      const size_t p = (size_t)(p0 + (r & 7)), q = (size_t)(q0 + (r >> 3));
      return AX == 0 ? (q * ny + p) * (nx + 1) : (AX == 1 ? q * (ny + 1) * nx + p : q * nx + p);
    };
    auto tile_at = [&](int ta) -> int {  // tile index at ta along the axis
      return AX == 0 ? (tc[2] * nty + tc[1]) * ntx + ta : (AX == 1 ? (tc[2] * nty + ta) * ntx + tc[0]
                                                                   : (ta * nty + tc[1]) * ntx + tc[0]);
    };
    const bool act = line_ok(lane);
    const size_t lbase = act ? line_base(lane) : 0;

    for (int ta = t_beg; ta < t_end;) {
      if (chains && A.ts.quiet[tile_at(ta)]) { ++ta; continue; }
      int tb = ta + 1;
      while (tb < t_end && !A.ts.quiet[tile_at(tb)]) ++tb;
      int s0 = ta * kTile, s1 = min(tb * kTile, n_ax);
      ta = tb;
      if (quarters) {
        s0 += 4 * part;
        s1 = min(s0 + 4, s1);
        if (s0 >= s1) {  // no cell of this tile there (its line ends before)
          if (lane == 0) A.clip[(size_t)(4 * stage + 2 * hf + 1) * T_all + tile_at(s0 >> 3)] = 0.0;
          continue;
        }
      }
      const int lo = s0 - 3, hi = s1 + 3;
      const bool inl = s1 < n_ax || bca == 0;  // a cell lies beyond the segment's end

      // Asynchronous loads of the batch of positions pb .. pb + 3 into ring
      // rows row (c, e) and (pb & 4) (u, Theta): cells lo .. hi, faces s0 ..
      // s1 (of p - 3), Theta of cells s0 .. s1 - 1 (of p - 4).
      auto load_one = [&](int p, int pb, int row, int r, bool ok, size_t lb, size_t fb) {
        if (!ok) return;
        const int j = p - pb;
        if (p >= lo && p <= hi) {
          const bool in = p >= 0 && p < n_ax;
          const int q = in ? p : map_idx(p, n_ax, bca);
          const double *pc = src, *pe = src_e;
          // beyond the segment the tile may be quiet: its cells are in the caller's arrays
          if (!first && (p < s0 || p >= s1) && A.ts.quiet[tile_at(q >> 3)]) { pc = A.c; pe = A.e; }
          const size_t id = lb + stride * q;
          cp8(&W.c[(row + j) * kRow + r], pc + id);
          cp8(&W.e[(row + j) * kRow + r], pe + id);
        }
        const int f = p - 3, frow = ((pb & kBatch) + j) * kRow + r;
        if (f >= s0 && f <= s1) cp8(&W.u[frow], uf + fb + stride * ((bca == 0 && f == n_ax) ? 0 : f));
        if (old_th && f > s0 && f <= s1) cp8(&W.th[frow], A.theta + lb + stride * (f - 1));
      };
      auto load = [&](int pb, int row) {
        if (AX == 0) {
          const int p = pb + (lane & 3);
#pragma unroll 1
          for (int r = lane >> 2; r < 32; r += 8) load_one(p, pb, row, r, line_ok(r), line_base(r), face_base(r));
        } else {
          const size_t fb = act ? face_base(lane) : 0;
#pragma unroll 1
          for (int p = pb; p < pb + kBatch; ++p) load_one(p, pb, row, lane, act, lbase, fb);
        }
        cp_commit();
      };
      // x walk: the new values of the cells qb .. qb + 3 from the rings (row:
      // qb's c, e row) to memory
      auto store = [&](int qb, int row) {
        __syncwarp();
#pragma unroll 1
        for (int r = lane >> 2; r < 32; r += 8) {
          const int j = lane & 3, q = qb + j;
          if (line_ok(r) && q >= s0 && q < s1) {
            const size_t id = line_base(r) + q;
            dst[id] = W.c[(row + j) * kRow + r];
            dst_e[id] = W.e[(row + j) * kRow + r];
            if (first && keep) A.theta[id] = W.th[(((qb + kBatch) & kBatch) + j) * kRow + r];
          }
        }
        __syncwarp();
      };

      load(s0 - kBatch, 0);
      load(s0, kBatch);

      double Tq[5], Dq[6];  // T[p-4 .. p], D[p-6 .. p-1], D[j] = T[j+1] - T[j]
      double cq[5];         // c[p-4 .. p]
      double ep1 = 0.0, Fl = 0.0, Gl = 0.0, al = 0.0, clip = 0.0;
      int run = 0;
      bool listed_p = false;
      unsigned tags = 0u;   // of cells p, p - 1, ..: two bits each
      // bit i: at position p - i every line's c is 0 or 1 and its predecessor's
      unsigned same_c = 0u;
      int row = 1;          // ring row of position p (c, e): lo is the second of its batch
#pragma unroll
      for (int i = 0; i < 5; ++i) Tq[i] = cq[i] = 0.0;
#pragma unroll
      for (int i = 0; i < 6; ++i) Dq[i] = 0.0;

#pragma unroll 1
      for (int p = lo; p <= hi; ++p, row = row == kRing - 1 ? 0 : row + 1) {
        if ((p & (kBatch - 1)) == 0 || p == lo) {
          // the batch of p is complete; the next one goes where the cells
          // updated two batches ago were (the first two are both under way)
          cp_wait_all();
          __syncwarp();
          if (p >= s0) {
            const int nrow = row >= 2 * kBatch ? row - 2 * kBatch : row + kBatch;
            if (AX == 0 && p - 2 * kBatch >= s0) store(p - 2 * kBatch, nrow);
            if (p + kBatch <= hi) load(p + kBatch, nrow);
          }
        }
        const int slot = row * kRow + lane, fslot = (p & (kRingF - 1)) * kRow + lane;
        // cell p enters the window
        const double cw = W.c[slot], ev = W.e[slot];
        const double cv = first ? cw : c_value(cw);
        tags = tags << 2 | (first ? 0u : c_tag(cw));
        const bool sc = p > lo && same_bits(cv, cq[4]), pure = is01(cv);
        const bool same = sc && same_bits(ev, ep1);
        run = same ? run + 1 : 1;
#pragma unroll
        for (int i = 0; i < 4; ++i) { Tq[i] = Tq[i + 1]; cq[i] = cq[i + 1]; }
#pragma unroll
        for (int i = 0; i < 5; ++i) Dq[i] = Dq[i + 1];
        cq[4] = cv;
        ep1 = ev;
        same_c = same_c << 1 | (__all_sync(kFull, !act || (sc && pure)) ? 1u : 0u);
        if (__any_sync(kFull, act && !same)) {
          double T = ev * (dbits(cv) ? g.rCp_l : g.rCp_g);
          if (!(same_c & 1u) && !pure) T = temp_of(g, ev, cv);
          Dq[5] = same ? 0.0 : T - Tq[3];
          Tq[4] = same ? Tq[3] : T;
        } else {
          Dq[5] = 0.0;
          Tq[4] = Tq[3];
        }
        if (p < s0 + 3) continue;

        // face k, between cells k - 1 and k
        const int k = p - 3;
        const bool listed = act && (k < s1 || inl) && !(run >= 7 && is01(cq[1]) && !(tags >> 6 & 1u));
        nfaces += (k < s1 && listed ? 1 : 0) + (listed_p && !listed ? 1 : 0);
        double Fv = 0.0, Gv = 0.0, a = 0.0;
        const bool any_l = __any_sync(kFull, listed_p);
        if (any_l || __any_sync(kFull, listed && k < s1)) {
          a = W.u[fslot] * g.lam;
          const bool pos = dgt0(a);
          const double cd = pos ? cq[0] : cq[1];
          const double Tf = face_temperature(F32, pos ? Tq[0] : Tq[1], pos ? Dq[0] : dneg(Dq[4]), pos ? Dq[1] : dneg(Dq[3]),
                                             pos ? Dq[2] : dneg(Dq[2]), pos ? Dq[3] : dneg(Dq[1]));
          if (same_c & 8u) {  // cells k - 1 and k hold the same 0 or 1 on every line
            Fv = flux01(cd, a);
            Gv = energy_flux01(g, Tf, cd, a);
          } else {
            Fv = pure_flux(cd, a);
            if (act && dnz(a) && is_mixed_b(cd, g)) {
              const int dq = pos ? k - 1 : k;  // the donor's position
              if (bca != 0 && (dq < 0 || dq >= n_ax)) {
                const size_t li = AX == 0 ? lbase / (size_t)nx : (size_t)(q0 + (lane >> 3)) * nx + p0 + (lane & 7);
                Fv = A.gf[(dq < 0 ? 0 : lines) + li];
              } else {
                const size_t di = lbase + stride * map_idx(dq, n_ax, bca);
                Fv = pos ? A.fr[di] : A.fl[di];
              }
            }
            Gv = energy_flux(g, Tf, cd, Fv, a);
          }
          if (!dnz(a)) { Fv = 0.0; Gv = 0.0; }
        }
        if (k > s0) {  // cell k - 1, between its two faces
          const int q = k - 1;
          const int qs = (row >= kBatch ? row - kBatch : row + 2 * kBatch) * kRow + lane;
          const double c = cq[0], e = W.e[qs];
          double cn = c, en = e;
          unsigned tag = tags >> 8 & 3u;
          double th = 0.0;
          const bool dirty = (tag & 1u) != 0;
          const bool cc = dirty ? (tag & 2u) != 0 : dgthalf(c);
          const bool own = (same_c & 24u) == 24u;  // cells k - 2, k - 1, k likewise: both donors are c
          if (any_l || (first && keep)) {
            if (old_th) th = W.th[fslot];
            else th = own || frozen ? (cc ? g.Cp_l : g.Cp_g) * Tq[0] : theta_now(g, Tq[0], c, cc, true);
          }
          const bool csame = own && (first || __all_sync(kFull, !act || cc == (dbits(c) != 0)));
          if (any_l) {
            const double e2 = (e + (Gl - th * al)) - (Gv - th * a);
            if (listed_p) en = e2;
            if (!csame) {
              const double2 r = update_c(c, Fl, al, Fv, a, cc, !frozen);
              if (listed_p) {
                cn = r.x;
                if (dnz(r.y)) clip += r.y;
              }
            }
            if (listed_p && !dirty && (!deq(cn, c) || !deq(en, e))) tag = 1u | (cc ? 2u : 0u);
          }
          if (!keep) tag = 0u;
          const size_t id = lbase + stride * q;
          if (!csame) {
            const bool mixed = act && is_mixed_b(cn, g);
            if (__any_sync(kFull, mixed)) {
              bool take = mixed;
              if (last) {
                // the shift moves the mixed cells with a nonzero shift
                double ddv = A.dd_uniform;
                if (mixed && A.dd) ddv = __ldg(A.dd + id);
                tag = mixed && dnz(ddv) ? (dlt0(ddv) ? 1u : 2u) : 0u;
                const bool edge = tag != 0 && shift_edge(cn);
                take = tag != 0 && !edge;
                const unsigned me = __ballot_sync(kFull, edge);
                if (me) {
                  if (edge) W.pend[1][npend_e + __popc(me & lt)] = (uint32_t)id;
                  npend_e += __popc(me);
                  if (npend_e > kPend - 32) walk_flush(W.pend[1], npend_e, nlist, A.cnt + 13, N, lane);
                }
              }
              const unsigned mt = __ballot_sync(kFull, take);
              if (mt) {
                if (take) W.pend[0][npend + __popc(mt & lt)] = (uint32_t)id;
                npend += __popc(mt);
                if (npend > kPend - 32) walk_flush(W.pend[0], npend, nlist, A.cnt + 4 * (stage + 1), 0, lane);
              }
            }
          }
          const double cnw = tag ? c_with(cn, tag) : cn;
          if (AX == 0) {
            W.c[qs] = cnw;
            W.e[qs] = en;
            if (first && keep) W.th[fslot] = th;
          } else if (act) {
            dst[id] = cnw;
            dst_e[id] = en;
            if (first && keep) A.theta[id] = th;
          }
          if ((q & 3) == 3 || q == s1 - 1) {
            // the clipped volume of this quarter of the tile, one slot per stage
            double cs = 0.0;
            if (__any_sync(kFull, dnz(clip))) {
              cs = clip;
#pragma unroll
              for (int o = 16; o > 0; o >>= 1) cs += __shfl_down_sync(kFull, cs, o);
              clip = 0.0;
            }
            if (lane == 0) {
              double* slot0 = A.clip + (size_t)(4 * stage + 2 * hf) * T_all + tile_at(q >> 3);
              slot0[(q & 4) ? T_all : 0] = cs;
              if (!quarters && q == s1 - 1 && !(q & 4)) slot0[T_all] = 0.0;  // a line's end in the first quarter
            }
          }
        }
        Fl = Fv;
        Gl = Gv;
        al = a;
        listed_p = listed && k < s1;
      }
      if (AX == 0) {
        // the cells of the last two batches that the loop has not stored
        const int pe = hi & ~(kBatch - 1);                       // the batch of hi
        const int er = row >= (hi & (kBatch - 1)) + 1 ? row - (hi & (kBatch - 1)) - 1 : row + kRing - (hi & (kBatch - 1)) - 1;
        const int r1 = er >= kBatch ? er - kBatch : er + 2 * kBatch;  // of the batch before
        if (pe - kBatch >= s0) store(pe - kBatch, r1);
        store(pe, er);
      }
      __syncwarp();
    }
  }
  walk_flush(W.pend[0], npend, nlist, A.cnt + 4 * (stage + 1), 0, lane);
  if (last) walk_flush(W.pend[1], npend_e, nlist, A.cnt + 13, N, lane);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) nfaces += __shfl_down_sync(kFull, nfaces, o);
  if (lane == 0 && nfaces) atomicAdd(A.cnt + 4 * stage + 1, nfaces);
}

template <int AX, bool F32>
__global__ void __launch_bounds__(32 * kWalkWarps, kWalkPerSM) k_walk(StepArgs A, int stage) {
  __shared__ WalkWarp W[kWalkWarps];
  pdl_wait();
  walk_body<AX, F32>(A, stage, vb_self(), W[threadIdx.x >> 5]);
}

// Grouped: every box of a batch in one launch, each CTA on its box's arguments.
template <int AX, bool F32, int NRM>
__global__ void __launch_bounds__(kMixThreads) k_mix_grp(GroupMap m, const StepArgs* __restrict__ args, int stage) {
  unsigned b;
  const VB vb = vb_group(m, b);
  __shared__ StepArgs sA;
  mix_body<AX, F32, NRM>(cta_args(args, b, sA), stage, vb);
}
template <int AX, bool F32>
__global__ void __launch_bounds__(32 * kWalkWarps, kWalkPerSM)
k_walk_grp(GroupMap m, const StepArgs* __restrict__ args, int stage) {
  __shared__ WalkWarp W[kWalkWarps];
  unsigned b;
  const VB vb = vb_group(m, b);
  __shared__ StepArgs sA;
  walk_body<AX, F32>(cta_args(args, b, sA), stage, vb, W[threadIdx.x >> 5]);
}

// CTAs of k_mix: one mixed cell per thread up to one wave; cells outnumber
// the mixed ones by far, so a box of a batch gets one per `work` cells
unsigned mix_ctas(const GridDev& g) {
  const size_t N = (size_t)g.n[0] * g.n[1] * g.n[2];
  return (unsigned)std::min<size_t>((N + kMixThreads - 1) / kMixThreads, 152 * 4);
}
// CTAs of k_walk: a warp per tile quarter, at most one wave
unsigned walk_ctas(const GridDev& g) {
  return (unsigned)std::min<long long>((4ll * tile_total(g) + kWalkWarps - 1) / kWalkWarps, 152 * kWalkPerSM);
}

// In a batch of boxes (no quarters): per_warp halves or chains of halves a warp if
// every tile is active.
unsigned walk_ctas_grp(const GridDev& g, int chain, int per_warp) {
  const long long items = 2ll * tile_total(g) / chain;
  return (unsigned)std::max<long long>(1, (items + per_warp * kWalkWarps - 1) / (per_warp * kWalkWarps));
}

template <int AX>
static cudaError_t stage_t(const StepArgs& A, int stage, cudaStream_t st) {
  const GridDev& g = A.g;
  const unsigned nm = mix_ctas(g);
  if (g.mlp == 1) {
    const cudaError_t err = launch_mlp_sweep_normals(g, (stage & 1) ? A.s_c : A.c, stage != 0, A.list[stage & 1],
                                                     A.cnt + 4 * stage, A.plane, st);
    if (err != cudaSuccess) return err;
    if (g.f32) launch_pdl(k_mix<AX, true, 1>, nm, kMixThreads, st, A, stage);
    else launch_pdl(k_mix<AX, false, 1>, nm, kMixThreads, st, A, stage);
  } else if (g.mlp == 2) {
    launch_pdl(k_mix<AX, false, 2>, nm, kMixThreads, st, A, stage);
  } else if (g.f32) {
    launch_pdl(k_mix<AX, true, 0>, nm, kMixThreads, st, A, stage);
  } else {
    launch_pdl(k_mix<AX, false, 0>, nm, kMixThreads, st, A, stage);
  }
  prof_mark(AX == 0 ? "sweep_x.mix" : (AX == 1 ? "sweep_y.mix" : "sweep_z.mix"), st);
  if (g.f32) launch_pdl(k_walk<AX, true>, walk_ctas(g), 32 * kWalkWarps, st, A, stage);
  else launch_pdl(k_walk<AX, false>, walk_ctas(g), 32 * kWalkWarps, st, A, stage);
  prof_mark(AX == 0 ? "sweep_x.walk" : (AX == 1 ? "sweep_y.walk" : "sweep_z.walk"), st);
  return cudaGetLastError();
}

cudaError_t launch_stage(const StepArgs& A, int axis, int stage, cudaStream_t st) {
  if (axis == 0) return stage_t<0>(A, stage, st);
  if (axis == 1) return stage_t<1>(A, stage, st);
  return stage_t<2>(A, stage, st);
}

template <int AX>
static void stage_grp_t(int f32, int youngs, const GroupMap* m, const unsigned* n, const StepArgs* a, int stage,
                        cudaStream_t st) {
  if (n[0]) {
    if (youngs) k_mix_grp<AX, false, 2><<<n[0], kMixThreads, 0, st>>>(m[0], a, stage);
    else if (f32) k_mix_grp<AX, true, 0><<<n[0], kMixThreads, 0, st>>>(m[0], a, stage);
    else k_mix_grp<AX, false, 0><<<n[0], kMixThreads, 0, st>>>(m[0], a, stage);
  }
  prof_mark("group.mix", st);
  if (n[1]) {
    if (f32) k_walk_grp<AX, true><<<n[1], 32 * kWalkWarps, 0, st>>>(m[1], a, stage);
    else k_walk_grp<AX, false><<<n[1], 32 * kWalkWarps, 0, st>>>(m[1], a, stage);
  }
  prof_mark("group.walk", st);
}

cudaError_t launch_stage_grp(int axis, int stage, int f32, int youngs, const GroupMap* maps, const unsigned* ctas,
                             const StepArgs* a, cudaStream_t st) {
  if (axis == 0) stage_grp_t<0>(f32, youngs, maps, ctas, a, stage, st);
  else if (axis == 1) stage_grp_t<1>(f32, youngs, maps, ctas, a, stage, st);
  else stage_grp_t<2>(f32, youngs, maps, ctas, a, stage, st);
  return cudaGetLastError();
}

}  // namespace vofgb
