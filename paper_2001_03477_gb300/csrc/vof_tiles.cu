// vof_tiles.cu -- the tile pass at the start of an in-place time step: which
// 8^3 tiles are quiet (no cell of them can change in this step, so the
// step's kernels skip them), the list of the others, the mixed cells the first
// sweep starts from, and the quiet tiles' shares of the sums of c and e.
//
// A tile is uniform when all its cells hold the same (c, e) bits; it is quiet
// when it is uniform with c exactly 0 or 1 and every one of its 26 neighbour
// tiles is uniform with the same bits.  The neighbours then contain the 3-cell
// halo of the tile, so every 7-cell sweep window of a tile cell, and every
// window the earlier sweeps of the step use for the cells those windows
// reach, sees one value: the cells are no-ops in all three sweeps (a cell
// that does not change is not marked in the frozen state either) and remain
// pure for the shift.  Beyond a zero-gradient boundary the halo repeats the
// boundary cells, so a missing neighbour tile counts as equal; a periodic
// axis wraps.  On a periodic axis whose last tile holds fewer than 3 cells
// the halo of the first tile reaches past it into the one before, and that
// one's into the first: the two are neighbours as well.  (Where such grids
// skipped no tile, two steps of a 118 x 165 x 153 drop took 1234 us, now 646.)
#include "vof_launch.h"
#include "vof_sums.cuh"

namespace vofgb {

namespace {

constexpr unsigned kFullT = 0xffffffffu;


// CTA: 32 x 8 threads covering four tiles along x (32 cells), one along y
// and one along z (the threads walk its 8 planes).  Each tile's flag and
// reference values; integer compares only (no FP64 work and nothing kept
// beyond registers), so the pass streams c and e at the memory's rate.
__device__ __forceinline__ void k_tiles_body(const GridDev& g, const double* __restrict__ c, const double* __restrict__ e, const TileScratch& ts, int ntx, int nty, int* __restrict__ counters, int* __restrict__ stats, const VB vb) {
  __shared__ unsigned uni_w[8];
  __shared__ double ref[4][2];
  const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int j = tx >> 3;  // tile of this thread within the CTA
  const int x = vb.bx * 32 + tx, y = vb.by * kTile + ty, z0 = vb.bz * kTile;
  const int xt = vb.bx * 4 + j;
  const bool tile_ok = xt * kTile < nx;
  long long cb[kTile], eb[kTile];
  const bool xy_ok = x < nx && y < ny;
#pragma unroll
  for (int zi = 0; zi < kTile; ++zi) {
    const int z = z0 + zi;
    const bool ok = xy_ok && z < nz;
    const size_t id = ((size_t)z * ny + y) * nx + x;
    cb[zi] = ok ? dbits(__ldg(c + id)) : 0;
    eb[zi] = ok ? dbits(__ldg(e + id)) : 0;
  }
  if ((vb.bx | vb.by | vb.bz) == 0 && ty == 0 && tx < kStepCounters) {
    counters[tx] = 0;
    if (tx == 0) stats[8] = 0;  // receivers, counted by the step's last kernel
  }
  // reference of each tile: its first cell, which this CTA's thread
  // (8 j, 0) holds as its first value
  if (ty == 0 && (tx & 7) == 0 && tile_ok) {
    ref[j][0] = __longlong_as_double(cb[0]);
    ref[j][1] = __longlong_as_double(eb[0]);
  }
  __syncthreads();
  const long long cr = tile_ok ? dbits(ref[j][0]) : 0, er = tile_ok ? dbits(ref[j][1]) : 0;
  bool uniform = true;
#pragma unroll
  for (int zi = 0; zi < kTile; ++zi)
    if (xy_ok && z0 + zi < nz) uniform = uniform && cb[zi] == cr && eb[zi] == er;
  const unsigned bal = __ballot_sync(kFullT, uniform);
  if (tx == 0) uni_w[ty] = bal;
  __syncthreads();
  if (ty == 0 && (tx & 7) == 0 && tile_ok) {
    unsigned all = 0xffffffffu;
#pragma unroll
    for (int w = 0; w < 8; ++w) all &= uni_w[w];
    const bool tile_uni = ((all >> (8 * j)) & 0xFFu) == 0xFFu;
    const size_t t = ((size_t)vb.bz * nty + vb.by) * ntx + xt;
    ts.uni[t] = tile_uni ? 1 : 0;
    ts.vc[t] = __longlong_as_double(cr);
    ts.ve[t] = __longlong_as_double(er);
  }
}

// (c and e are read at addresses known from the start, and the grid ahead on the
// stream may be what writes them: the step before without sums, a program's own
// kernel)
__global__ void __launch_bounds__(256) k_tiles(StepArgs A) {
  pdl_wait();
  k_tiles_body(A.g, after_wait(A.c), after_wait(A.e), A.ts, A.nt[0], A.nt[1], A.cnt, A.stats, vb_self());
}

// neighbour tile index along one axis: -1 when it lies beyond a
// zero-gradient boundary (the halo repeats the boundary: counts as equal),
// wrapped on a periodic axis
__device__ __forceinline__ int tile_nb(int p, int n, int bc) {
  if (p < 0) return bc ? -1 : p + n;
  if (p >= n) return bc ? -1 : p - n;
  return p;
}

// the further neighbour of tile p along a periodic axis whose last tile holds
// fewer than 3 cells, or -2 where there is none (up to 3 tiles the next ones
// are all there are)
__device__ __forceinline__ int tile_far(int p, int n, int cells, int bc) {
  const int r = cells & (kTile - 1);
  if (bc != 0 || r == 0 || r > 2 || n < 4) return -2;
  return p == 0 ? n - 2 : (p == n - 2 ? 0 : -2);
}

// n x v for the bit pattern v (the same for every lane of the warp): a
// whole tile (n = 512 = 2^9) by adding 9 to the exponent when the product is
// a normal number, and +-0 as itself -- both exact, as the FP64 product is,
// and without an FP64 instruction; otherwise the FP64 product, in a call
// under a warp vote so that the common case issues no predicated multiply
__device__ __noinline__ double times_cells_mul(int n, long long v) { return (double)n * __longlong_as_double(v); }
__device__ __forceinline__ double times_cells(int n, long long v) {
  const int ex = (int)((v >> 52) & 0x7FF);
  const bool shift = n == kTile * kTile * kTile && ex >= 1 && ex <= 0x7FE - 9;
  const bool zero = ((unsigned long long)v << 1) == 0ull;
  double r = __longlong_as_double(shift ? v + (9LL << 52) : v);
  if (__any_sync(kFullT, !shift && !zero)) r = times_cells_mul(n, v);
  return r;
}

// One warp per tile: quiet flag (lanes 0..26 check the tile and its 26
// neighbours at once; the far ones, where there are any, in two rounds).  A quiet tile's sum row is (cells) x value; any other
// tile joins the active list, and its mixed cells the first stage's list
// (one atomic per tile and list; both orders vary from run to run).
__device__ __forceinline__ void k_quiet_body(const StepArgs& A, const VB vb) {
  const GridDev& g = A.g;
  const TileScratch& ts = A.ts;
  const int ntx = A.nt[0], nty = A.nt[1], ntz = A.nt[2];
  const long long nt = (long long)ntx * nty * ntz;
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const long long wpb = blockDim.x >> 5;
  // tile t goes to CTA t mod gx: neighbouring tiles (the interface's, whose
  // cells are read) spread over the SMs
  for (long long t = vb.bx + (long long)vb.gx * (threadIdx.x >> 5); t < nt; t += (long long)vb.gx * wpb) {
    const int tx = (int)(t % ntx), ty = (int)((t / ntx) % nty), tz = (int)(t / ((long long)ntx * nty));
    // lane o < 27: the tile at offset (o % 3 - 1, o / 3 % 3 - 1, o / 9 - 1);
    // one beyond a zero-gradient boundary counts as equal
    bool nb_ok = true, nb_uni = true;
    long long nb_c = 0, nb_e = 0;
    auto look = [&](int px, int py, int pz) {
      nb_ok = (px | py | pz) >= 0;
      if (nb_ok) {
        const size_t u = ((size_t)pz * nty + py) * ntx + px;
        nb_uni = ts.uni[u] != 0;
        nb_c = dbits(ts.vc[u]);
        nb_e = dbits(ts.ve[u]);
      }
    };
    if (lane < 27)
      look(tile_nb(tx + lane % 3 - 1, ntx, g.bc[0]), tile_nb(ty + (lane / 3) % 3 - 1, nty, g.bc[1]),
           tile_nb(tz + lane / 9 - 1, ntz, g.bc[2]));
    const bool uni = __shfl_sync(kFullT, nb_uni ? 1 : 0, 13) != 0;  // lane 13: the tile itself
    const long long cr = __shfl_sync(kFullT, nb_c, 13), er = __shfl_sync(kFullT, nb_e, 13);
    bool same = lane >= 27 || !nb_ok || (nb_uni && nb_c == cr && nb_e == er);
    const int fx = tile_far(tx, ntx, g.n[0], g.bc[0]), fy = tile_far(ty, nty, g.n[1], g.bc[1]),
              fz = tile_far(tz, ntz, g.n[2], g.bc[2]);
    if (fx >= 0 || fy >= 0 || fz >= 0) {  // a far neighbour is a fourth choice along its axis
      const int kx = fx >= 0 ? 4 : 3, ky = fy >= 0 ? 4 : 3, kz = fz >= 0 ? 4 : 3;
      for (int o = lane; o < kx * ky * kz; o += 32) {
        const int ox = o % kx, oy = (o / kx) % ky, oz = o / (kx * ky);
        look(ox == 3 ? fx : tile_nb(tx + ox - 1, ntx, g.bc[0]), oy == 3 ? fy : tile_nb(ty + oy - 1, nty, g.bc[1]),
             oz == 3 ? fz : tile_nb(tz + oz - 1, ntz, g.bc[2]));
        same = same && (!nb_ok || (nb_uni && nb_c == cr && nb_e == er));
      }
    }
    const bool all = __all_sync(kFullT, same);
    const bool pure = cr == 0 || cr == 0x3FF0000000000000LL;
    const bool q = uni && pure && all;
    const int x0 = tx * kTile, y0 = ty * kTile, z0 = tz * kTile;
    if (lane == 0) ts.quiet[t] = q ? 1 : 0;
    if (q) {
      const int n = min(kTile, g.n[0] - x0) * min(kTile, g.n[1] - y0) * min(kTile, g.n[2] - z0);
      const double sc = times_cells(n, cr), se = times_cells(n, er);
      if (lane < kNSums) A.rows[(size_t)t * kNSums + lane] = lane == kSumC ? sc : (lane == kSumE ? se : 0.0);
      continue;
    }
    if (lane == 0) A.tlist[atomicAdd(A.cnt + 14, 1)] = (uint32_t)t;
    if (uni && pure) continue;  // no mixed cell
    unsigned mine = 0u;  // bit r: this lane's r-th cell is mixed
#pragma unroll
    for (int r = 0; r < kTile * kTile * kTile / 32; ++r) {
      const int o = lane + 32 * r, x = x0 + (o & 7), y = y0 + ((o >> 3) & 7), z = z0 + (o >> 6);
      if (x < g.n[0] && y < g.n[1] && z < g.n[2] &&
          is_mixed_b(__ldg(A.c + ((size_t)z * g.n[1] + y) * g.n[0] + x), g))
        mine |= 1u << r;
    }
    const int k = __popc(mine);
    const int total = __reduce_add_sync(kFullT, k);
    if (total == 0) continue;
    int base = 0;
    if (lane == 0) base = atomicAdd(A.cnt + 0, total);
    base = __shfl_sync(kFullT, base, 0);
#pragma unroll 1
    for (int r = 0; r < kTile * kTile * kTile / 32; ++r) {
      const unsigned m = __ballot_sync(kFullT, (mine >> r) & 1u);
      if ((mine >> r) & 1u) {
        const int o = lane + 32 * r;
        A.list[0][base + __popc(m & lt)] =
            (uint32_t)(((size_t)(z0 + (o >> 6)) * g.n[1] + y0 + ((o >> 3) & 7)) * g.n[0] + x0 + (o & 7));
      }
      base += __popc(m);
    }
  }
}

__global__ void __launch_bounds__(256) k_quiet(StepArgs A) {
  pdl_wait();
  k_quiet_body(A, vb_self());
}

size_t al256t(size_t b) { return (b + 255) & ~(size_t)255; }

}  // namespace

void tile_counts(const GridDev& g, int nt[3]) {
  for (int a = 0; a < 3; ++a) nt[a] = (g.n[a] + kTile - 1) / kTile;
}

int tile_total(const GridDev& g) {
  int nt[3];
  tile_counts(g, nt);
  return nt[0] * nt[1] * nt[2];
}

size_t tile_scratch_bytes(const GridDev& g) {
  int nt[3];
  tile_counts(g, nt);
  const size_t T = (size_t)nt[0] * nt[1] * nt[2];
  return al256t(T) + al256t(T * 8) + al256t(T * 8) + al256t(T);
}

TileScratch carve_tile_scratch(const GridDev& g, void* ws) {
  int nt[3];
  tile_counts(g, nt);
  const size_t T = (size_t)nt[0] * nt[1] * nt[2];
  char* b = static_cast<char*>(ws);
  TileScratch s;
  s.uni = reinterpret_cast<uint8_t*>(b);   b += al256t(T);
  s.vc = reinterpret_cast<double*>(b);     b += al256t(T * 8);
  s.ve = reinterpret_cast<double*>(b);     b += al256t(T * 8);
  s.quiet = reinterpret_cast<uint8_t*>(b);
  return s;
}

__global__ void __launch_bounds__(256) k_tiles_grp(GroupMap m, const StepArgs* __restrict__ args) {
  unsigned b;
  const VB vb = vb_group(m, b);
  __shared__ StepArgs sA;
  const StepArgs& A = cta_args(args, b, sA);
  k_tiles_body(A.g, A.c, A.e, A.ts, A.nt[0], A.nt[1], A.cnt, A.stats, vb);
}
__global__ void __launch_bounds__(256) k_quiet_grp(GroupMap m, const StepArgs* __restrict__ args) {
  unsigned b;
  const VB vb = vb_group(m, b);
  __shared__ StepArgs sA;
  k_quiet_body(cta_args(args, b, sA), vb);
}

cudaError_t launch_tiles_grp(const GroupMap& mt, const GroupMap& mq, const StepArgs* a, unsigned ct, unsigned cq,
                             cudaStream_t st) {
  if (ct) k_tiles_grp<<<ct, dim3(32, 8), 0, st>>>(mt, a);
  prof_mark("group.tiles", st);
  if (cq) k_quiet_grp<<<cq, 256, 0, st>>>(mq, a);
  prof_mark("group.quiet", st);
  return cudaGetLastError();
}

unsigned quiet_ctas(const GridDev& g) {
  const long long T = tile_total(g);
  // one warp per tile, 8 per CTA
  return (unsigned)((T + 7) / 8 < 152 * 8 ? (T + 7) / 8 : 152 * 8);
}

cudaError_t launch_tiles(const StepArgs& A, cudaStream_t st) {
  launch_pdl(k_tiles, dim3((unsigned)((A.nt[0] + 3) / 4), (unsigned)A.nt[1], (unsigned)A.nt[2]), dim3(32, 8), st, A);
  prof_mark("tiles", st);
  launch_pdl(k_quiet, quiet_ctas(A.g), 256, st, A);
  prof_mark("tiles.quiet", st);
  return cudaGetLastError();
}

}  // namespace vofgb
