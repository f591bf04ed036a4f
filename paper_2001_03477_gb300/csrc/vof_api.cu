// vof_api.cu -- C ABI of the library (declared in include/vofgb.h): argument
// checks, parameter marshalling and the stream-ordered time step.
#include <cstring>
#include <mutex>

#include "../../include/vofgb.h"
#include "vof_launch.h"

namespace vofgb {

__device__ int g_vof_status;

static thread_local int t_last_cuda = 0;

void set_last_cuda_error(int err) { t_last_cuda = err; }

int* device_status_ptr() {
  static std::mutex mu;
  static int* ptrs[64] = {nullptr};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
  std::lock_guard<std::mutex> lk(mu);
  if (!ptrs[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_vof_status) != cudaSuccess) return nullptr;
    ptrs[dev] = static_cast<int*>(p);
  }
  return ptrs[dev];
}

static bool grid_ok(const vof_grid* g) {
  if (!g) return false;
  if (g->nx < 1 || g->ny < 1 || g->nz < 1) return false;
  // cell lists hold 32-bit entries (cell index << 1 | face side)
  if ((long long)g->nx * g->ny * g->nz >= (1LL << 31)) return false;
  for (int d = 0; d < 3; ++d)
    if (g->bc[d] != 0 && g->bc[d] != 1) return false;
  if (!(g->h > 0.0) || !(g->Cp_l > 0.0) || !(g->Cp_g > 0.0)) return false;
  if (!(g->eps_mixed >= 0.0 && g->eps_mixed < 0.5)) return false;
  if (g->precision != VOF_F64 && g->precision != VOF_F32_FLUX) return false;
  if (g->scheme != VOF_SCHEME_WY && g->scheme != VOF_SCHEME_LE) return false;
  if (g->normal != VOF_NORMAL_MYC && g->normal != VOF_NORMAL_MLP && g->normal != VOF_NORMAL_YOUNGS) return false;
  if (g->normal == VOF_NORMAL_MLP && (!g->mlp || ((uintptr_t)g->mlp & 15) != 0)) return false;
  return true;
}

static GridDev to_dev(const vof_grid* g, double dt) {
  GridDev d;
  d.n[0] = g->nx; d.n[1] = g->ny; d.n[2] = g->nz;
  d.bc[0] = g->bc[0]; d.bc[1] = g->bc[1]; d.bc[2] = g->bc[2];
  d.lam = dt / g->h;
  d.Cp_l = g->Cp_l; d.Cp_g = g->Cp_g; d.T_sat = g->T_sat; d.eps = g->eps_mixed;
  d.rCp_l = 1.0 / g->Cp_l;
  d.rCp_g = 1.0 / g->Cp_g;
  double ome = 1.0 - g->eps_mixed;
  std::memcpy(&d.eps_bits, &g->eps_mixed, 8);
  std::memcpy(&d.one_m_eps, &ome, 8);
  d.f32 = g->precision == VOF_F32_FLUX ? 1 : 0;
  d.le = g->scheme == VOF_SCHEME_LE ? 1 : 0;
  d.mlp = g->normal == VOF_NORMAL_MLP ? 1 : (g->normal == VOF_NORMAL_YOUNGS ? 2 : 0);
  d.mlp_params = d.mlp == 1 ? g->mlp : nullptr;
  return d;
}

static size_t cells(const vof_grid* g) { return (size_t)g->nx * g->ny * g->nz; }

static size_t face_count(const vof_grid* g, int axis) {
  size_t nx = g->nx, ny = g->ny, nz = g->nz;
  if (axis == 0) return nz * ny * (nx + 1);
  if (axis == 1) return nz * (ny + 1) * nx;
  return (nz + 1) * ny * nx;
}

static bool overlap(const void* a, size_t na, const void* b, size_t nb) {
  if (!a || !b) return false;
  const char* pa = static_cast<const char*>(a);
  const char* pb = static_cast<const char*>(b);
  return pa < pb + nb && pb < pa + na;
}

static vof_status cuda_status(cudaError_t e) {
  if (e == cudaSuccess) return VOF_OK;
  t_last_cuda = (int)e;
  return VOF_ECUDA;
}

static size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

}  // namespace vofgb

using namespace vofgb;

extern "C" {

vof_status vof_reconstruct(const vof_grid* g, const double* c, double* m, double* alpha, uint8_t* mixed,
                           void* stream) {
  if (!grid_ok(g) || !c || !m || !alpha || !mixed) return VOF_EINVAL;
  size_t N = cells(g);
  if (overlap(c, N * 8, m, 3 * N * 8) || overlap(c, N * 8, alpha, N * 8) || overlap(c, N * 8, mixed, N))
    return VOF_EINVAL;
  return cuda_status(launch_reconstruct(to_dev(g, 0.0), c, m, alpha, mixed, (cudaStream_t)stream));
}

size_t vof_sweep_workspace_bytes(const vof_grid* g) {
  if (!grid_ok(g)) return 0;
  return sweep_scratch_bytes(to_dev(g, 0.0));
}

static vof_status sweep_common(int axis, const vof_grid* g, const double* c_in, const double* e_in, double* c_out,
                               double* e_out, const double* uf, double dt, uint8_t* state, double* theta,
                               double* flux_out, double* diag, void* workspace, size_t workspace_bytes,
                               void* stream) {
  if (!grid_ok(g) || !c_in || !c_out || !uf || !workspace) return VOF_EINVAL;
  if (e_in && (!e_out || (state && !theta))) return VOF_EINVAL;
  if (!(dt >= 0.0)) return VOF_EINVAL;
  if (((uintptr_t)workspace & 255) != 0) return VOF_EINVAL;
  const GridDev d = to_dev(g, dt);
  const size_t need = sweep_scratch_bytes(d);
  if (workspace_bytes < need) return VOF_EINVAL;
  size_t N = cells(g), B = N * 8;
  // either fully in place (c_out == c_in and e_out == e_in) or no overlap
  const bool inplace = c_out == c_in && (!e_in || e_out == e_in);
  if (!inplace) {
    if (overlap(c_in, B, c_out, B)) return VOF_EINVAL;
    if (e_in && (overlap(e_in, B, e_out, B) || overlap(c_in, B, e_out, B) || overlap(e_in, B, c_out, B)))
      return VOF_EINVAL;
  }
  if (e_in && (overlap(c_out, B, e_out, B) || overlap(c_in, B, e_in, B))) return VOF_EINVAL;
  if (flux_out && (overlap(flux_out, face_count(g, axis) * 8, c_out, B) ||
                   (e_out && overlap(flux_out, face_count(g, axis) * 8, e_out, B))))
    return VOF_EINVAL;
  if (overlap(workspace, need, c_in, B) || overlap(workspace, need, c_out, B) ||
      (e_in && (overlap(workspace, need, e_in, B) || overlap(workspace, need, e_out, B))))
    return VOF_EINVAL;
  // stand-alone sweep: diag[0] += clipped volume
  static const signed char kMap[kNSums] = {-1, -1, 0, -1, -1, -1};
  SweepScratch sc = carve_sweep_scratch(axis, d, workspace, sums_to_diag(diag, kMap));
  return cuda_status(launch_sweep(axis, d, c_in, e_in, c_out, e_in ? e_out : nullptr, uf, state, theta, flux_out, sc,
                                  (cudaStream_t)stream));
}

vof_status vof_advect_sweep_x(const vof_grid* g, const double* c_in, const double* e_in, double* c_out,
                              double* e_out, const double* u_face, double dt, uint8_t* state, double* theta,
                              double* flux_out, double* diag, void* workspace, size_t workspace_bytes,
                              void* stream) {
  return sweep_common(0, g, c_in, e_in, c_out, e_out, u_face, dt, state, theta, flux_out, diag, workspace,
                      workspace_bytes, stream);
}
vof_status vof_advect_sweep_y(const vof_grid* g, const double* c_in, const double* e_in, double* c_out,
                              double* e_out, const double* v_face, double dt, uint8_t* state, double* theta,
                              double* flux_out, double* diag, void* workspace, size_t workspace_bytes,
                              void* stream) {
  return sweep_common(1, g, c_in, e_in, c_out, e_out, v_face, dt, state, theta, flux_out, diag, workspace,
                      workspace_bytes, stream);
}
vof_status vof_advect_sweep_z(const vof_grid* g, const double* c_in, const double* e_in, double* c_out,
                              double* e_out, const double* w_face, double dt, uint8_t* state, double* theta,
                              double* flux_out, double* diag, void* workspace, size_t workspace_bytes,
                              void* stream) {
  return sweep_common(2, g, c_in, e_in, c_out, e_out, w_face, dt, state, theta, flux_out, diag, workspace,
                      workspace_bytes, stream);
}

vof_status energy_advect_consistent(const vof_grid* g, int axis, const double* c_before, const double* c_after,
                                    const double* e_in, double* e_out, const double* flux_F, const double* u_face,
                                    double dt, uint8_t* state, double* theta, void* stream) {
  if (!grid_ok(g) || axis < 0 || axis > 2 || !c_before || !c_after || !e_in || !e_out || !flux_F || !u_face)
    return VOF_EINVAL;
  if (state && !theta) return VOF_EINVAL;
  if (!(dt >= 0.0)) return VOF_EINVAL;
  size_t B = cells(g) * 8;
  if (overlap(e_in, B, e_out, B) || overlap(c_before, B, e_out, B) || overlap(c_after, B, e_out, B)) return VOF_EINVAL;
  return cuda_status(launch_energy(axis, to_dev(g, dt), c_before, c_after, e_in, e_out, flux_F, u_face, state, theta,
                                   (cudaStream_t)stream));
}

size_t vof_shift_workspace_bytes(const vof_grid* g) {
  if (!grid_ok(g)) return 0;
  return shift_scratch_bytes(to_dev(g, 0.0));
}

vof_status vof_phase_change_shift(const vof_grid* g, const double* c_in, const double* e_in, double* c_out,
                                  double* e_out, const double* dd, double dd_uniform, uint8_t* state, double* diag,
                                  void* workspace, size_t workspace_bytes, void* stream) {
  if (!grid_ok(g) || !c_in || !e_in || !c_out || !e_out || !workspace) return VOF_EINVAL;
  if (((uintptr_t)workspace & 255) != 0) return VOF_EINVAL;
  const GridDev d = to_dev(g, 0.0);
  const size_t need = shift_scratch_bytes(d);
  if (workspace_bytes < need) return VOF_EINVAL;
  size_t B = cells(g) * 8;
  // either fully in place (c_out == c_in and e_out == e_in) or no overlap
  const bool inplace = c_out == c_in && e_out == e_in;
  if (!inplace && (overlap(c_in, B, c_out, B) || overlap(e_in, B, e_out, B) || overlap(c_in, B, e_out, B) ||
                   overlap(e_in, B, c_out, B)))
    return VOF_EINVAL;
  if (overlap(c_out, B, e_out, B) || overlap(c_in, B, e_in, B)) return VOF_EINVAL;
  if (overlap(workspace, need, c_in, B) || overlap(workspace, need, c_out, B) || overlap(workspace, need, e_in, B) ||
      overlap(workspace, need, e_out, B) || (dd && overlap(workspace, need, dd, B)) ||
      (state && overlap(workspace, need, state, cells(g))) || (diag && overlap(workspace, need, diag, 5 * 8)))
    return VOF_EINVAL;
  // diag = {sum dc, clamped, sum de, sum c_out, sum e_out}
  static const signed char kMap[kNSums] = {3, 4, -1, 0, 1, 2};
  const SumOut so = sums_to_diag(diag, kMap);
  return cuda_status(launch_shift(d, c_in, e_in, c_out, e_out, dd, dd_uniform, state, carve_shift_scratch(d, workspace),
                                  so, so, (cudaStream_t)stream));
}

// workspace layout: theta | sum rows (kNSums doubles per tile) |
// reduction scratch | work counts (12 ints) and, 128 bytes in, the step's
// counters (kStepCounters ints, cleared by the tile pass) | tiles | scratch
// fields c, e | the mixed cells' fluxes | ghost fluxes | planes | lists |
// active tiles | clipped volumes.  The step's last kernel sums every
// active tile's cells, the tile pass the quiet ones', so one fixed-order
// reduction of the rows gives the sums.  The size is at least that of the
// stand-alone sweeps' and shift's scratch behind the first five regions and a
// byte per cell: a program's one buffer of vof_step_workspace_bytes() has always
// served those calls too.
struct StepLayout {
  size_t off_th, off_rows, off_red, off_stats, off_tiles, off_sc, off_se, off_fl, off_fr, off_gf, off_plane,
      off_l0, off_l1, off_tlist, off_clip, total;
  int ntiles;
};

static StepLayout step_layout(const vof_grid* g) {
  StepLayout L;
  GridDev d = to_dev(g, 0.0);
  const size_t N = cells(g);
  size_t lines = 0;
  for (int a = 0; a < 3; ++a) lines = N / (size_t)d.n[a] > lines ? N / (size_t)d.n[a] : lines;
  L.ntiles = tile_total(d);
  const size_t T = (size_t)L.ntiles;
  size_t o = 0;
  auto take = [&](size_t b) { const size_t at = o; o += align256(b); return at; };
  L.off_th = take(N * 8);
  L.off_rows = take(T * kNSums * 8);
  L.off_red = take(reduce_scratch_bytes());
  L.off_stats = take(256);
  L.off_tiles = take(tile_scratch_bytes(d));
  const size_t base = o;
  L.off_sc = take(N * 8);
  L.off_se = take(N * 8);
  L.off_fl = take(N * 8);
  L.off_fr = take(N * 8);
  L.off_gf = take(2 * lines * 8);
  L.off_plane = take(N * 32);
  L.off_l0 = take(N * 4);
  L.off_l1 = take(N * 4);
  L.off_tlist = take(T * 4);
  L.off_clip = take(12 * T * 8);
  const size_t sw = sweep_scratch_bytes(d), sh = shift_scratch_bytes(d);
  const size_t other = base + align256(N) + align256(sw > sh ? sw : sh);
  L.total = o > other ? o : other;
  return L;
}

size_t vof_step_workspace_bytes(const vof_grid* g) {
  if (!grid_ok(g)) return 0;
  return step_layout(g).total;
}

}  // extern "C"

namespace vofgb {

bool step_box(const vof_grid* g, double* c, double* e, const double* u, const double* v, const double* w,
              double dt, const double* dd, double dd_uniform, double* sums, char* ws, StepBox* out) {
  if (!grid_ok(g) || !c || !e || !u || !v || !w || !(dt >= 0.0) || !ws) return false;
  const StepLayout L = step_layout(g);
  const GridDev d = to_dev(g, dt);
  StepBox& B = *out;
  B.cells = cells(g);
  StepArgs& A = B.args;
  A.g = d;
  A.c = c;
  A.e = e;
  A.s_c = reinterpret_cast<double*>(ws + L.off_sc);
  A.s_e = reinterpret_cast<double*>(ws + L.off_se);
  A.uf[0] = u; A.uf[1] = v; A.uf[2] = w;
  A.theta = reinterpret_cast<double*>(ws + L.off_th);
  A.fl = reinterpret_cast<double*>(ws + L.off_fl);
  A.fr = reinterpret_cast<double*>(ws + L.off_fr);
  A.gf = reinterpret_cast<double*>(ws + L.off_gf);
  A.plane = reinterpret_cast<double*>(ws + L.off_plane);
  A.list[0] = reinterpret_cast<uint32_t*>(ws + L.off_l0);
  A.list[1] = reinterpret_cast<uint32_t*>(ws + L.off_l1);
  A.tlist = reinterpret_cast<uint32_t*>(ws + L.off_tlist);
  A.clip = reinterpret_cast<double*>(ws + L.off_clip);
  A.rows = reinterpret_cast<double*>(ws + L.off_rows);
  A.ts = carve_tile_scratch(d, ws + L.off_tiles);
  tile_counts(d, A.nt);
  A.stats = reinterpret_cast<int*>(ws + L.off_stats);
  A.cnt = reinterpret_cast<int*>(ws + L.off_stats + 128);
  A.status = device_status_ptr();
  A.dd = dd;
  A.dd_uniform = dd_uniform;
  A.pairs = reinterpret_cast<uint2*>(A.theta);
  A.pair_cap = (unsigned)B.cells;
  A.chain = 0;
  B.grid_tiles = dim3((unsigned)((A.nt[0] + 3) / 4), (unsigned)A.nt[1], (unsigned)A.nt[2]);
  B.red = ReduceBox{A.rows, L.ntiles, sums, reinterpret_cast<double*>(ws + L.off_red)};
  return true;
}

}  // namespace vofgb

extern "C" {

vof_status vof_step(const vof_grid* g, double* c, double* e, const double* u, const double* v, const double* w,
                    double dt, long step_index, const double* dd, double dd_uniform, double* sums, void* workspace,
                    size_t workspace_bytes, void* stream) {
  if (!grid_ok(g) || !c || !e || !u || !v || !w || !workspace) return VOF_EINVAL;
  if (!(dt >= 0.0) || step_index < 0) return VOF_EINVAL;
  if (((uintptr_t)workspace & 255) != 0) return VOF_EINVAL;
  StepLayout L = step_layout(g);
  if (workspace_bytes < L.total) return VOF_EINVAL;
  size_t N = cells(g), B = N * 8;
  if (overlap(c, B, e, B) || overlap(c, B, workspace, L.total) || overlap(e, B, workspace, L.total))
    return VOF_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  StepBox bx;
  if (!step_box(g, c, e, u, v, w, dt, dd, dd_uniform, sums, static_cast<char*>(workspace), &bx)) return VOF_EINVAL;
  const StepArgs& A = bx.args;
  cudaError_t err = launch_tiles(A, st);
  const int odd = (int)(step_index % 2);
  for (int s = 0; s < 3 && err == cudaSuccess; ++s) err = launch_stage(A, odd ? 2 - s : s, s, st);
  if (err == cudaSuccess) err = launch_shift_step(A, odd, st);
  // sums[0..1] = sum c, sum e; sums[2] = clip; sums[3..5] = shift diagnostics
  if (err == cudaSuccess && sums)
    err = launch_reduce_fused(ReduceJob{bx.red.rows, bx.red.nblocks, kNSums, 0, kNSums, sums}, bx.red.scratch,
                              A.cnt + (kStepCounters - 1), st);
  return cuda_status(err);
}

vof_status vof_step_work_counts(const vof_grid* g, const void* workspace, int* counts, void* stream) {
  if (!grid_ok(g) || !workspace || !counts) return VOF_EINVAL;
  const StepLayout L = step_layout(g);
  const char* ws = static_cast<const char*>(workspace);
  cudaStream_t st = (cudaStream_t)stream;
  cudaError_t err = cudaMemcpyAsync(counts, ws + L.off_stats, VOF_NCOUNTS * sizeof(int), cudaMemcpyDeviceToHost, st);
  if (err == cudaSuccess) err = cudaStreamSynchronize(st);
  return cuda_status(err);
}

size_t vof_mass_transfer_workspace_bytes(const vof_grid* g) {
  if (!grid_ok(g)) return 0;
  return mdot_scratch_bytes(cells(g));
}

vof_status vof_mass_transfer(const vof_grid* g, const double* c, const double* e, double k_l, double k_g,
                             double h_fg, double* mdot, double* d_gamma, double* grad_n, double dd_per_mdot,
                             double* dd, void* workspace, size_t workspace_bytes, void* stream) {
  if (!grid_ok(g) || !c || !e || !mdot || !workspace) return VOF_EINVAL;
  if (!(h_fg > 0.0) || !(k_l >= 0.0) || !(k_g >= 0.0) || !(dd_per_mdot == dd_per_mdot)) return VOF_EINVAL;
  if (((uintptr_t)workspace & 255) != 0) return VOF_EINVAL;
  const size_t N = cells(g), B = N * 8;
  const size_t need = mdot_scratch_bytes(N);
  if (workspace_bytes < need) return VOF_EINVAL;
  const void* outs[4] = {mdot, d_gamma, grad_n, dd};
  for (int a = 0; a < 4; ++a) {
    if (!outs[a]) continue;
    if (overlap(outs[a], B, c, B) || overlap(outs[a], B, e, B) || overlap(outs[a], B, workspace, need))
      return VOF_EINVAL;
    for (int b = a + 1; b < 4; ++b)
      if (overlap(outs[a], B, outs[b], B)) return VOF_EINVAL;
  }
  if (overlap(workspace, need, c, B) || overlap(workspace, need, e, B)) return VOF_EINVAL;
  return cuda_status(launch_mass_transfer(to_dev(g, 0.0), g->h, c, e, k_l, k_g, h_fg, dd_per_mdot, mdot, d_gamma,
                                          grad_n, dd, workspace, (cudaStream_t)stream));
}

vof_status vof_mass_transfer_work_counts(const vof_grid* g, const void* workspace, int* counts, void* stream) {
  if (!grid_ok(g) || !workspace || !counts) return VOF_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  cudaError_t err = cudaMemcpyAsync(counts, mdot_counters(to_dev(g, 0.0), const_cast<void*>(workspace)),
                                    2 * sizeof(int), cudaMemcpyDeviceToHost, st);
  if (err == cudaSuccess) err = cudaStreamSynchronize(st);
  return cuda_status(err);
}

size_t vof_velocity_extension_workspace_bytes(const vof_grid* g) {
  if (!grid_ok(g)) return 0;
  return ext_scratch_bytes(cells(g));
}

vof_status vof_velocity_extension(const vof_grid* g, const double* c, const double* mdot, double rho_l,
                                  double rho_g, double dt, double tol, int max_iter, double* u, double* v,
                                  double* w, double* ut, double* vt, double* wt, int* iterations,
                                  double* residual, void* workspace, size_t workspace_bytes, void* stream) {
  if (!grid_ok(g) || !c || !mdot || !workspace) return VOF_EINVAL;
  if (!(rho_l > 0.0) || !(rho_g > 0.0) || !(dt >= 0.0) || !(tol > 0.0) || max_iter < 1) return VOF_EINVAL;
  const bool add = u || v || w, put = ut || vt || wt;
  if ((add && !(u && v && w)) || (put && !(ut && vt && wt)) || (!add && !put)) return VOF_EINVAL;
  if (((uintptr_t)workspace & 255) != 0) return VOF_EINVAL;
  const size_t N = cells(g), B = N * 8;
  const size_t need = ext_scratch_bytes(N);
  if (workspace_bytes < need) return VOF_EINVAL;
  const void* outs[6] = {u, v, w, ut, vt, wt};
  for (int a = 0; a < 6; ++a) {
    if (!outs[a]) continue;
    const size_t fa = face_count(g, a % 3) * 8;
    if (overlap(outs[a], fa, c, B) || overlap(outs[a], fa, mdot, B) || overlap(outs[a], fa, workspace, need))
      return VOF_EINVAL;
    for (int b = a + 1; b < 6; ++b)
      if (outs[b] && overlap(outs[a], fa, outs[b], face_count(g, b % 3) * 8)) return VOF_EINVAL;
  }
  if (overlap(workspace, need, c, B) || overlap(workspace, need, mdot, B)) return VOF_EINVAL;
  int it = 0, st = 0;
  double res = 0.0;
  cudaError_t err = launch_velocity_extension(to_dev(g, 0.0), g->h, c, mdot, rho_l, rho_g, dt, tol, max_iter, u, v,
                                              w, ut, vt, wt, workspace, (cudaStream_t)stream, &it, &res, &st);
  if (err != cudaSuccess) return cuda_status(err);
  if (iterations) *iterations = it;
  if (residual) *residual = res;
  return st ? VOF_ESOLVE : VOF_OK;
}

size_t vof_heat_diffusion_workspace_bytes(const vof_grid* g) {
  if (!grid_ok(g)) return 0;
  return dif_scratch_bytes(cells(g));
}

vof_status vof_heat_diffusion(const vof_grid* g, const double* c, double* e, double k_l, double k_g, double dt,
                              double tol, int max_iter, int heat_capacity, const double* wall_T, int* iterations,
                              double* change, void* workspace, size_t workspace_bytes, void* stream) {
  if (!grid_ok(g) || !c || !e || !workspace) return VOF_EINVAL;
  if (!(k_l >= 0.0) || !(k_g >= 0.0) || !(dt > 0.0) || !(tol > 0.0) || max_iter < 1) return VOF_EINVAL;
  if (heat_capacity != VOF_CP_PHASE && heat_capacity != VOF_CP_MIXTURE) return VOF_EINVAL;
  if (wall_T) {
    for (int f = 0; f < 6; ++f) {
      const double Tw = wall_T[f];
      if (Tw != Tw) continue;                                   // NaN: no wall temperature on this face
      if (g->bc[f / 2] != 1 || !(Tw > -1e300 && Tw < 1e300)) return VOF_EINVAL;  // finite, zero-gradient axis
    }
  }
  if (((uintptr_t)workspace & 255) != 0) return VOF_EINVAL;
  const size_t N = cells(g), B = N * 8;
  const size_t need = dif_scratch_bytes(N);
  if (workspace_bytes < need) return VOF_EINVAL;
  if (overlap(c, B, e, B) || overlap(workspace, need, c, B) || overlap(workspace, need, e, B)) return VOF_EINVAL;
  int it = 0, st = 0;
  double ch = 0.0;
  cudaError_t err = launch_heat_diffusion(to_dev(g, 0.0), g->h, c, e, k_l, k_g, dt, tol, max_iter,
                                          heat_capacity == VOF_CP_PHASE ? 1 : 0, wall_T, workspace,
                                          (cudaStream_t)stream, &it, &ch, &st);
  if (err != cudaSuccess) return cuda_status(err);
  if (iterations) *iterations = it;
  if (change) *change = ch;
  return st ? VOF_ESOLVE : VOF_OK;
}

vof_status vof_get_device_status(void) {
  int* p = device_status_ptr();
  if (!p) return VOF_ECUDA;
  int h = 0;
  cudaError_t e = cudaMemcpy(&h, p, sizeof(int), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_status(e);
  int z = 0;
  e = cudaMemcpy(p, &z, sizeof(int), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return cuda_status(e);
  if (h & DEV_WAIT) return VOF_EWAIT;
  return (h & DEV_CFL) ? VOF_ECFL : VOF_OK;
}

const char* vof_status_string(int status) {
  switch (status) {
    case VOF_OK: return "ok";
    case VOF_EINVAL: return "invalid argument";
    case VOF_ECUDA: return "CUDA error";
    case VOF_ECFL: return "face CFL number above 1";
    case VOF_ESOLVE: return "iterative solve not converged (or no free-flow face for the velocity extension)";
    case VOF_EWAIT: return "a bounded device wait gave up (tensor-core completion not seen in time)";
    default: return "unknown status";
  }
}

int vof_last_cuda_error(void) { return t_last_cuda; }

}  // extern "C"
