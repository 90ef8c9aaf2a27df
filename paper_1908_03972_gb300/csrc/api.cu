// api.cu -- C interface of libpmgfr and the solver orchestration: FAS
// V-cycle (Section 3), pseudo-transient continuation with SER (Section 2.4),
// ESDIRK3 physical steps.  Every arithmetic step runs in the kernels of
// k_residual.cu, k_blocks.cu and k_misc.cu; the host only sequences launches,
// keeps the pseudo-time schedule and reads one norm per V-cycle.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <string>
#include <array>
#include <utility>

#include "pmg_internal.h"

using namespace pmg;

struct pmg_ctx {
  Ctx c;
};

static thread_local std::string g_err;

static pmg_status fail(pmg_status st, const std::string& msg) {
  g_err = msg;
  return st;
}

#define PMG_CK(call)                                                                   \
  do {                                                                                 \
    cudaError_t e_ = (call);                                                           \
    if (e_ != cudaSuccess) return fail(PMG_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

#define PMG_CK_LAUNCH()                                                                \
  do {                                                                                 \
    cudaError_t e_ = cudaGetLastError();                                               \
    if (e_ != cudaSuccess) return fail(PMG_ECUDA, std::string("kernel launch: ") + cudaGetErrorString(e_)); \
  } while (0)

template <class T>
static cudaError_t dalloc(T** p, size_t count) {
  return cudaMalloc((void**)p, count * sizeof(T) > 0 ? count * sizeof(T) : 8);
}

// ESDIRK schemes of Section 2.4 (first stage explicit, stiffly accurate,
// L-stable), with published coefficients:
//  order 2: three stages (Kennedy & Carpenter 2016), g = 1 - 1/sqrt 2,
//           b1 = b2 = 1/(2 sqrt 2), c = (0, 2g, 1);
//  order 3: four stages, the implicit tableau of ARK3(2)4L[2]SA;
//  order 4: six stages, the implicit tableau of ARK4(3)6L[2]SA (g = 1/4).
static void esdirk_table(Ctx& c, int order) {
  memset(c.A, 0, sizeof(c.A));
  memset(c.b, 0, sizeof(c.b));
  memset(c.c, 0, sizeof(c.c));
  if (order == 2) {
    const double g = 1.0 - 1.0 / std::sqrt(2.0), w = 1.0 / (2.0 * std::sqrt(2.0));
    c.A[1][0] = g; c.A[1][1] = g;
    c.b[0] = w; c.b[1] = w; c.b[2] = g;
    for (int j = 0; j < 3; ++j) c.A[2][j] = c.b[j];
    c.c[1] = 2 * g; c.c[2] = 1.0;
    c.stages = 3;
    return;
  }
  if (order == 4) {
    const double g = 0.25;
    for (int i = 1; i < 6; ++i) c.A[i][i] = g;
    c.A[1][0] = g;
    c.A[2][0] = 8611.0 / 62500.0;
    c.A[2][1] = -1743.0 / 31250.0;
    c.A[3][0] = 5012029.0 / 34652500.0;
    c.A[3][1] = -654441.0 / 2922500.0;
    c.A[3][2] = 174375.0 / 388108.0;
    c.A[4][0] = 15267082809.0 / 155376265600.0;
    c.A[4][1] = -71443401.0 / 120774400.0;
    c.A[4][2] = 730878875.0 / 902184768.0;
    c.A[4][3] = 2285395.0 / 8070912.0;
    const double b[6] = {82889.0 / 524892.0, 0.0, 15625.0 / 83664.0, 69875.0 / 102672.0, -2260.0 / 8211.0, g};
    const double cc[6] = {0.0, 0.5, 83.0 / 250.0, 31.0 / 50.0, 17.0 / 20.0, 1.0};
    for (int j = 0; j < 6; ++j) { c.b[j] = b[j]; c.A[5][j] = b[j]; c.c[j] = cc[j]; }
    c.stages = 6;
    return;
  }
  const double g = 1767732205903.0 / 4055673282236.0;
  c.A[1][0] = g; c.A[1][1] = g;
  c.A[2][0] = 2746238789719.0 / 10658868560708.0;
  c.A[2][1] = -640167445237.0 / 6845629431997.0;
  c.A[2][2] = g;
  c.b[0] = 1471266399579.0 / 7840856788654.0;
  c.b[1] = -4482444167858.0 / 7529755066697.0;
  c.b[2] = 11266239266428.0 / 11593286722821.0;
  c.b[3] = g;
  for (int j = 0; j < 4; ++j) c.A[3][j] = c.b[j];
  c.c[0] = 0.0; c.c[1] = 2 * g; c.c[2] = 3.0 / 5.0; c.c[3] = 1.0;
  c.stages = 4;
}

static void free_level(LevelDev& L) {
  double** ptrs[] = {&L.q,     &L.q2, &L.qb, &L.S,  &L.F,  &L.Pd, &L.met,
                     &L.Fcom,  &L.Dfull, &L.rs, &L.cs, &L.Gb, &L.Qj, &L.fJinv, &L.Cgauge};
  for (double** p : ptrs) { if (*p) cudaFree(*p); *p = nullptr; }
  int** iptrs[] = {&L.d_toff, &L.d_tlayer, &L.d_telems, &L.d_tlnbr};
  for (int** p : iptrs) { if (*p) cudaFree(*p); *p = nullptr; }
  L.face = nullptr;   // face, metW and faceW lie in met's allocation
  L.metW = L.faceW = nullptr;
  if (L.Dinv) cudaFree(L.Dinv);
  L.Dinv = nullptr;
}

static void nk_free(Ctx& c) {
  double** ptrs[] = {&c.nk_q, &c.nk_F, &c.nk_src, &c.nk_w, &c.nk_t, &c.nk_x,
                     &c.nk_V, &c.nk_Z, &c.nk_part, &c.nk_dots, &c.nk_coef};
  for (double** p : ptrs) { if (*p) cudaFree(*p); *p = nullptr; }
  if (c.h_nk) cudaFreeHost(c.h_nk);
  c.h_nk = nullptr;
  c.nk_m = 0;
}

// Multi-sweep tiles of a coarse level (k_tile.cu): build and upload them, or
// drop them (depth 0).  Returns PMG_EINVAL when the tile does not fit (512
// threads, 227 KB of shared memory per CTA).
static pmg_status set_level_tiles(Ctx& c, LevelDev& L, int core, int depth) {
  int** iptrs[] = {&L.d_toff, &L.d_tlayer, &L.d_telems, &L.d_tlnbr};
  for (int** p : iptrs) { if (*p) cudaFree(*p); *p = nullptr; }
  L.tiled = false;
  L.n_tiles = L.tile_M = L.tile_depth = 0;
  L.tile_core = 0;
  if (depth <= 0) return PMG_OK;
  TileSet ts;
  try {
    ts = build_tiles(c.mesh, core, depth);
  } catch (const std::exception& ex) {
    return fail(PMG_EINVAL, ex.what());
  }
  const size_t bytes = tile_smem_bytes(L.P, c.cfg.block_prec, ts.max_elems);
  const int threads = ts.max_elems * tile_face_points(L.P);
  if (!(bytes > 0 && bytes <= (size_t)227 * 1024 && threads <= 512))
    return fail(PMG_EINVAL, "tile of " + std::to_string(ts.max_elems) + " elements does not fit a CTA");
  if (dalloc(&L.d_toff, ts.off.size()) || dalloc(&L.d_tlayer, ts.layer_end.size()) ||
      dalloc(&L.d_telems, ts.elems.size()) || dalloc(&L.d_tlnbr, ts.lnbr.size()))
    return fail(PMG_ENOMEM, "device allocation failed for tile data");
  PMG_CK(cudaMemcpy(L.d_toff, ts.off.data(), ts.off.size() * sizeof(int), cudaMemcpyHostToDevice));
  PMG_CK(cudaMemcpy(L.d_tlayer, ts.layer_end.data(), ts.layer_end.size() * sizeof(int), cudaMemcpyHostToDevice));
  PMG_CK(cudaMemcpy(L.d_telems, ts.elems.data(), ts.elems.size() * sizeof(int), cudaMemcpyHostToDevice));
  PMG_CK(cudaMemcpy(L.d_tlnbr, ts.lnbr.data(), ts.lnbr.size() * sizeof(int), cudaMemcpyHostToDevice));
  PMG_CK(prepare_tile_kernel(L.P, c.cfg.block_prec, bytes));
  L.tiled = true;
  L.n_tiles = ts.n_tiles;
  L.tile_M = ts.max_elems;
  L.tile_depth = depth;
  L.tile_core = core;
  return PMG_OK;
}

extern "C" {

const char* pmg_last_error(void) { return g_err.c_str(); }

pmg_status pmg_create(const pmg_config* cfg, void* stream, pmg_ctx** out) {
  if (!cfg || !out) return fail(PMG_EINVAL, "null argument");
  if (cfg->n_levels < 1 || cfg->n_levels > kMaxLevels) return fail(PMG_EINVAL, "n_levels must be in 1..8");
  for (int l = 0; l < cfg->n_levels; ++l) {
    if (cfg->P[l] < 0 || cfg->P[l] > kMaxP) return fail(PMG_EINVAL, "P must be in 0..5");
    if (l > 0 && cfg->P[l] >= cfg->P[l - 1]) return fail(PMG_EINVAL, "P levels must decrease");
    if (cfg->n_smooth[l] < 1) return fail(PMG_EINVAL, "smoothing counts must be >= 1");
  }
  if (cfg->block_prec != PMG_PREC_FP64 && cfg->block_prec != PMG_PREC_FP32 && cfg->block_prec != PMG_PREC_BF16R)
    return fail(PMG_EINVAL, "unknown block precision");
  if (cfg->flux_prec != PMG_FLUX_FP64 && cfg->flux_prec != PMG_FLUX_DW_SMOOTH && cfg->flux_prec != PMG_FLUX_DW)
    return fail(PMG_EINVAL, "unknown flux precision");
  if (!(cfg->gamma > 1.0)) return fail(PMG_EINVAL, "gamma must exceed 1");
  if (cfg->esdirk_order != 0 && (cfg->esdirk_order < 2 || cfg->esdirk_order > 4))
    return fail(PMG_EINVAL, "esdirk_order must be 2, 3 or 4 (0 means 3)");
  if (cfg->cfl_mode && !(cfg->cfl_init > 0.0 && cfg->cfl_max >= cfg->cfl_init))
    return fail(PMG_EINVAL, "cfl_mode needs 0 < cfl_init <= cfl_max");
  if (!(cfg->mu >= 0.0) || !std::isfinite(cfg->mu)) return fail(PMG_EINVAL, "mu must be finite and >= 0");
  if (cfg->mu > 0.0 && !(cfg->Pr > 0.0 && std::isfinite(cfg->Pr)))
    return fail(PMG_EINVAL, "Pr must be finite and > 0 when mu > 0");
  for (int v = 0; v < 4; ++v)
    if (!std::isfinite(cfg->res_scale[v])) return fail(PMG_EINVAL, "res_scale must be finite");
  if (!std::isfinite(cfg->copy_wait_s)) return fail(PMG_EINVAL, "copy_wait_s must be finite");
  if (cfg->device_loop != 0 && cfg->device_loop != 1) return fail(PMG_EINVAL, "device_loop must be 0 or 1");
  if (cfg->max_pseudo < 0) return fail(PMG_EINVAL, "max_pseudo must be >= 0");
  if (cfg->refresh_every < 1) return fail(PMG_EINVAL, "refresh_every must be >= 1");
  if (cfg->dim != 0 && cfg->dim != 2 && cfg->dim != 3) return fail(PMG_EINVAL, "dim must be 2 or 3 (0 means 2)");
  if (cfg->dim == 3) {
    if (cfg->cfl_mode) return fail(PMG_EINVAL, "hexahedral runs set dtau directly (cfl_mode = 0)");
    for (int l = 0; l < cfg->n_levels; ++l)
      if (cfg->P[l] > 3) return fail(PMG_EINVAL, "hexahedral levels take P <= 3");
    for (int v = 0; v < 5; ++v)
      if (!std::isfinite(cfg->res_scale3[v])) return fail(PMG_EINVAL, "res_scale3 must be finite");
  }
  int dev;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return fail(PMG_ECUDA, std::string("no CUDA device: ") + cudaGetErrorString(e));
  pmg_ctx* h = new pmg_ctx();
  Ctx& c = h->c;
  c.cfg = *cfg;
  c.device = dev;
  c.dim = cfg->dim == 3 ? 3 : 2;
  c.nv = c.dim + 2;
  c.nfc = 2 * c.dim;
  if (c.dim == 3) c.cfg.flux_prec = PMG_FLUX_FP64;   // the hexahedral residual is binary64 throughout
  if (stream) {
    c.stream = (cudaStream_t)stream;
  } else {
    e = cudaStreamCreateWithFlags(&c.stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) { delete h; return fail(PMG_ECUDA, cudaGetErrorString(e)); }
    c.own_stream = true;
  }
  c.ph.gamma = cfg->gamma;
  c.ph.gm1 = cfg->gamma - 1.0;
  c.ph.Cp = cfg->gamma / (cfg->gamma - 1.0);
  c.ph.eps_min = cfg->cutoff ? cfg->kappa * cfg->Ma_inf : 0.0;
  c.ph.p_ref = cfg->p_gauge;
  c.ph.inv_gamma = 1.0 / cfg->gamma;
  c.ph.inv_gm1 = 1.0 / (cfg->gamma - 1.0);
  c.ph.inv_Cp = (cfg->gamma - 1.0) / cfg->gamma;
  c.ph.mu = cfg->mu;
  c.ph.kT = cfg->mu > 0.0 ? cfg->mu * c.ph.Cp / cfg->Pr : 0.0;
  for (int v = 0; v < 5; ++v) { c.ph.nw[v] = 1.0; c.ph.qinf[v] = 0.0; }
  if (c.dim == 3) {
    for (int v = 0; v < 5; ++v) c.ph.nw[v] = cfg->res_scale3[v] > 0.0 ? 1.0 / cfg->res_scale3[v] : 1.0;
    for (int v = 0; v < 5; ++v) c.ph.qinf[v] = cfg->q_inf3[v];
  } else {
    for (int v = 0; v < 4; ++v) c.ph.nw[v] = cfg->res_scale[v] > 0.0 ? 1.0 / cfg->res_scale[v] : 1.0;
    for (int v = 0; v < 4; ++v) c.ph.qinf[v] = cfg->q_inf[v];
  }
  c.ph.wait_ns = cfg->copy_wait_s == 0.0 ? 1e9 : cfg->copy_wait_s < 0.0 ? -1.0 : std::min(cfg->copy_wait_s, 60.0) * 1e9;
  c.phw = make_physw(c.ph);
  esdirk_table(c, cfg->esdirk_order == 0 ? 3 : cfg->esdirk_order);
  const size_t nhist = 2 * ((size_t)cfg->max_pseudo + 1);
  if (dalloc(&c.d_scal, 4) != cudaSuccess || dalloc(&c.d_flag, 4) != cudaSuccess ||
      dalloc(&c.d_dtau, 1) != cudaSuccess || cudaMallocHost((void**)&c.h_scal, 8 * sizeof(double)) != cudaSuccess ||
      cudaMallocHost((void**)&c.h_dtau, sizeof(double)) != cudaSuccess ||
      cudaMalloc((void**)&c.d_loop, sizeof(LoopState)) != cudaSuccess ||
      cudaMallocHost((void**)&c.h_loop, sizeof(LoopState)) != cudaSuccess || dalloc(&c.d_hist, nhist) != cudaSuccess ||
      cudaMallocHost((void**)&c.h_hist, nhist * sizeof(double)) != cudaSuccess) {
    pmg_destroy(h);
    return fail(PMG_ENOMEM, "device allocation failed");
  }
  // d_scal[1]: set by kernels whose bounded wait for a bulk copy gave up;
  // d_flag: 1 + the highest singular element of the last rebuild.  Both start
  // at zero (cudaMalloc may hand back memory another context left behind).
  if (cudaMemset(c.d_scal, 0, 4 * sizeof(double)) != cudaSuccess ||
      cudaMemset(c.d_flag, 0, 4 * sizeof(int)) != cudaSuccess) {
    pmg_destroy(h);
    return fail(PMG_ECUDA, "device memset failed");
  }
  *out = h;
  return PMG_OK;
}

void pmg_destroy(pmg_ctx* h) {
  if (!h) return;
  Ctx& c = h->c;
  cudaStreamSynchronize(c.stream);
  nk_free(c);
  for (int g = 0; g < 2; ++g)
    if (c.graph[g]) cudaGraphExecDestroy(c.graph[g]);
  if (c.loop_exec) cudaGraphExecDestroy(c.loop_exec);
  if (c.d_loop) cudaFree(c.d_loop);
  if (c.h_loop) cudaFreeHost(c.h_loop);
  if (c.d_hist) cudaFree(c.d_hist);
  if (c.h_hist) cudaFreeHost(c.h_hist);
  for (int l = 0; l < kMaxLevels; ++l) free_level(c.lev[l]);
  double** ptrs[] = {&c.src, &c.qn, &c.qcn, &c.d_partial, &c.d_scal, &c.d_tmp0, &c.d_tmp1, &c.d_dtau, &c.d_dx};
  for (double** p : ptrs) { if (*p) cudaFree(*p); *p = nullptr; }
  for (int j = 0; j < 6; ++j) if (c.Rst[j]) cudaFree(c.Rst[j]);
  if (c.d_faces) cudaFree(c.d_faces);
  if (c.d_flag) cudaFree(c.d_flag);
  if (c.h_scal) cudaFreeHost(c.h_scal);
  if (c.h_dtau) cudaFreeHost(c.h_dtau);
  for (auto& e : c.prof.ev) cudaEventDestroy(e);
  if (c.own_stream) cudaStreamDestroy(c.stream);
  delete h;
}

// Gauge storage on a curved mesh: on a level with P below the geometry order
// the discrete metric identity holds only to the interpolation error, and the
// gauge momentum flux (p - p_gauge) leaves out p_gauge times that residual.
// Cgauge = R(uniform state, absolute pressure) - R(the same state, gauge
// storage) is that constant, computed once: the convective parts of the two
// evaluations are the same operations on the same numbers.  The state moves
// with the free stream (or u = 1) so that the preconditioned flux has eps > 0;
// far-field faces see the same state.
static pmg_status compute_gauge_constant(Ctx& c, int l) {
  LevelDev& L = c.lev[l];
  if (dalloc(&L.Cgauge, L.tot)) return fail(PMG_ENOMEM, "device allocation failed for level data");
  const size_t plane = (size_t)c.E * L.N;
  const int T_slot = c.nv - 1;
  double qu[5] = {c.ph.p_ref, 1.0, 0.0, 0.0, 0.0};
  qu[T_slot] = c.ph.p_ref;   // rho = 1
  if (c.ph.qinf[0] > 0.0 && c.ph.qinf[T_slot] > 0.0)
    for (int v = 0; v < c.nv; ++v) qu[v] = c.ph.qinf[v];
  std::vector<double> h(L.tot);
  for (int v = 0; v < c.nv; ++v) std::fill(h.begin() + v * plane, h.begin() + (v + 1) * plane, qu[v]);
  const Phys keep = c.ph;
  const PhysW keepw = c.phw;
  for (int v = 0; v < c.nv; ++v) c.ph.qinf[v] = qu[v];
  // gauge form: stored p - p_gauge
  PMG_CK(cudaMemcpy(c.d_tmp0, h.data(), L.tot * 8, cudaMemcpyHostToDevice));
  launch_shift_pressure(plane, -keep.p_ref, c.d_tmp0, c.stream);
  c.phw = make_physw(c.ph);
  launch_face_flux(c, L, c.d_tmp0, c.stream);
  launch_volume(c, L, l, c.d_tmp0, c.d_tmp1, RES_PURE, 0.0, nullptr, nullptr, nullptr, nullptr, nullptr, c.stream);
  // absolute form
  PMG_CK(cudaMemcpyAsync(c.d_tmp0, h.data(), L.tot * 8, cudaMemcpyHostToDevice, c.stream));
  c.ph.p_ref = 0.0;
  c.phw = make_physw(c.ph);
  launch_face_flux(c, L, c.d_tmp0, c.stream);
  launch_volume(c, L, l, c.d_tmp0, L.Cgauge, RES_PURE, 0.0, nullptr, nullptr, nullptr, nullptr, nullptr, c.stream);
  Scale5 one;
  for (double& x : one.s) x = 1.0;
  launch_plane_combine(L.Cgauge, L.Cgauge, 1.0, c.d_tmp1, -1.0, one, nullptr, 0.0, one, plane, L.tot, c.stream);
  const cudaError_t le = cudaGetLastError();
  const cudaError_t se = cudaStreamSynchronize(c.stream);
  c.ph = keep;
  c.phw = keepw;
  if (le != cudaSuccess || se != cudaSuccess)
    return fail(PMG_ECUDA, std::string("gauge constant: ") + cudaGetErrorString(le != cudaSuccess ? le : se));
  return PMG_OK;
}

// R += Cgauge on the levels that have one (the residual calls' output).
static void add_gauge_constant(Ctx& c, int l, double* R) {
  LevelDev& L = c.lev[l];
  if (!L.Cgauge) return;
  Scale5 one;
  for (double& x : one.s) x = 1.0;
  launch_plane_combine(R, R, 1.0, L.Cgauge, 1.0, one, nullptr, 0.0, one, (size_t)c.E * L.N, L.tot, c.stream);
}

pmg_status pmg_upload_mesh(pmg_ctx* h, const pmg_mesh* m) {
  if (!h || !m || !m->nodes || !m->nbr) return fail(PMG_EINVAL, "null argument");
  Ctx& c = h->c;
  if (c.mesh_ready) return fail(PMG_EINVAL, "mesh already uploaded");
  if (m->n_elem < 1 || m->geom_order < 1 || m->geom_order > 4) return fail(PMG_EINVAL, "bad mesh sizes");
  if (c.ph.p_ref != 0.0 && c.cfg.P[0] < m->geom_order && m->geom_order > 1)
    return fail(PMG_EINVAL, "p_gauge != 0 needs P >= geometry order on the finest level (the metric identity)");
  const int T_slot = c.dim == 3 ? 4 : 3;   // temperature in q_inf
  for (int i = 0; i < m->n_elem * c.nfc; ++i) {
    if (m->nbr[i * 3] != -1) continue;
    const int bc = m->nbr[i * 3 + 1];
    if (bc == PMG_BC_SLIP_WALL && c.ph.mu > 0.0) return fail(PMG_EINVAL, "slip walls are for mu = 0 only");
    if (bc == PMG_BC_NOSLIP_WALL && !(c.ph.eps_min > 0.0))
      return fail(PMG_EINVAL, "a no-slip wall needs the eps cut-off (cutoff = 1, kappa Ma_inf > 0)");
    if (bc == PMG_BC_FARFIELD && !(c.ph.qinf[0] > 0.0 && c.ph.qinf[T_slot] > 0.0))
      return fail(PMG_EINVAL, "far-field faces need a free stream with p > 0 and T > 0");
  }
  c.E = m->n_elem;
  c.mesh.E = m->n_elem;
  c.mesh.Ng = m->geom_order;
  int nn = 1;
  for (int d = 0; d < c.dim; ++d) nn *= m->geom_order + 1;
  c.mesh.nodes.assign(m->nodes, m->nodes + (size_t)c.E * nn * c.dim);
  c.mesh.nbr.assign(m->nbr, m->nbr + (size_t)c.E * c.nfc * 3);
  std::vector<Ref1D> refs;
  std::vector<LevelGeomHost> geo(c.cfg.n_levels);
  try {
    if (c.dim == 3) build_faces3(c.mesh);
    else build_faces(c.mesh);
    for (int l = 0; l < c.cfg.n_levels; ++l) {
      refs.push_back(make_ref1d(c.cfg.P[l]));
      if (c.dim == 3) build_level_geometry3(c.mesh, refs[l], geo[l]);
      else build_level_geometry(c.mesh, refs[l], geo[l]);
    }
  } catch (const std::exception& ex) {
    return fail(PMG_EINVAL, ex.what());
  }
  {
    std::vector<double> dx = c.dim == 3 ? std::vector<double>(c.E, 1.0) : element_sizes(c.mesh);
    PMG_CK(dalloc(&c.d_dx, dx.size()));
    PMG_CK(cudaMemcpy(c.d_dx, dx.data(), dx.size() * 8, cudaMemcpyHostToDevice));
  }
  c.n_faces = (int)c.mesh.faces.size();
  // face list followed by the neighbour table
  std::vector<int> fbuf((size_t)c.n_faces * 5 + (size_t)c.E * c.nfc * 3);
  for (int f = 0; f < c.n_faces; ++f) {
    const FaceRec& r = c.mesh.faces[f];
    int* o = &fbuf[(size_t)f * 5];
    o[0] = r.eL; o[1] = r.fL; o[2] = r.eR; o[3] = r.fR; o[4] = r.rev;
  }
  memcpy(&fbuf[(size_t)c.n_faces * 5], c.mesh.nbr.data(), sizeof(int) * c.E * c.nfc * 3);
  PMG_CK(dalloc(&c.d_faces, fbuf.size()));
  PMG_CK(cudaMemcpy(c.d_faces, fbuf.data(), sizeof(int) * fbuf.size(), cudaMemcpyHostToDevice));
  size_t maxtot = 0;
  int maxblocks = 1;
  PMG_CK(cudaDeviceGetAttribute(&c.sms, cudaDevAttrMultiProcessorCount, c.device));
  size_t wbytes = c.cfg.block_prec == PMG_PREC_FP64 ? 8 : c.cfg.block_prec == PMG_PREC_BF16R ? 2 : 4;
  for (int l = 0; l < c.cfg.n_levels; ++l) {
    LevelDev& L = c.lev[l];
    const Ref1D& r = refs[l];
    L.level = l;
    L.P = r.P; L.n1 = r.P + 1;
    L.N = c.dim == 3 ? L.n1 * L.n1 * L.n1 : L.n1 * L.n1;
    L.NF = c.dim == 3 ? L.n1 * L.n1 : L.n1;
    L.n = c.nv * L.N;
    L.tot = (size_t)c.nv * c.E * L.N;
    maxtot = std::max(maxtot, L.tot);
    memset(&L.op, 0, sizeof(L.op));
    for (int i = 0; i < L.n1; ++i) {
      for (int k = 0; k < L.n1; ++k) L.op.D[i][k] = r.D[i * L.n1 + k];
      L.op.lm[i] = r.lm[i]; L.op.lp[i] = r.lp[i]; L.op.gL[i] = r.gL[i]; L.op.gR[i] = r.gR[i];
    }
    // D - gL lm^T - gR lp^T: the derivative with the extrapolated part of both
    // faces' corrections folded in, so that the divergence of a line is
    // Dt F + gL (common flux at -1) + gR (common flux at +1)
    for (int i = 0; i < L.n1; ++i)
      for (int k = 0; k < L.n1; ++k) {
        L.op.Dt[i][k] = (double)((long double)r.D[i * L.n1 + k] - (long double)r.gL[i] * r.lm[k] -
                                 (long double)r.gR[i] * r.lp[k]);
        L.op.hlm[k] = 0.5 * r.lm[k];
        L.op.hlp[k] = 0.5 * r.lp[k];
      }
    // BR2 lifting factor: penalty eta_f = 4 (faces of a quadrilateral) times
    // the DG correction's g_R'(1) = (P+1)^2 / 2
    L.op.pen = 4.0 * 0.5 * L.n1 * L.n1;
    memset(&L.opw, 0, sizeof(L.opw));
    for (int i = 0; i < L.n1; ++i) {
      for (int k = 0; k < L.n1; ++k) L.opw.Dt[i][k] = dw_const(L.op.Dt[i][k]);
      L.opw.gL[i] = dw_const(L.op.gL[i]);
      L.opw.gR[i] = dw_const(L.op.gR[i]);
    }
    size_t nn2 = (size_t)c.E * L.n * L.n;
    if (dalloc(&L.q, L.tot) || dalloc(&L.qb, L.tot) || dalloc(&L.S, L.tot) || dalloc(&L.F, L.tot) ||
        dalloc(&L.Pd, L.tot) ||
        dalloc(&L.Fcom, (size_t)c.nv * c.E * c.nfc * L.NF) || dalloc(&L.Dfull, nn2) ||
        cudaMalloc(&L.Dinv, nn2 * wbytes) || dalloc(&L.rs, (size_t)c.E * L.n) || dalloc(&L.cs, (size_t)c.E * L.n))
      return fail(PMG_ENOMEM, "device allocation failed for level data");
    // Small levels are smoothed by a fused one-launch sweep (k_fused.cu; coarse
    // P = 0 levels of hexahedra k3_fused.cu), which evaluates every face from both
    // of its elements: the extra face work runs on SM sub-partitions the split
    // launches leave idle and a launch is saved, until that work fills them.  The
    // limits in elements per SM are where the two cross on 152 SMs.  us a sweep,
    // split / fused, 20 sweeps of one level (finest or coarse, the launches are the
    // same), FP32 blocks (FP64 blocks cross at the same sizes):
    //   double-word P = 2: 11.6 / 10.0 at 64 elements, 13.5 / 12.2 at 1936, 13.5 /
    //     13.5 at 2304; P = 1: 10.0 / 8.5 at 64, 11.6 / 11.0 at 4096, 11.8 / 12.2 at
    //     5184; P = 0: 8.5 / 6.7 at 64, 9.5 / 7.3 at 8100;
    //   binary64 P = 2: 16.2 / 14.7 at 64, 17.9 / 16.2 at 1156, 18.4 / 21.5 at 1600;
    //     P = 1: 15.3 / 13.6 at 64, 15.9 / 14.8 at 2304, 16.0 / 19.6 at 3136; P = 0:
    //     13.6 / 10.7 at 64, 14.1 / 11.0 at 3136;
    //   double-word faces in absolute pressure: the crossings of binary64 at P = 2
    //     (15.4 / 14.7 at 1600, 15.9 / 16.5 at 1936) and P = 1 (13.5 / 13.5 at 3136).
    // A finest P = 0 level keeps to the limit of P = 1.  PMG_FUSE_MAX_P sets the
    // highest fused P instead (-1: none).
    bool boundary = false;
    for (const FaceRec& fr : c.mesh.faces) boundary = boundary || fr.eR < 0;
    const bool words = flux_dw_sweep(c) && c.ph.p_ref != 0.0;
    const int small1 = words ? 28 : 16, per_sm[3] = {l == 0 ? small1 : 1 << 20, small1, words ? 14 : 8};
    bool fuse = L.P <= 2 && c.E <= (long long)per_sm[L.P <= 2 ? L.P : 2] * c.sms;
    bool fuse3 = fused3_applies(L.P, c.E, c.sms);
    if (const char* env = getenv("PMG_FUSE_MAX_P")) {
      fuse = L.P <= atoi(env) && L.P <= 3;
      fuse3 = fuse3 && atoi(env) >= 0;
    }
    L.fused = c.dim == 3 ? l > 0 && fuse3 : fuse && c.ph.mu == 0.0 && !boundary;
    // Coarse levels with P <= 1 that the double-word sweep arithmetic serves
    // (gauge storage, mu = 0, no boundary faces) may be smoothed by the fused
    // one-sweep kernel or by the multi-sweep tiles (k_tile.cu); pmg_autotune
    // chooses between them.  Without it: up to PMG_TILE_DEPTH (P = 0) or
    // PMG_TILE_DEPTH1 (P = 1) sweeps per launch on cores of PMG_TILE_CORE
    // (default 32) or PMG_TILE_CORE1 (default 16) elements.
    L.tileable = c.dim == 2 && l > 0 && L.P <= 1 && c.ph.mu == 0.0 && !boundary && c.ph.p_ref != 0.0 &&
                 flux_dw_sweep(c);
    if ((L.fused || L.tileable) && dalloc(&L.q2, L.tot))
      return fail(PMG_ENOMEM, "device allocation failed for level data");
    if (L.fused && L.tileable) {
      int depth = 0, core = L.P == 0 ? 32 : 16;
      if (const char* env = getenv(L.P == 0 ? "PMG_TILE_DEPTH" : "PMG_TILE_DEPTH1")) depth = atoi(env);
      if (const char* env = getenv(L.P == 0 ? "PMG_TILE_CORE" : "PMG_TILE_CORE1")) core = atoi(env);
      if (depth > 0 && core > 0) {
        pmg_status ts = set_level_tiles(c, L, core, depth);
        if (ts) return ts;
      }
    }
    if (c.ph.mu > 0.0) {
      const size_t ng = c.dim == 3 ? (size_t)12 * c.E * L.N : (size_t)6 * c.E * L.N;
      const size_t nj = c.dim == 3 ? (size_t)4 * c.E * 6 * L.NF : (size_t)3 * c.E * 4 * L.n1;
      if (dalloc(&L.Gb, ng) || dalloc(&L.Qj, nj) || dalloc(&L.fJinv, geo[l].fJinv.size()))
        return fail(PMG_ENOMEM, "device allocation failed for level data");
      // the gradient launch leaves out P = 0, where the broken gradient is zero
      PMG_CK(cudaMemset(L.Gb, 0, ng * 8));
      PMG_CK(cudaMemcpy(L.fJinv, geo[l].fJinv.data(), geo[l].fJinv.size() * 8, cudaMemcpyHostToDevice));
    }
    PMG_CK(cudaMemset(L.S, 0, L.tot * 8));
    PMG_CK(cudaMemset(L.q, 0, L.tot * 8));
    {
      // metrics and face geometry, and both in double-word where the sweeps
      // take them so, in one buffer and one copy
      const size_t nm = geo[l].met.size(), nfc = geo[l].face.size(), nb = nm + nfc;
      const bool words = volume_dw_applies(c);
      std::vector<double> buf(words ? 2 * nb : nb);
      std::copy(geo[l].met.begin(), geo[l].met.end(), buf.begin());
      std::copy(geo[l].face.begin(), geo[l].face.end(), buf.begin() + nm);
      if (words)
        for (size_t i = 0; i < nb; ++i) {
          const dw w = dw_const(buf[i]);
          memcpy(&buf[nb + i], &w, sizeof(w));
        }
      if (dalloc(&L.met, buf.size())) return fail(PMG_ENOMEM, "device allocation failed for level data");
      PMG_CK(cudaMemcpy(L.met, buf.data(), buf.size() * 8, cudaMemcpyHostToDevice));
      L.face = L.met + nm;
      if (words) {
        L.metW = reinterpret_cast<dw*>(L.met + nb);
        L.faceW = L.metW + nm;
      }
    }
    c.xy_host[l] = geo[l].xy;
    maxblocks = std::max(maxblocks, c.dim == 3 ? residual_blocks_for3(L.P, c.E) : residual_blocks_for(L.P, c.E));
  }
  for (int l = 0; l + 1 < c.cfg.n_levels; ++l) {
    std::vector<double> R, I;
    make_transfer(refs[l], refs[l + 1], R, I);
    int nf = refs[l].P + 1, nc = refs[l + 1].P + 1;
    memset(&c.xfer[l], 0, sizeof(XferTab));
    for (int i = 0; i < nc; ++i)
      for (int q = 0; q < nf; ++q) c.xfer[l].R[i][q] = R[i * nf + q];
    for (int i = 0; i < nf; ++i)
      for (int k = 0; k < nc; ++k) c.xfer[l].I[i][k] = I[i * nc + k];
  }
  size_t tot0 = c.lev[0].tot;
  c.tmp_size = maxtot;
  if (dalloc(&c.src, tot0) || dalloc(&c.qn, tot0) || dalloc(&c.qcn, tot0) || dalloc(&c.d_tmp0, maxtot) ||
      dalloc(&c.d_tmp1, maxtot) || dalloc(&c.d_partial, (size_t)maxblocks))
    return fail(PMG_ENOMEM, "device allocation failed for stage data");
  for (int j = 0; j < c.stages; ++j)
    if (dalloc(&c.Rst[j], tot0)) return fail(PMG_ENOMEM, "device allocation failed for stage data");
  PMG_CK(cudaMemset(c.src, 0, tot0 * 8));
  c.n_partial = maxblocks;
  PMG_CK(prepare_kernels(c));
  PMG_CK(prepare_assemble(c));
  if (c.dim == 2) {
    PMG_CK(prepare_residual_kernels(c));
    PMG_CK(prepare_volume_dw_kernels(c));
  } else {
    PMG_CK(prepare_apply3(c));
  }
  if (c.ph.p_ref != 0.0 && c.mesh.Ng > 1)
    for (int l = 1; l < c.cfg.n_levels; ++l)
      if (c.cfg.P[l] < c.mesh.Ng) {
        pmg_status gs = compute_gauge_constant(c, l);
        if (gs) return gs;
      }
  c.mesh_ready = true;
  return PMG_OK;
}

}  // extern "C"

// ------------------------------------------------------------------ helpers
static pmg_status check_level(const Ctx& c, int level) {
  if (!c.mesh_ready) return fail(PMG_ESTATE, "mesh not uploaded");
  if (level < 0 || level >= c.cfg.n_levels) return fail(PMG_EINVAL, "level out of range");
  return PMG_OK;
}

static cudaError_t copy_in(const Ctx& c, double* dst, const double* src, size_t count, int on_device) {
  return cudaMemcpyAsync(dst, src, count * 8, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                         c.stream);
}

static cudaError_t copy_out(const Ctx& c, double* dst, const double* src, size_t count, int on_device) {
  cudaError_t e = cudaMemcpyAsync(dst, src, count * 8, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                                  c.stream);
  if (e != cudaSuccess) return e;
  return cudaStreamSynchronize(c.stream);
}

// Whether this context's kernels may read or write the n doubles at p
// themselves: memory of its own device from the first to the last byte, where a
// double may lie.  A copy also takes peers' memory and any address, and refuses
// a buffer that ends too early, where a kernel would fault.
static bool own_memory(const Ctx& c, const void* p, size_t n) {
  if (reinterpret_cast<uintptr_t>(p) % sizeof(double)) return false;
  for (const char* b : {(const char*)p, (const char*)p + n * sizeof(double) - 1}) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, b) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    if (a.type != cudaMemoryTypeDevice || a.device != c.device) return false;
  }
  return true;
}

// A caller's state into dst as the device holds it (pressure relative to p_gauge).
static cudaError_t state_in(const Ctx& c, double* dst, const double* src, const LevelDev& L, int on_device) {
  if (on_device && own_memory(c, src, L.tot)) {
    launch_copy_shift(L.tot / c.nv, L.tot, -c.ph.p_ref, src, dst, c.stream);
    return cudaGetLastError();
  }
  const cudaError_t e = copy_in(c, dst, src, L.tot, on_device);
  if (e == cudaSuccess) launch_shift_pressure(L.tot / c.nv, -c.ph.p_ref, dst, c.stream);
  return e;
}

static int residual_block_count(const Ctx& c, int l) {
  return c.dim == 3 ? residual_blocks_for3(c.lev[l].P, c.E) : residual_blocks_for(c.lev[l].P, c.E);
}

// ------------------------------------------------------------- profiler
// Event pairs around individual launches (only outside graph capture).
static void prof_harvest(Ctx& c) {
  Profiler& p = c.prof;
  if (p.used == 0) return;
  cudaEventSynchronize(p.ev[2 * (p.used - 1) + 1]);
  for (int k = 0; k < p.used; ++k) {
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, p.ev[2 * k], p.ev[2 * k + 1]) == cudaSuccess) {
      int cls = p.tag[k] / kMaxLevels, lvl = p.tag[k] % kMaxLevels;
      p.ms[cls][lvl] += ms;
      p.count[cls][lvl] += 1;
    }
  }
  p.used = 0;
}

static int prof_begin(Ctx& c, int cls, int level) {
  Profiler& p = c.prof;
  if (!p.on) return -1;
  if (p.used == (int)p.tag.size()) prof_harvest(c);
  int k = p.used++;
  p.tag[k] = cls * kMaxLevels + level;
  cudaEventRecord(p.ev[2 * k], c.stream);
  return k;
}

static void prof_end(Ctx& c, int k) {
  if (k >= 0) cudaEventRecord(c.prof.ev[2 * k + 1], c.stream);
}

struct ProfScope {
  Ctx& c;
  int k;
  ProfScope(Ctx& cc, int cls, int level) : c(cc), k(prof_begin(cc, cls, level)) {}
  ~ProfScope() { prof_end(c, k); }
};

// Level system residual F_l(q_l) - S_l into lev[l].F (norm into d_scal[0] if asked).
static void system_residual(Ctx& c, int l, bool norm, bool have_grad = false) {
  LevelDev& L = c.lev[l];
  {
    ProfScope ps(c, K_FACE, l);
    launch_face_flux(c, L, L.q, c.stream, false, have_grad);
  }
  {
    ProfScope ps(c, K_VOLUME, l);
    const double* qref = l > 0 ? L.qb : (c.split_stage ? c.qn : nullptr);
    launch_volume(c, L, l, L.q, L.F, RES_SYSTEM, 1.0 / c.omega_dt, l == 0 ? c.src : nullptr, l > 0 ? L.S : nullptr,
                  nullptr, nullptr, norm ? c.d_partial : nullptr, c.stream, qref);
  }
  if (norm) {
    ProfScope ps(c, K_NORM, l);
    launch_norm_final(c.d_partial, residual_block_count(c, l), c.d_scal, c.stream);
  }
}

static void refresh_level(Ctx& c, int l) {
  LevelDev& L = c.lev[l];
  {
    ProfScope ps(c, K_ASSEMBLE, l);
    launch_assemble(c, L, L.q, c.d_dtau, 1.0 / c.omega_dt, c.stream);
  }
  {
    ProfScope ps(c, K_FACTOR, l);
    launch_factor(c, L, l, c.cfg.block_prec, c.d_flag, c.stream);
  }
  L.assembled = L.factored = true;
}

// n element-Jacobi sweeps q += D^-1 (F_l(q) - S_l) (eq. smoothing_element_jacobi
// on the level system).  With F_valid, lev[l].F already holds F_l(q) - S_l
// for the current state and the first sweep only applies the blocks; every
// other sweep is one face-flux launch and one volume launch that forms the
// residual and updates the state in place, or one fused launch (coarse
// levels then form the first residual again).  final_residual leaves
// F_l(q) - S_l of the smoothed state in lev[l].F (and its norm, if asked).
// Fused levels return the number of state-buffer swaps.
static int sweeps(Ctx& c, int l, int n, bool F_valid, bool final_residual, bool final_norm) {
  LevelDev& L = c.lev[l];
  if (L.tiled) {
    int swaps = 0;
    for (int done = 0; done < n; done += L.tile_depth) {
      const int ns = std::min(L.tile_depth, n - done);
      {
        ProfScope ps(c, K_FUSED, l);
        launch_tile_sweeps(c, L, L.q, L.q2, ns, 1.0 / c.omega_dt, L.S, L.qb, c.cfg.block_prec, c.stream);
      }
      std::swap(L.q, L.q2);
      ++swaps;
    }
    if (final_residual) system_residual(c, l, final_norm);
    return swaps;
  }
  const double *qref = l > 0 ? L.qb : (c.split_stage ? c.qn : nullptr), *src = l == 0 ? c.src : nullptr,
               *S = l > 0 ? L.S : nullptr;
  int s = 0;
  if (F_valid && n > 0 && (l == 0 || !L.fused)) {
    ProfScope ps(c, K_APPLY, l);
    launch_apply(c, L, c.cfg.block_prec, L.F, L.q, 1, c.stream);
    s = 1;
  }
  if (L.fused) {
    const int swaps = n - s;
    for (; s < n; ++s) {
      {
        ProfScope ps(c, K_FUSED, l);
        launch_fused_sweep(c, L, L.q, L.q2, 1.0 / c.omega_dt, src, S, qref, c.cfg.block_prec, c.stream);
      }
      std::swap(L.q, L.q2);
    }
    if (final_residual) system_residual(c, l, final_norm);
    return swaps;
  }
  // viscous: each update also leaves the broken gradients of its result (have_grad) for the next face launch
  bool have_grad = false;
  for (; s < n; ++s) {
    {
      ProfScope ps(c, K_FACE, l);
      launch_face_flux(c, L, L.q, c.stream, true, have_grad);
    }
    {
      ProfScope ps(c, K_VOLUME, l);
      if (volume_dw_applies(c))
        launch_volume_apply_dw(c, L, L.q, 1.0 / c.omega_dt, src, S, qref, c.cfg.block_prec, c.stream);
      else
        launch_volume_apply(c, L, L.q, 1.0 / c.omega_dt, src, S, qref, c.cfg.block_prec, c.stream,
                            s + 1 < n || final_residual);
    }
    have_grad = c.ph.mu > 0.0;
  }
  if (final_residual) system_residual(c, l, final_norm, have_grad);
  return 0;
}

// After an odd number of swaps, move the state back to the level's first
// buffer so that every V-cycle (and a captured graph) starts from the same one.
static void restore_buffer(Ctx& c, int l, int swaps) {
  LevelDev& L = c.lev[l];
  if (!L.fused || (swaps & 1) == 0) return;
  cudaMemcpyAsync(L.q2, L.q, L.tot * 8, cudaMemcpyDeviceToDevice, c.stream);
  std::swap(L.q, L.q2);
}

// FAS V-cycle from level l (Section 3).
static void vcycle_level(Ctx& c, int l, bool refresh) {
  LevelDev& L = c.lev[l];
  if (refresh) refresh_level(c, l);
  const int nl = c.cfg.n_levels;
  // On entry lev[l].F = F_l(q) - S_l: from the norm evaluation on the finest
  // level, from the forcing evaluation (= -P d) on coarser ones.
  if (l == nl - 1) {
    restore_buffer(c, l, sweeps(c, l, c.cfg.n_smooth[l], true, false, false));
    return;
  }
  int swaps = sweeps(c, l, c.cfg.n_smooth[l], true, true, false);   // pre-smoothing, ends with F(q^a)
  LevelDev& C = c.lev[l + 1];
  const XferTab& X = c.xfer[l];
  {
    ProfScope ps(c, K_RESTRICT, l + 1);
    launch_restrict_fas(c, L, C, X, L.q, C.q, C.qb, L.F, C.Pd, c.stream);   // q^b = P q^a, P d = -P (F - S)
  }
  {
    ProfScope ps(c, K_FACE, l + 1);
    launch_face_flux(c, C, C.q, c.stream);                             // S = F(q^b) + P d
  }
  {
    ProfScope ps(c, K_VOLUME, l + 1);
    launch_volume(c, C, l + 1, C.q, C.F, RES_FORCING, 1.0 / c.omega_dt, nullptr, nullptr, C.S, C.Pd, nullptr,
                  c.stream, C.qb);
  }
  vcycle_level(c, l + 1, refresh);
  {
    ProfScope ps(c, K_PROLONG, l);
    launch_prolong_add(c, L, C, X, C.q, C.qb, L.q, c.stream);         // q += I (q^a_c - q^b_c)
  }
  swaps += sweeps(c, l, c.cfg.n_smooth[l], false, l == 0, l == 0);   // post-smoothing
  restore_buffer(c, l, swaps);
}

static pmg_status launch_vcycle(Ctx& c, bool refresh) {
  if (!c.cfg.use_graph || c.prof.on) {
    vcycle_level(c, 0, refresh);
    PMG_CK_LAUNCH();
    return PMG_OK;
  }
  int g = refresh ? 1 : 0;
  if (!c.graph[g] || c.graph_inv_odt[g] != 1.0 / c.omega_dt || c.graph_split[g] != (int)c.split_stage) {
    if (c.graph[g]) { cudaGraphExecDestroy(c.graph[g]); c.graph[g] = nullptr; }
    cudaGraph_t graph;
    PMG_CK(cudaStreamBeginCapture(c.stream, cudaStreamCaptureModeThreadLocal));
    vcycle_level(c, 0, refresh);
    cudaError_t le = cudaGetLastError();
    cudaError_t ee = cudaStreamEndCapture(c.stream, &graph);
    if (le != cudaSuccess) return fail(PMG_ECUDA, std::string("capture launch: ") + cudaGetErrorString(le));
    if (ee != cudaSuccess) return fail(PMG_ECUDA, std::string("capture: ") + cudaGetErrorString(ee));
    cudaError_t ie = cudaGraphInstantiate(&c.graph[g], graph, 0);
    cudaGraphDestroy(graph);
    if (ie != cudaSuccess) return fail(PMG_ECUDA, std::string("graph instantiate: ") + cudaGetErrorString(ie));
    c.graph_inv_odt[g] = 1.0 / c.omega_dt;
    c.graph_split[g] = (int)c.split_stage;
  }
  PMG_CK(cudaGraphLaunch(c.graph[g], c.stream));
  return PMG_OK;
}

static pmg_status wait_flag_status(Ctx& c) {
  if (c.h_scal[1] == 0.0) return PMG_OK;
  c.h_scal[1] = 0.0;
  cudaMemsetAsync(c.d_scal + 1, 0, sizeof(double), c.stream);
  return fail(PMG_ETIMEOUT, "a kernel's bounded wait for its bulk shared-memory copy gave up (it finished from "
                            "global memory)");
}

// Reads the flag of the bounded bulk-copy waits (after the work queued so far).
static pmg_status check_wait_flag(Ctx& c) {
  PMG_CK(cudaMemcpyAsync(c.h_scal + 1, c.d_scal + 1, sizeof(double), cudaMemcpyDeviceToHost, c.stream));
  PMG_CK(cudaStreamSynchronize(c.stream));
  return wait_flag_status(c);
}

static pmg_status read_norm(Ctx& c, double* out) {
  PMG_CK(cudaMemcpyAsync(c.h_scal, c.d_scal, 2 * sizeof(double), cudaMemcpyDeviceToHost, c.stream));
  PMG_CK(cudaStreamSynchronize(c.stream));
  pmg_status ws = wait_flag_status(c);
  if (ws) return ws;
  *out = std::sqrt(c.h_scal[0]);
  if (c.prof.on) prof_harvest(c);
  return PMG_OK;
}

// dtau_min of the CFL form for the current finest state (d_scal[2]).
static pmg_status compute_dtau_min(Ctx& c, double* out) {
  launch_dtau_min(c, c.d_partial, c.d_scal + 2, c.stream);
  PMG_CK_LAUNCH();
  PMG_CK(cudaMemcpyAsync(c.h_scal + 2, c.d_scal + 2, sizeof(double), cudaMemcpyDeviceToHost, c.stream));
  PMG_CK(cudaStreamSynchronize(c.stream));
  *out = c.h_scal[2];
  return PMG_OK;
}

static pmg_status set_dtau(Ctx& c, double dtau) {
  // the pinned mirror is only rewritten after the stream has consumed it
  PMG_CK(cudaStreamSynchronize(c.stream));
  *c.h_dtau = dtau;
  PMG_CK(cudaMemcpyAsync(c.d_dtau, c.h_dtau, sizeof(double), cudaMemcpyHostToDevice, c.stream));
  return PMG_OK;
}

static pmg_status check_singular(Ctx& c) {
  int flag = 0;
  PMG_CK(cudaMemcpyAsync(&flag, c.d_flag, sizeof(int), cudaMemcpyDeviceToHost, c.stream));
  PMG_CK(cudaStreamSynchronize(c.stream));
  if (flag) {
    cudaMemsetAsync(c.d_flag, 0, sizeof(int), c.stream);
    const int lv = (flag - 1) / c.E, e = (flag - 1) % c.E;
    return fail(PMG_ESINGULAR, "element block " + std::to_string(e) + " of level " + std::to_string(lv) +
                                   " is singular to working precision (pivot not above n eps)");
  }
  return PMG_OK;
}

// ------------------------------------------------------ device-side stage loop
// The graph: WHILE(h_loop) { controller -> IF(h_refresh) { V-cycle with
// smoother rebuild } -> IF(h_plain) { V-cycle } }.  The V-cycle bodies are
// captured from the same launch sequence as the host loop's graphs, for the
// current omega dt and stage form.
static pmg_status build_loop_graph(Ctx& c) {
  if (c.loop_exec) { cudaGraphExecDestroy(c.loop_exec); c.loop_exec = nullptr; }
  cudaGraph_t g = nullptr;
  PMG_CK(cudaGraphCreate(&g, 0));
  struct GraphGuard {
    cudaGraph_t g;
    ~GraphGuard() { if (g) cudaGraphDestroy(g); }
  } guard{g};
  cudaGraphConditionalHandle h_loop, h_refresh, h_plain;
  PMG_CK(cudaGraphConditionalHandleCreate(&h_loop, g, 1, cudaGraphCondAssignDefault));
  cudaGraphNodeParams wp = {};
  wp.type = cudaGraphNodeTypeConditional;
  wp.conditional.handle = h_loop;
  wp.conditional.type = cudaGraphCondTypeWhile;
  wp.conditional.size = 1;
  cudaGraphNode_t wnode;
  PMG_CK(cudaGraphAddNode(&wnode, g, nullptr, nullptr, 0, &wp));
  cudaGraph_t body = wp.conditional.phGraph_out[0];
  PMG_CK(cudaGraphConditionalHandleCreate(&h_refresh, body, 0, cudaGraphCondAssignDefault));
  PMG_CK(cudaGraphConditionalHandleCreate(&h_plain, body, 0, cudaGraphCondAssignDefault));
  // controller node, captured alone into the body
  LoopParams prm;
  prm.tol = c.cfg.tol;
  prm.refresh_every = c.cfg.refresh_every;
  prm.refresh_always = c.cfg.refresh_always;
  prm.max_pseudo = c.cfg.max_pseudo;
  const int mp1 = c.cfg.max_pseudo + 1;
  PMG_CK(cudaStreamBeginCaptureToGraph(c.stream, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
  launch_loop_controller(c.d_loop, c.d_scal, c.d_flag, c.d_dtau, c.d_hist, c.d_hist + mp1, prm, h_loop, h_refresh,
                         h_plain, c.stream);
  {
    cudaError_t le = cudaGetLastError();
    cudaGraph_t got = nullptr;
    cudaError_t ee = cudaStreamEndCapture(c.stream, &got);
    if (le != cudaSuccess) return fail(PMG_ECUDA, std::string("loop capture launch: ") + cudaGetErrorString(le));
    if (ee != cudaSuccess) return fail(PMG_ECUDA, std::string("loop capture: ") + cudaGetErrorString(ee));
  }
  cudaGraphNode_t ctl;
  size_t nn = 1;
  PMG_CK(cudaGraphGetNodes(body, &ctl, &nn));
  if (nn != 1) return fail(PMG_ECUDA, "loop graph: the controller capture did not give one node");
  cudaGraphNode_t prev = ctl;
  for (int r = 1; r >= 0; --r) {   // IF refresh, then IF plain
    cudaGraphNodeParams ip = {};
    ip.type = cudaGraphNodeTypeConditional;
    ip.conditional.handle = r ? h_refresh : h_plain;
    ip.conditional.type = cudaGraphCondTypeIf;
    ip.conditional.size = 1;
    cudaGraphNode_t inode;
    PMG_CK(cudaGraphAddNode(&inode, body, &prev, nullptr, 1, &ip));
    cudaGraph_t vbody = ip.conditional.phGraph_out[0];
    PMG_CK(cudaStreamBeginCaptureToGraph(c.stream, vbody, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
    vcycle_level(c, 0, r == 1);
    cudaError_t le = cudaGetLastError();
    cudaGraph_t got = nullptr;
    cudaError_t ee = cudaStreamEndCapture(c.stream, &got);
    if (le != cudaSuccess) return fail(PMG_ECUDA, std::string("V-cycle capture launch: ") + cudaGetErrorString(le));
    if (ee != cudaSuccess) return fail(PMG_ECUDA, std::string("V-cycle capture: ") + cudaGetErrorString(ee));
    prev = inode;
  }
  cudaError_t ie = cudaGraphInstantiate(&c.loop_exec, g, 0);
  if (ie != cudaSuccess) {
    c.loop_exec = nullptr;
    return fail(PMG_ECUDA, std::string("loop graph instantiate: ") + cudaGetErrorString(ie));
  }
  c.loop_inv_odt = 1.0 / c.omega_dt;
  c.loop_split = (int)c.split_stage;
  return PMG_OK;
}

// The stage's pseudo-iterations as one graph launch (cfg.device_loop); the
// initial residual norm is in d_scal[0].  One synchronisation at the end reads
// the loop state and the norm / dtau history.
static pmg_status stage_solve_device(Ctx& c, double dtau_init, double dtau_max, int* iters, double* drop,
                                     int* n_refresh) {
  if (!c.loop_exec || c.loop_inv_odt != 1.0 / c.omega_dt || c.loop_split != (int)c.split_stage) {
    pmg_status st = build_loop_graph(c);
    if (st) return st;
  }
  LoopState& h = *c.h_loop;
  PMG_CK(cudaStreamSynchronize(c.stream));   // the pinned mirror is free to rewrite
  memset(&h, 0, sizeof(h));
  h.dtau = dtau_init;
  h.dtau_max = dtau_max;
  h.status = LOOP_RUNNING;
  PMG_CK(cudaMemcpyAsync(c.d_loop, &h, sizeof(LoopState), cudaMemcpyHostToDevice, c.stream));
  PMG_CK(cudaGraphLaunch(c.loop_exec, c.stream));
  const size_t mp1 = (size_t)c.cfg.max_pseudo + 1;
  PMG_CK(cudaMemcpyAsync(&h, c.d_loop, sizeof(LoopState), cudaMemcpyDeviceToHost, c.stream));
  PMG_CK(cudaMemcpyAsync(c.h_hist, c.d_hist, 2 * mp1 * sizeof(double), cudaMemcpyDeviceToHost, c.stream));
  PMG_CK(cudaMemcpyAsync(c.h_scal + 1, c.d_scal + 1, sizeof(double), cudaMemcpyDeviceToHost, c.stream));
  PMG_CK(cudaStreamSynchronize(c.stream));
  const int nrec = std::min(h.iters, c.cfg.max_pseudo) + 1;
  for (int k = 0; k < nrec; ++k) {
    c.hist_norm.push_back(c.h_hist[k]);
    c.hist_dtau.push_back(c.h_hist[mp1 + k]);
  }
  if (n_refresh) *n_refresh += h.n_refresh;
  if (iters) *iters = h.iters;
  const double nm = h.final_norm, n0 = h.n0;
  switch (h.status) {
    case LOOP_CONVERGED:
      if (drop) *drop = n0 > 0 ? nm / n0 : 0.0;
      return PMG_OK;
    case LOOP_NONFINITE:
      if (drop) *drop = nm;
      return fail(PMG_ENONFINITE, "non-finite residual norm");
    case LOOP_SINGULAR:
      if (drop) *drop = n0 > 0 ? nm / n0 : nm;
      return check_singular(c);
    case LOOP_TIMEOUT:
      if (drop) *drop = n0 > 0 ? nm / n0 : nm;
      return wait_flag_status(c);
    case LOOP_NOTCONV:
      if (drop) *drop = n0 > 0 ? nm / n0 : nm;
      return fail(PMG_ENOTCONV, "stage not converged within max_pseudo V-cycles");
    default:
      return fail(PMG_ECUDA, "device stage loop ended in an unknown state");
  }
}

// Pseudo-transient continuation of the current stage (Section 2.4).
// ------------------------------------------------- Newton-Krylov stage solver
// Newton on the stage system with restarted, right-preconditioned FGMRES
// (Saad 1993) in the space where each equation is divided by its residual
// scale; classical Gram-Schmidt done twice, Givens rotations on the host.
// The Jacobian acts only through differences of binary64 stage residuals
// (the matrix-free products the paper's introduction describes); the
// preconditioner is the element-block Jacobi smoother's blocks or one FAS
// V-cycle (Section 3) -- the P-multigrid preconditioner the paper's
// concluding section proposes.
static pmg_nk_options nk_defaults(const Ctx& c, const pmg_nk_options* o) {
  pmg_nk_options r;
  memset(&r, 0, sizeof(r));
  if (o) r = *o;
  else r.precond = PMG_NK_PC_VCYCLE;
  if (r.max_newton <= 0) r.max_newton = 30;
  if (r.krylov_dim <= 0) r.krylov_dim = 20;
  if (r.max_krylov <= 0) r.max_krylov = 2 * r.krylov_dim;
  if (!(r.eta > 0.0)) r.eta = 1e-2;
  if (!(r.dtau_pc > 0.0)) r.dtau_pc = c.cfg.dtau_max;
  if (r.pc_refresh <= 0) r.pc_refresh = 1;
  if (!(r.delta0 > 0.0)) r.delta0 = 1e-7;
  if (r.max_backtrack < 0) r.max_backtrack = 6;
  if (!(r.pc_eps > 0.0)) r.pc_eps = 0.1;
  if (!(r.max_update > 0.0)) r.max_update = 0.2;
  if (!(r.ptc_dtau > 0.0)) r.ptc_dtau = 0.0;
  return r;
}

static pmg_status nk_alloc(Ctx& c, int m) {
  if (c.nk_V && c.nk_m >= m) return PMG_OK;
  nk_free(c);
  const size_t n = c.lev[0].tot;
  if (dalloc(&c.nk_q, n) || dalloc(&c.nk_F, n) || dalloc(&c.nk_src, n) || dalloc(&c.nk_w, n) ||
      dalloc(&c.nk_t, n) || dalloc(&c.nk_x, n) || dalloc(&c.nk_V, (size_t)(m + 1) * n) ||
      dalloc(&c.nk_Z, (size_t)m * n) || dalloc(&c.nk_part, (size_t)kDotBlocks * (m + 2)) ||
      dalloc(&c.nk_dots, (size_t)3 * m + 3) || dalloc(&c.nk_coef, (size_t)m + 1) ||
      cudaMallocHost((void**)&c.h_nk, ((size_t)3 * m + 3) * sizeof(double)) != cudaSuccess) {
    nk_free(c);
    return fail(PMG_ENOMEM, "device allocation failed for the Newton-Krylov vectors");
  }
  c.nk_m = m;
  return PMG_OK;
}

// The vectors and the finest level's operators the solver works with.
struct NkWork {
  Ctx& c;
  LevelDev& L;
  pmg_nk_options o;
  size_t n, plane;
  Scale5 one, W, Winv, sinv;
  int m;
  double ptc_inv = 0.0;   // 1 / dtau of pseudo-transient Newton, 0 for Newton
  double dpc;             // the preconditioner's dtau

  NkWork(Ctx& cc, const pmg_nk_options& oo) : c(cc), L(cc.lev[0]), o(oo) {
    n = L.tot;
    plane = (size_t)c.E * L.N;
    m = o.krylov_dim;
    dpc = o.dtau_pc;
    for (int v = 0; v < 5; ++v) {
      one.s[v] = 1.0;
      W.s[v] = v < c.nv ? c.ph.nw[v] : 1.0;
      Winv.s[v] = 1.0 / W.s[v];
      sinv.s[v] = 1.0;
    }
  }
  void combine(double* out, const double* x0, double a0, const double* x1, double a1, const Scale5& s0,
               const double* x2, double a2, const Scale5& s2) {
    launch_plane_combine(out, x0, a0, x1, a1, s0, x2, a2, s2, plane, n, c.stream);
  }
  void copy(double* dst, const double* src) { combine(dst, src, 1.0, nullptr, 0.0, one, nullptr, 0.0, one); }
  // h_nk[0..count) <- nk_dots[0..count)
  pmg_status fetch(int count) {
    PMG_CK(cudaMemcpyAsync(c.h_nk, c.nk_dots, count * sizeof(double), cudaMemcpyDeviceToHost, c.stream));
    PMG_CK(cudaStreamSynchronize(c.stream));
    return PMG_OK;
  }
  // ||x||_2 of a vector of the finest size
  pmg_status norm2(const double* x, double* out) {
    launch_multi_dot(x, n, 1, x, n, c.nk_part, c.nk_dots, c.stream);
    pmg_status st = fetch(1);
    if (st) return st;
    *out = std::sqrt(std::max(c.h_nk[0], 0.0));
    return PMG_OK;
  }
  // state scales: the option, else the RMS of the variable in q (+ |p_gauge| for p)
  pmg_status set_state_scales(const double* q) {
    for (int v = 0; v < c.nv; ++v) {
      double sv = o.state_scale[v];
      if (!(sv > 0.0)) {
        launch_multi_dot(q + v * plane, plane, 1, q + v * plane, plane, c.nk_part, c.nk_dots, c.stream);
        pmg_status st = fetch(1);
        if (st) return st;
        sv = std::sqrt(std::max(c.h_nk[0], 0.0) / (double)plane) + (v == 0 ? std::fabs(c.ph.p_ref) : 0.0);
        if (!(sv > 0.0) || !std::isfinite(sv)) sv = 1.0;
      }
      sinv.s[v] = 1.0 / sv;
    }
    return PMG_OK;
  }
  // w = W A z = -W (F(q + h z) - F(q)) / h at q = nk_q (F(q) in nk_F),
  // + W Gamma(q) z / dtau in pseudo-transient Newton
  pmg_status apply_A(const double* z, double* w) {
    combine(c.nk_t, z, 1.0, nullptr, 0.0, sinv, nullptr, 0.0, one);
    double ss;
    pmg_status st = norm2(c.nk_t, &ss);
    if (st) return st;
    const double rms = ss / std::sqrt((double)n);
    if (!(rms > 0.0)) {
      PMG_CK(cudaMemsetAsync(w, 0, n * sizeof(double), c.stream));
      return PMG_OK;
    }
    const double h = o.delta0 / rms;
    combine(L.q, c.nk_q, 1.0, nullptr, 0.0, one, z, h, one);
    system_residual(c, 0, false);
    Scale5 Wh;
    for (int v = 0; v < 5; ++v) Wh.s[v] = -W.s[v] / h;
    combine(w, L.F, 1.0, c.nk_F, -1.0, Wh, nullptr, 0.0, one);
    if (ptc_inv > 0.0) launch_gamma_apply(c.nv, plane, c.nk_q, z, w, ptc_inv, W, c.ph, c.stream);
    ++c.nk_count[3];
    PMG_CK_LAUNCH();
    return PMG_OK;
  }
  // z = M^-1 (v / W): the element blocks, or one V-cycle on the stage system
  // with source src - F(q) + eps v / W from q, z = (q' - q) / eps
  pmg_status apply_M(const double* v, double* z, bool* refresh, double eps) {
    if (o.precond == PMG_NK_PC_BLOCK) {
      combine(c.nk_t, v, 1.0, nullptr, 0.0, Winv, nullptr, 0.0, one);
      launch_apply(c, L, c.cfg.block_prec, c.nk_t, z, 0, c.stream);
      PMG_CK_LAUNCH();
      return PMG_OK;
    }
    combine(c.src, c.nk_src, 1.0, c.nk_F, -1.0, one, v, eps, Winv);
    copy(L.q, c.nk_q);
    system_residual(c, 0, false);   // the V-cycle starts from lev[0].F = F(q) - S
    pmg_status st;
    if (*refresh) {
      st = set_dtau(c, dpc);
      if (st) return st;
    }
    st = launch_vcycle(c, *refresh);
    if (st) return st;
    if (*refresh) {
      st = check_singular(c);
      if (st) return st;
      *refresh = false;
    }
    combine(z, L.q, 1.0 / eps, c.nk_q, -1.0 / eps, one, nullptr, 0.0, one);
    copy(c.src, c.nk_src);
    ++c.nk_count[2];
    PMG_CK_LAUNCH();
    return PMG_OK;
  }

  // One inexact Newton correction: FGMRES on A x = F(q) into nk_x.
  pmg_status krylov(double eps, bool refresh) {
    PMG_CK(cudaMemsetAsync(c.nk_x, 0, n * sizeof(double), c.stream));
    combine(c.nk_V, c.nk_F, 1.0, nullptr, 0.0, W, nullptr, 0.0, one);   // b = W F
    double beta0;
    pmg_status st = norm2(c.nk_V, &beta0);
    if (st) return st;
    const double target = o.eta * beta0;
    double res = beta0;
    int it = 0;
    bool first = true;
    std::vector<double> H((size_t)(m + 1) * m), cs(m), sn(m), g(m + 1), y(m);
    while (it < o.max_krylov && res > target) {
      double beta = beta0;
      if (!first) {   // restart from r = b - A x
        st = apply_A(c.nk_x, c.nk_w);
        if (st) return st;
        combine(c.nk_V, c.nk_F, 1.0, nullptr, 0.0, W, c.nk_w, -1.0, one);
        st = norm2(c.nk_V, &beta);
        if (st) return st;
      }
      first = false;
      if (!(beta > 0.0)) break;
      combine(c.nk_V, c.nk_V, 1.0 / beta, nullptr, 0.0, one, nullptr, 0.0, one);
      std::fill(g.begin(), g.end(), 0.0);
      g[0] = beta;
      int jl = -1;
      for (int j = 0; j < m; ++j) {
        double* Vj = c.nk_V + (size_t)j * n;
        double* Zj = c.nk_Z + (size_t)j * n;
        st = apply_M(Vj, Zj, &refresh, eps);
        if (st) return st;
        st = apply_A(Zj, c.nk_w);
        if (st) return st;
        // classical Gram-Schmidt, twice
        launch_multi_dot(c.nk_V, n, j + 1, c.nk_w, n, c.nk_part, c.nk_dots, c.stream);
        launch_combination(c.nk_w, c.nk_V, n, j + 1, c.nk_dots, -1.0, n, c.stream);
        launch_multi_dot(c.nk_V, n, j + 1, c.nk_w, n, c.nk_part, c.nk_dots + m + 1, c.stream);
        launch_combination(c.nk_w, c.nk_V, n, j + 1, c.nk_dots + m + 1, -1.0, n, c.stream);
        launch_multi_dot(c.nk_w, n, 1, c.nk_w, n, c.nk_part, c.nk_dots + 2 * m + 2, c.stream);
        PMG_CK_LAUNCH();
        st = fetch(2 * m + 3);
        if (st) return st;
        for (int i = 0; i <= j; ++i) H[(size_t)i * m + j] = c.h_nk[i] + c.h_nk[m + 1 + i];
        const double hn = std::sqrt(std::max(c.h_nk[2 * m + 2], 0.0));
        for (int i = 0; i < j; ++i) {
          const double a = H[(size_t)i * m + j], b = H[(size_t)(i + 1) * m + j];
          H[(size_t)i * m + j] = cs[i] * a + sn[i] * b;
          H[(size_t)(i + 1) * m + j] = -sn[i] * a + cs[i] * b;
        }
        const double a = H[(size_t)j * m + j], r = std::hypot(a, hn);
        cs[j] = r > 0.0 ? a / r : 1.0;
        sn[j] = r > 0.0 ? hn / r : 0.0;
        H[(size_t)j * m + j] = r;
        g[j + 1] = -sn[j] * g[j];
        g[j] = cs[j] * g[j];
        res = std::fabs(g[j + 1]);
        ++it;
        ++c.nk_count[1];
        jl = j;
        if (!(hn > 0.0) || res <= target || it >= o.max_krylov) break;
        combine(c.nk_V + (size_t)(j + 1) * n, c.nk_w, 1.0 / hn, nullptr, 0.0, one, nullptr, 0.0, one);
      }
      if (jl < 0) break;
      for (int i = jl; i >= 0; --i) {
        double t = g[i];
        for (int k = i + 1; k <= jl; ++k) t -= H[(size_t)i * m + k] * y[k];
        y[i] = H[(size_t)i * m + i] != 0.0 ? t / H[(size_t)i * m + i] : 0.0;
      }
      for (int i = 0; i <= jl; ++i) c.h_nk[i] = y[i];
      PMG_CK(cudaMemcpyAsync(c.nk_coef, c.h_nk, (jl + 1) * sizeof(double), cudaMemcpyHostToDevice, c.stream));
      launch_combination(c.nk_x, c.nk_Z, n, jl + 1, c.nk_coef, 1.0, n, c.stream);
      PMG_CK_LAUNCH();
      PMG_CK(cudaStreamSynchronize(c.stream));   // h_nk is rewritten by the next fetch
    }
    return PMG_OK;
  }
};

// Newton steps until ||F|| <= tol ||F^0||; iters = Newton steps, *vcycles
// (may be NULL) = the preconditioner's V-cycles.  Leaves the iterate in
// lev[0].q with F(q) in lev[0].F.
static pmg_status nk_stage_solve(Ctx& c, int* iters, double* drop, int* n_refresh, int* vcycles) {
  NkWork w(c, c.nk);
  pmg_status st = nk_alloc(c, w.m);
  if (st) return st;
  LevelDev& L = c.lev[0];
  const long long vc0 = c.nk_count[2];
  auto finish = [&](int k, double nrm, double n0) {
    if (iters) *iters = k;
    if (drop) *drop = n0 > 0.0 ? nrm / n0 : nrm;
    if (vcycles) *vcycles = (int)(c.nk_count[2] - vc0);
  };
  PMG_CK(cudaMemcpyAsync(c.nk_src, c.src, w.n * sizeof(double), cudaMemcpyDeviceToDevice, c.stream));
  system_residual(c, 0, true);
  PMG_CK_LAUNCH();
  double nrm;
  st = read_norm(c, &nrm);
  if (st) return st;
  ++c.nk_count[3];
  w.copy(c.nk_q, L.q);
  w.copy(c.nk_F, L.F);
  c.F0_valid = true;
  st = w.set_state_scales(L.q);
  if (st) return st;
  const double n0 = nrm;
  // pseudo-transient Newton: dtau from ptc_dtau, SER (exponent 1.5, no bound)
  const bool ptc = w.o.ptc_dtau > 0.0;
  double dtau = w.o.ptc_dtau;
  // on an error after this point: the stage source and the last accepted
  // iterate go back where the caller expects them
  auto recover = [&](pmg_status err) {
    cudaMemcpyAsync(c.src, c.nk_src, w.n * sizeof(double), cudaMemcpyDeviceToDevice, c.stream);
    cudaMemcpyAsync(L.q, c.nk_q, w.n * sizeof(double), cudaMemcpyDeviceToDevice, c.stream);
    cudaStreamSynchronize(c.stream);
    c.F0_valid = false;
    return err;
  };
  for (int k = 0;; ++k) {
    c.hist_norm.push_back(nrm);
    c.hist_dtau.push_back(ptc ? dtau : 0.0);
    if (nrm <= c.cfg.tol * n0 || n0 == 0.0) {
      finish(k, nrm, n0);
      return PMG_OK;
    }
    if (!std::isfinite(nrm)) {
      finish(k, nrm, n0);
      return fail(PMG_ENONFINITE, "non-finite residual norm");
    }
    if (k >= w.o.max_newton) {
      finish(k, nrm, n0);
      return fail(PMG_ENOTCONV, "stage not converged within max_newton Newton steps");
    }
    const bool refresh = k % w.o.pc_refresh == 0;
    if (ptc) {
      w.ptc_inv = 1.0 / dtau;
      w.dpc = std::min(dtau, w.o.dtau_pc);
    }
    if (refresh) {
      if (n_refresh) ++*n_refresh;
      if (w.o.precond == PMG_NK_PC_BLOCK) {   // blocks at the iterate (lev[0].q holds it here)
        st = set_dtau(c, w.dpc);
        if (st) return recover(st);
        refresh_level(c, 0);
        st = check_singular(c);
        if (st) return recover(st);
      }
    }
    st = w.krylov(w.o.pc_eps * nrm, refresh && w.o.precond == PMG_NK_PC_VCYCLE);
    if (st) return recover(st);
    // backtracking on ||F||, from a step that changes p and T by at most
    // max_update (pseudo-transient Newton takes that step as it is)
    launch_rel_change(c.nk_q, c.nk_x, w.plane, c.nv - 1, c.ph.p_ref, c.nk_part, c.nk_dots, c.stream);
    PMG_CK_LAUNCH();
    st = w.fetch(1);
    if (st) return recover(st);
    double lam = c.h_nk[0] > w.o.max_update ? w.o.max_update / c.h_nk[0] : 1.0, nn = 0.0;
    const int n_back = ptc ? 0 : w.o.max_backtrack;
    for (int t = 0; t <= n_back; ++t) {
      w.combine(L.q, c.nk_q, 1.0, nullptr, 0.0, w.one, c.nk_x, lam, w.one);
      system_residual(c, 0, true);
      PMG_CK_LAUNCH();
      st = read_norm(c, &nn);
      if (st) return recover(st);
      ++c.nk_count[3];
      if (std::isfinite(nn) && nn <= (1.0 - 1e-4 * lam) * nrm) break;
      if (t < n_back) lam *= 0.5;
    }
    if (ptc && nn > 0.0 && std::isfinite(nn)) dtau *= std::pow(nrm / nn, 1.5);
    w.copy(c.nk_q, L.q);
    w.copy(c.nk_F, L.F);
    ++c.nk_count[0];
    nrm = nn;
  }
}

static pmg_status stage_solve(Ctx& c, int* iters, double* drop, int* n_refresh, int* vcycles = nullptr) {
  if (c.stage_solver == PMG_STAGE_NK) return nk_stage_solve(c, iters, drop, n_refresh, vcycles);
  if (vcycles) *vcycles = -1;   // the caller counts pseudo-iterations
  if (!c.F0_valid) {
    system_residual(c, 0, true);
    PMG_CK_LAUNCH();
    c.F0_valid = true;
  }
  if (c.cfg.device_loop && c.cfg.use_graph && !c.prof.on) {
    double dtau_init = c.cfg.dtau_init, dtau_max = c.cfg.dtau_max;
    if (c.cfg.cfl_mode) {
      double dm;
      pmg_status st = compute_dtau_min(c, &dm);
      if (st) return st;
      if (!(dm > 0.0) || !std::isfinite(dm)) return fail(PMG_ENONFINITE, "dtau_min is not a positive number");
      dtau_init = c.cfg.cfl_init * dm;
      dtau_max = c.cfg.cfl_max * dm;
    }
    return stage_solve_device(c, dtau_init, dtau_max, iters, drop, n_refresh);
  }
  double nm;
  pmg_status st = read_norm(c, &nm);
  if (st) return st;
  double dtau_init = c.cfg.dtau_init, dtau_max = c.cfg.dtau_max;
  if (c.cfg.cfl_mode) {   // Section 2.4: dtau = CFL dtau_min, SER acting on the CFL number
    double dm;
    st = compute_dtau_min(c, &dm);
    if (st) return st;
    if (!(dm > 0.0) || !std::isfinite(dm)) return fail(PMG_ENONFINITE, "dtau_min is not a positive number");
    dtau_init = c.cfg.cfl_init * dm;
    dtau_max = c.cfg.cfl_max * dm;
  }
  double n0 = nm, prev = nm, dtau = dtau_init, built = 0.0;
  for (int m = 0;; ++m) {
    if (m == 0) n0 = nm;
    c.hist_norm.push_back(nm);
    c.hist_dtau.push_back(m > 0 ? std::min(dtau * std::pow(prev / nm, 1.5), dtau_max) : dtau);
    if (nm <= c.cfg.tol * n0 || n0 == 0.0) {
      if (iters) *iters = m;
      if (drop) *drop = n0 > 0 ? nm / n0 : 0.0;
      return PMG_OK;
    }
    if (!std::isfinite(nm)) {
      if (iters) *iters = m;
      if (drop) *drop = nm;
      return fail(PMG_ENONFINITE, "non-finite residual norm");
    }
    if (m >= c.cfg.max_pseudo) {
      if (iters) *iters = m;
      if (drop) *drop = nm / n0;
      return fail(PMG_ENOTCONV, "stage not converged within max_pseudo V-cycles");
    }
    if (m > 0) dtau = std::min(dtau * std::pow(prev / nm, 1.5), dtau_max);
    bool refresh = (m == 0) || (m % c.cfg.refresh_every == 0 && (c.cfg.refresh_always || built < dtau_max));
    if (refresh) {
      built = dtau;
      st = set_dtau(c, dtau);
      if (st) return st;
      if (n_refresh) ++*n_refresh;
    }
    st = launch_vcycle(c, refresh);
    if (st) return st;
    if (refresh) {
      st = check_singular(c);
      if (st) return st;
    }
    prev = nm;
    st = read_norm(c, &nm);
    if (st) return st;
  }
}

extern "C" {

pmg_status pmg_point_coords(pmg_ctx* h, int level, double* xy) {
  if (!h || !xy) return fail(PMG_EINVAL, "null argument");
  pmg_status st = check_level(h->c, level);
  if (st) return st;
  const std::vector<double>& xyh = h->c.xy_host[level];
  memcpy(xy, xyh.data(), xyh.size() * 8);
  return PMG_OK;
}

pmg_status pmg_set_state(pmg_ctx* h, int level, const double* q, int on_device) {
  if (!h || !q) return fail(PMG_EINVAL, "null argument");
  Ctx& c = h->c;
  pmg_status st = check_level(c, level);
  if (st) return st;
  PMG_CK(state_in(c, c.lev[level].q, q, c.lev[level], on_device));
  PMG_CK_LAUNCH();
  PMG_CK(cudaStreamSynchronize(c.stream));
  if (level == 0) c.F0_valid = false;
  return PMG_OK;
}

// ------------------------------------------------------- checkpoint / restore
// File: 72-byte header (magic, version, E, P of every level, geometry order,
// a hash of the mesh and of the discretisation settings), then the finest
// state as stored on the device (variable-major FP64, pressure relative to
// p_gauge), so that a restored run repeats the next step bit for bit.
namespace {
constexpr char kCkptMagic[8] = {'P', 'M', 'G', 'F', 'R', 'C', 'K', '1'};
struct CkptHeader {
  char magic[8];
  int32_t version, n_elem, geom_order, n_levels;
  int32_t P[8];
  uint64_t mesh_hash, config_hash;
};
static_assert(sizeof(CkptHeader) == 72, "checkpoint header layout");

uint64_t fnv1a(uint64_t h, const void* data, size_t n) {
  const unsigned char* b = (const unsigned char*)data;
  for (size_t i = 0; i < n; ++i) { h ^= b[i]; h *= 1099511628211ull; }
  return h;
}

uint64_t mesh_hash(const Ctx& c) {
  uint64_t h = 1469598103934665603ull;
  h = fnv1a(h, c.mesh.nodes.data(), c.mesh.nodes.size() * sizeof(double));
  return fnv1a(h, c.mesh.nbr.data(), c.mesh.nbr.size() * sizeof(int));
}

uint64_t config_hash(const Ctx& c) {
  // the settings that define the discrete system (not the solver schedule)
  const pmg_config& g = c.cfg;
  double d[8 + 4] = {g.gamma, g.Ma_inf, g.kappa, (double)g.cutoff, g.p_gauge, g.mu, g.Pr, (double)g.n_levels,
                     g.res_scale[0], g.res_scale[1], g.res_scale[2], g.res_scale[3]};
  uint64_t h = fnv1a(1469598103934665603ull, d, sizeof(d));
  return fnv1a(h, g.P, sizeof(g.P));
}

CkptHeader make_header(const Ctx& c) {
  CkptHeader hd;
  memset(&hd, 0, sizeof(hd));
  memcpy(hd.magic, kCkptMagic, 8);
  hd.version = 1;
  hd.n_elem = c.E;
  hd.geom_order = c.mesh.Ng;
  hd.n_levels = c.cfg.n_levels;
  for (int l = 0; l < c.cfg.n_levels; ++l) hd.P[l] = c.cfg.P[l];
  hd.mesh_hash = mesh_hash(c);
  hd.config_hash = config_hash(c);
  return hd;
}
}  // namespace

pmg_status pmg_dtau_min(pmg_ctx* h, double* out) {
  if (!h || !out) return fail(PMG_EINVAL, "null argument");
  Ctx& c = h->c;
  if (!c.mesh_ready) return fail(PMG_ESTATE, "no mesh uploaded");
  return compute_dtau_min(c, out);
}

pmg_status pmg_checkpoint(pmg_ctx* h, const char* path) {
  if (!h || !path) return fail(PMG_EINVAL, "null argument");
  Ctx& c = h->c;
  if (!c.mesh_ready) return fail(PMG_ESTATE, "no mesh uploaded");
  const LevelDev& L = c.lev[0];
  std::vector<double> buf(L.tot);
  PMG_CK(cudaMemcpyAsync(buf.data(), L.q, L.tot * 8, cudaMemcpyDeviceToHost, c.stream));
  PMG_CK(cudaStreamSynchronize(c.stream));
  CkptHeader hd = make_header(c);
  FILE* f = fopen(path, "wb");
  if (!f) return fail(PMG_EINVAL, std::string("cannot open ") + path + " for writing");
  bool ok = fwrite(&hd, sizeof(hd), 1, f) == 1 && fwrite(buf.data(), 8, buf.size(), f) == buf.size();
  ok = (fclose(f) == 0) && ok;
  if (!ok) return fail(PMG_EINVAL, std::string("write failed: ") + path);
  return PMG_OK;
}

pmg_status pmg_restore(pmg_ctx* h, const char* path) {
  if (!h || !path) return fail(PMG_EINVAL, "null argument");
  Ctx& c = h->c;
  if (!c.mesh_ready) return fail(PMG_ESTATE, "no mesh uploaded");
  LevelDev& L = c.lev[0];
  FILE* f = fopen(path, "rb");
  if (!f) return fail(PMG_EINVAL, std::string("cannot open ") + path);
  CkptHeader hd;
  std::vector<double> buf(L.tot);
  bool ok = fread(&hd, sizeof(hd), 1, f) == 1;
  ok = ok && fread(buf.data(), 8, buf.size(), f) == buf.size();
  char extra;
  ok = ok && fread(&extra, 1, 1, f) == 0;   // nothing after the state
  fclose(f);
  if (!ok) return fail(PMG_EINVAL, std::string("not a checkpoint of this size: ") + path);
  CkptHeader want = make_header(c);
  if (memcmp(hd.magic, kCkptMagic, 8) != 0 || hd.version != 1)
    return fail(PMG_EINVAL, std::string("not a pmgfr checkpoint: ") + path);
  if (hd.n_elem != want.n_elem || hd.geom_order != want.geom_order || hd.n_levels != want.n_levels ||
      memcmp(hd.P, want.P, sizeof(hd.P)) != 0 || hd.mesh_hash != want.mesh_hash)
    return fail(PMG_EINVAL, "checkpoint is for another mesh or P hierarchy");
  if (hd.config_hash != want.config_hash) return fail(PMG_EINVAL, "checkpoint is for other discretisation settings");
  PMG_CK(cudaMemcpyAsync(L.q, buf.data(), L.tot * 8, cudaMemcpyHostToDevice, c.stream));
  PMG_CK(cudaStreamSynchronize(c.stream));
  c.F0_valid = false;
  return PMG_OK;
}

pmg_status pmg_get_state(pmg_ctx* h, int level, double* q, int on_device) {
  if (!h || !q) return fail(PMG_EINVAL, "null argument");
  Ctx& c = h->c;
  pmg_status st = check_level(c, level);
  if (st) return st;
  const LevelDev& L = c.lev[level];
  const bool direct = on_device && own_memory(c, q, L.tot);
  launch_copy_shift(L.tot / c.nv, L.tot, c.ph.p_ref, L.q, direct ? q : c.d_tmp0, c.stream);
  PMG_CK_LAUNCH();
  if (!direct) PMG_CK(copy_out(c, q, c.d_tmp0, L.tot, on_device));
  else PMG_CK(cudaStreamSynchronize(c.stream));
  return PMG_OK;
}

pmg_status pmg_residual(pmg_ctx* h, int level, const double* q, double* R, int on_device) {
  if (!h || !q || !R) return fail(PMG_EINVAL, "null argument");
  Ctx& c = h->c;
  pmg_status st = check_level(c, level);
  if (st) return st;
  LevelDev& L = c.lev[level];
  PMG_CK(state_in(c, c.d_tmp0, q, L, on_device));
  const double* qd = c.d_tmp0;
  double* Rd = on_device ? R : c.d_tmp1;
  launch_face_flux(c, L, qd, c.stream);
  launch_volume(c, L, level, qd, Rd, RES_PURE, 0.0, nullptr, nullptr, nullptr, nullptr, nullptr, c.stream);
  add_gauge_constant(c, level, Rd);
  PMG_CK_LAUNCH();
  if (!on_device) PMG_CK(copy_out(c, R, Rd, L.tot, 0));
  else PMG_CK(cudaStreamSynchronize(c.stream));
  return PMG_OK;
}

}  // extern "C"

// ----------------------------------------------------- allocation-free residual
// Scratch of pmg_residual_static: one file-scope device array shared by every
// call on a device (the gauge-shifted copy of the input state followed by the
// common face fluxes).  Host code never touches it by name as an address: the
// device address is looked up on every call with cudaGetSymbolAddress (which
// allocates nothing), so a context torn down and created again in the same
// process never sees a stale address.
static constexpr size_t kStaticScratchDoubles = (size_t)1 << 21;   // 16 MiB
static __device__ __align__(256) double g_static_scratch[kStaticScratchDoubles];

static cudaError_t static_scratch_address(double** out) {
  void* p = nullptr;
  cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
  *out = (double*)p;
  return e;
}

extern "C" {

pmg_status pmg_residual_static(pmg_ctx* h, int level, const double* q, double* R) {
  if (!h || !q || !R) return fail(PMG_EINVAL, "null argument");
  Ctx& c = h->c;
  pmg_status st = check_level(c, level);
  if (st) return st;
  LevelDev L = c.lev[level];   // shallow copy: only the scratch slots are redirected
  const bool visc = c.ph.mu > 0.0;
  const size_t n_state = L.tot, n_face = (size_t)c.nv * c.E * c.nfc * L.NF;
  const size_t n_grad = (size_t)(c.dim == 3 ? 12 : 6) * c.E * L.N;
  const size_t n_jump = c.dim == 3 ? (size_t)4 * c.E * 6 * L.NF : (size_t)3 * c.E * 4 * L.n1;
  const size_t n_visc = visc ? n_grad + n_jump : 0;
  if (n_state + n_face + n_visc > kStaticScratchDoubles)
    return fail(PMG_EINVAL, "pmg_residual_static: level needs " + std::to_string(n_state + n_face + n_visc) +
                                " scratch doubles, the static scratch holds " +
                                std::to_string(kStaticScratchDoubles));
  int cur = -1;
  PMG_CK(cudaGetDevice(&cur));
  if (cur != c.device) return fail(PMG_EINVAL, "pmg_residual_static: make the context's device current first");
  double* scratch = nullptr;
  PMG_CK(static_scratch_address(&scratch));
  double* qs = scratch;
  L.Fcom = scratch + n_state;
  if (visc) {   // broken gradients and face jumps of the viscous terms
    L.Gb = scratch + n_state + n_face;
    L.Qj = L.Gb + n_grad;
  }
  PMG_CK(state_in(c, qs, q, L, 1));
  launch_face_flux(c, L, qs, c.stream);
  launch_volume(c, L, level, qs, R, RES_PURE, 0.0, nullptr, nullptr, nullptr, nullptr, nullptr, c.stream);
  add_gauge_constant(c, level, R);
  PMG_CK_LAUNCH();
  PMG_CK(cudaStreamSynchronize(c.stream));
  return PMG_OK;
}

pmg_status pmg_set_stage(pmg_ctx* h, const double* src, double omega_dt, int on_device) {
  if (!h || !src) return fail(PMG_EINVAL, "null argument");
  Ctx& c = h->c;
  if (!c.mesh_ready) return fail(PMG_ESTATE, "mesh not uploaded");
  if (!(omega_dt > 0.0)) return fail(PMG_EINVAL, "omega_dt must be positive");
  PMG_CK(copy_in(c, c.src, src, c.lev[0].tot, on_device));
  PMG_CK(cudaStreamSynchronize(c.stream));
  c.omega_dt = omega_dt;
  c.stage_ready = true;
  c.split_stage = false;
  c.F0_valid = false;
  return PMG_OK;
}

pmg_status pmg_stage_residual(pmg_ctx* h, int level, const double* q, double* F, int on_device) {
  if (!h || !q || !F) return fail(PMG_EINVAL, "null argument");
  Ctx& c = h->c;
  pmg_status st = check_level(c, level);
  if (st) return st;
  if (!c.stage_ready) return fail(PMG_ESTATE, "stage data not set");
  LevelDev& L = c.lev[level];
  PMG_CK(state_in(c, c.d_tmp0, q, L, on_device));
  const double* qd = c.d_tmp0;
  double* Fd = on_device ? F : c.d_tmp1;
  launch_face_flux(c, L, qd, c.stream);
  launch_volume(c, L, level, qd, Fd, RES_STAGEF, 1.0 / c.omega_dt, level == 0 ? c.src : nullptr, nullptr, nullptr,
                nullptr, nullptr, c.stream);
  add_gauge_constant(c, level, Fd);
  PMG_CK_LAUNCH();
  if (!on_device) PMG_CK(copy_out(c, F, Fd, L.tot, 0));
  else PMG_CK(cudaStreamSynchronize(c.stream));
  return PMG_OK;
}

pmg_status pmg_assemble_blocks(pmg_ctx* h, int level, double dtau) {
  if (!h) return fail(PMG_EINVAL, "null argument");
  Ctx& c = h->c;
  if (!c.mesh_ready) return fail(PMG_ESTATE, "mesh not uploaded");
  if (level < -1 || level >= c.cfg.n_levels) return fail(PMG_EINVAL, "level out of range");
  if (!(dtau > 0.0)) return fail(PMG_EINVAL, "dtau must be positive");
  pmg_status st = set_dtau(c, dtau);
  if (st) return st;
  for (int l = 0; l < c.cfg.n_levels; ++l) {
    if (level >= 0 && l != level) continue;
    launch_assemble(c, c.lev[l], c.lev[l].q, c.d_dtau, 1.0 / c.omega_dt, c.stream);
    c.lev[l].assembled = true;
    c.lev[l].factored = false;
  }
  PMG_CK_LAUNCH();
  PMG_CK(cudaStreamSynchronize(c.stream));
  return PMG_OK;
}

pmg_status pmg_get_blocks(pmg_ctx* h, int level, double* D, int on_device) {
  if (!h || !D) return fail(PMG_EINVAL, "null argument");
  Ctx& c = h->c;
  pmg_status st = check_level(c, level);
  if (st) return st;
  if (!c.lev[level].assembled) return fail(PMG_ESTATE, "blocks not assembled");
  const LevelDev& L = c.lev[level];
  PMG_CK(copy_out(c, D, L.Dfull, (size_t)c.E * L.n * L.n, on_device));
  return PMG_OK;
}

pmg_status pmg_set_blocks(pmg_ctx* h, int level, const double* D, int on_device) {
  if (!h || !D) return fail(PMG_EINVAL, "null argument");
  Ctx& c = h->c;
  pmg_status st = check_level(c, level);
  if (st) return st;
  LevelDev& L = c.lev[level];
  PMG_CK(copy_in(c, L.Dfull, D, (size_t)c.E * L.n * L.n, on_device));
  PMG_CK(cudaStreamSynchronize(c.stream));
  L.assembled = true;
  L.factored = false;
  return PMG_OK;
}

pmg_status pmg_factor_blocks(pmg_ctx* h, int level) {
  if (!h) return fail(PMG_EINVAL, "null argument");
  Ctx& c = h->c;
  if (!c.mesh_ready) return fail(PMG_ESTATE, "mesh not uploaded");
  if (level < -1 || level >= c.cfg.n_levels) return fail(PMG_EINVAL, "level out of range");
  for (int l = 0; l < c.cfg.n_levels; ++l) {
    if (level >= 0 && l != level) continue;
    if (!c.lev[l].assembled) return fail(PMG_ESTATE, "blocks not assembled");
    launch_factor(c, c.lev[l], l, c.cfg.block_prec, c.d_flag, c.stream);
    c.lev[l].factored = true;
  }
  PMG_CK_LAUNCH();
  return check_singular(c);
}

pmg_status pmg_apply_blocks(pmg_ctx* h, int level, const double* r, double* x, int on_device) {
  if (!h || !r || !x) return fail(PMG_EINVAL, "null argument");
  Ctx& c = h->c;
  pmg_status st = check_level(c, level);
  if (st) return st;
  LevelDev& L = c.lev[level];
  if (!L.factored) return fail(PMG_ESTATE, "blocks not factored");
  const double* rd = r;
  double* xd = x;
  if (!on_device) {
    PMG_CK(copy_in(c, c.d_tmp0, r, L.tot, 0));
    rd = c.d_tmp0;
    xd = c.d_tmp1;
  }
  launch_apply(c, L, c.cfg.block_prec, rd, xd, 0, c.stream);
  PMG_CK_LAUNCH();
  if (!on_device) PMG_CK(copy_out(c, x, xd, L.tot, 0));
  else PMG_CK(cudaStreamSynchronize(c.stream));
  return PMG_OK;
}

pmg_status pmg_restrict(pmg_ctx* h, int lf, const double* qf, double* qc, int on_device) {
  if (!h || !qf || !qc) return fail(PMG_EINVAL, "null argument");
  Ctx& c = h->c;
  pmg_status st = check_level(c, lf);
  if (st) return st;
  if (lf + 1 >= c.cfg.n_levels) return fail(PMG_EINVAL, "no coarser level");
  LevelDev& F = c.lev[lf];
  LevelDev& C = c.lev[lf + 1];
  const double* in = qf;
  double* out = qc;
  if (!on_device) {
    PMG_CK(copy_in(c, c.d_tmp0, qf, F.tot, 0));
    in = c.d_tmp0;
    out = c.d_tmp1;
  }
  launch_restrict(c, F, C, c.xfer[lf], in, out, c.stream);
  PMG_CK_LAUNCH();
  if (!on_device) PMG_CK(copy_out(c, qc, out, C.tot, 0));
  else PMG_CK(cudaStreamSynchronize(c.stream));
  return PMG_OK;
}

pmg_status pmg_prolong(pmg_ctx* h, int lf, const double* qc, double* qf, int on_device) {
  if (!h || !qf || !qc) return fail(PMG_EINVAL, "null argument");
  Ctx& c = h->c;
  pmg_status st = check_level(c, lf);
  if (st) return st;
  if (lf + 1 >= c.cfg.n_levels) return fail(PMG_EINVAL, "no coarser level");
  LevelDev& F = c.lev[lf];
  LevelDev& C = c.lev[lf + 1];
  const double* in = qc;
  double* out = qf;
  if (!on_device) {
    PMG_CK(copy_in(c, c.d_tmp0, qc, C.tot, 0));
    in = c.d_tmp0;
    out = c.d_tmp1;
  }
  launch_prolong(c, F, C, c.xfer[lf], in, out, c.stream);
  PMG_CK_LAUNCH();
  if (!on_device) PMG_CK(copy_out(c, qf, out, F.tot, 0));
  else PMG_CK(cudaStreamSynchronize(c.stream));
  return PMG_OK;
}

pmg_status pmg_vcycle(pmg_ctx* h, double dtau, int refresh, double* res_norm_out) {
  if (!h) return fail(PMG_EINVAL, "null argument");
  Ctx& c = h->c;
  if (!c.mesh_ready) return fail(PMG_ESTATE, "mesh not uploaded");
  if (!c.stage_ready) return fail(PMG_ESTATE, "stage data not set");
  if (!(dtau > 0.0)) return fail(PMG_EINVAL, "dtau must be positive");
  if (!refresh)
    for (int l = 0; l < c.cfg.n_levels; ++l)
      if (!c.lev[l].factored) return fail(PMG_ESTATE, "smoother not built: call with refresh = 1 first");
  if (!c.F0_valid) {
    system_residual(c, 0, true);
    c.F0_valid = true;
  }
  double nm;
  pmg_status st = read_norm(c, &nm);
  if (st) return st;
  if (res_norm_out) *res_norm_out = nm;
  st = set_dtau(c, dtau);
  if (st) return st;
  st = launch_vcycle(c, refresh != 0);
  if (st) return st;
  if (refresh) {
    st = check_singular(c);
    if (st) return st;
  }
  return check_wait_flag(c);
}

pmg_status pmg_stage_solve(pmg_ctx* h, int* iters, double* drop) {
  if (!h) return fail(PMG_EINVAL, "null argument");
  Ctx& c = h->c;
  if (!c.mesh_ready) return fail(PMG_ESTATE, "mesh not uploaded");
  if (!c.stage_ready) return fail(PMG_ESTATE, "stage data not set");
  c.hist_norm.clear();
  c.hist_dtau.clear();
  return stage_solve(c, iters, drop, nullptr);
}

pmg_status pmg_set_stage_solver(pmg_ctx* h, int solver, const pmg_nk_options* opts) {
  if (!h) return fail(PMG_EINVAL, "null argument");
  Ctx& c = h->c;
  if (solver != PMG_STAGE_PTC && solver != PMG_STAGE_NK) return fail(PMG_EINVAL, "unknown stage solver");
  const pmg_nk_options o = nk_defaults(c, opts);
  if (o.krylov_dim > 64) return fail(PMG_EINVAL, "krylov_dim must be at most 64");
  if (o.precond != PMG_NK_PC_BLOCK && o.precond != PMG_NK_PC_VCYCLE)
    return fail(PMG_EINVAL, "unknown Newton-Krylov preconditioner");
  if (!(o.eta < 1.0) || !std::isfinite(o.dtau_pc) || !std::isfinite(o.delta0) || !(o.delta0 < 1.0) ||
      !std::isfinite(o.pc_eps) || !std::isfinite(o.max_update) || !std::isfinite(o.ptc_dtau))
    return fail(PMG_EINVAL,
                "Newton-Krylov options out of range (eta < 1, delta0 < 1, finite dtau_pc and ptc_dtau)");
  for (int v = 0; v < 5; ++v)
    if (!std::isfinite(o.state_scale[v])) return fail(PMG_EINVAL, "state_scale must be finite");
  c.stage_solver = solver;
  c.nk = o;
  return PMG_OK;
}

pmg_status pmg_nk_stats_read(pmg_ctx* h, pmg_nk_stats* out, int reset) {
  if (!h) return fail(PMG_EINVAL, "null argument");
  Ctx& c = h->c;
  if (out) {
    out->newton = c.nk_count[0];
    out->krylov = c.nk_count[1];
    out->vcycles = c.nk_count[2];
    out->residuals = c.nk_count[3];
  }
  if (reset)
    for (long long& v : c.nk_count) v = 0;
  return PMG_OK;
}

// ------------------------------------------------------------- autotuner
// Times the smoothing of every level the fused and tiled coarse-level kernels
// can serve under each candidate schedule and keeps the fastest: the split
// face and volume launches (P = 1), one fused launch per sweep, or tiles of
// 16, 32 or 64 core elements with 2, 3 or 4 sweeps per launch.  Each
// candidate runs the level's n_smooth sweeps once untimed and `reps` times
// between events on the context's stream, on the level's current data.
pmg_status pmg_autotune(pmg_ctx* h, int reps, const char* cache_path, pmg_tune_report* rep) {
  if (!h) return fail(PMG_EINVAL, "null argument");
  Ctx& c = h->c;
  if (!c.mesh_ready) return fail(PMG_ESTATE, "mesh not uploaded");
  if (!c.stage_ready) return fail(PMG_ESTATE, "stage data not set");
  for (int l = 0; l < c.cfg.n_levels; ++l)
    if (!c.lev[l].factored) return fail(PMG_ESTATE, "smoother not built: run a V-cycle with refresh = 1 first");
  if (reps < 1) reps = 1;
  pmg_tune_report local;
  memset(&local, 0, sizeof(local));
  local.n_levels = c.cfg.n_levels;
  int dev_sms = 0;
  cudaDeviceGetAttribute(&dev_sms, cudaDevAttrMultiProcessorCount, c.device);
  // cache: lines "P E n_smooth block_prec sms fused core depth"
  std::vector<std::array<int, 8>> cache;
  if (cache_path) {
    if (FILE* f = fopen(cache_path, "r")) {
      std::array<int, 8> r;
      while (fscanf(f, "%d %d %d %d %d %d %d %d", &r[0], &r[1], &r[2], &r[3], &r[4], &r[5], &r[6], &r[7]) == 8)
        cache.push_back(r);
      fclose(f);
    }
  }
  cudaEvent_t e0, e1;
  PMG_CK(cudaEventCreate(&e0));
  PMG_CK(cudaEventCreate(&e1));
  struct Cand { int fused, core, depth; };
  pmg_status result = PMG_OK;
  for (int l = 0; l < c.cfg.n_levels && result == PMG_OK; ++l) {
    LevelDev& L = c.lev[l];
    local.fused[l] = L.fused ? 1 : 0;
    local.tile_core[l] = L.tiled ? L.tile_core : 0;
    local.tile_depth[l] = L.tiled ? L.tile_depth : 0;
    if (!L.tileable) continue;
    const int n = c.cfg.n_smooth[l];
    const std::array<int, 5> key{L.P, c.E, n, c.cfg.block_prec, dev_sms};
    const int was_fused = L.fused, was_core = L.tiled ? L.tile_core : 0, was_depth = L.tiled ? L.tile_depth : 0;
    std::vector<Cand> cands;
    bool cached = false;
    for (const auto& r : cache)
      if (r[0] == key[0] && r[1] == key[1] && r[2] == key[2] && r[3] == key[3] && r[4] == key[4]) {
        cands = {{r[5], r[6], r[7]}};
        cached = true;
      }
    if (!cached) {
      if (L.P >= 1) cands.push_back({0, 0, 0});
      cands.push_back({1, 0, 0});
      for (int core : {16, 32, 64})
        for (int depth : {2, 3, 4}) cands.push_back({1, core, depth});
    }
    double best = 1e300, before = 0.0;
    Cand pick{was_fused, was_core, was_depth};
    for (const Cand& cd : cands) {
      L.fused = cd.fused != 0;
      if (set_level_tiles(c, L, cd.core, cd.fused ? cd.depth : 0) != PMG_OK) continue;   // does not fit
      restore_buffer(c, l, sweeps(c, l, n, false, false, false));
      PMG_CK(cudaEventRecord(e0, c.stream));
      for (int r = 0; r < reps; ++r) restore_buffer(c, l, sweeps(c, l, n, false, false, false));
      PMG_CK(cudaEventRecord(e1, c.stream));
      cudaError_t le = cudaGetLastError();
      if (le != cudaSuccess) { result = fail(PMG_ECUDA, std::string("autotune: ") + cudaGetErrorString(le)); break; }
      PMG_CK(cudaEventSynchronize(e1));
      float ms = 0.f;
      PMG_CK(cudaEventElapsedTime(&ms, e0, e1));
      const double us = 1000.0 * ms / (reps * n);
      if (cd.fused == was_fused && cd.core == was_core && (cd.fused ? cd.depth : 0) == was_depth) before = us;
      if (us < best) { best = us; pick = cd; }
      ++local.candidates[l];
    }
    if (result != PMG_OK) break;
    // keep the schedule in place unless another beats it by more than 2%:
    // timings of equivalent schedules differ by noise, and a change of
    // schedule changes the launch sequence for nothing
    if (!cached && before > 0.0 && best > 0.98 * before) {
      pick = Cand{was_fused, was_core, was_depth};
      best = before;
    }
    L.fused = pick.fused != 0;
    pmg_status st = set_level_tiles(c, L, pick.core, pick.fused ? pick.depth : 0);
    if (st) { result = st; break; }
    local.fused[l] = pick.fused;
    local.tile_core[l] = L.tiled ? pick.core : 0;
    local.tile_depth[l] = L.tiled ? pick.depth : 0;
    local.us_per_sweep[l] = best;
    local.us_per_sweep_before[l] = before;
    if (cache_path && !cached) {
      if (FILE* f = fopen(cache_path, "a")) {
        fprintf(f, "%d %d %d %d %d %d %d %d\n", key[0], key[1], key[2], key[3], key[4], pick.fused, local.tile_core[l],
                local.tile_depth[l]);
        fclose(f);
      }
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  // the V-cycle launch sequence changed: captured graphs are rebuilt on demand
  for (int g = 0; g < 2; ++g)
    if (c.graph[g]) { cudaGraphExecDestroy(c.graph[g]); c.graph[g] = nullptr; }
  if (c.loop_exec) { cudaGraphExecDestroy(c.loop_exec); c.loop_exec = nullptr; }
  c.F0_valid = false;
  if (rep) *rep = local;
  return result;
}

pmg_status pmg_profile(pmg_ctx* h, int enable) {
  if (!h) return fail(PMG_EINVAL, "null argument");
  Ctx& c = h->c;
  Profiler& p = c.prof;
  PMG_CK(cudaStreamSynchronize(c.stream));
  if (enable && p.ev.empty()) {
    const int pairs = 4096;
    p.ev.resize(2 * pairs);
    p.tag.resize(pairs);
    for (auto& e : p.ev) PMG_CK(cudaEventCreate(&e));
  }
  if (!enable && p.on) prof_harvest(c);
  p.on = enable != 0;
  if (enable) {
    p.used = 0;
    memset(p.ms, 0, sizeof(p.ms));
    memset(p.count, 0, sizeof(p.count));
  }
  return PMG_OK;
}

pmg_status pmg_profile_read(pmg_ctx* h, double* ms, long long* counts) {
  if (!h || !ms || !counts) return fail(PMG_EINVAL, "null argument");
  Ctx& c = h->c;
  PMG_CK(cudaStreamSynchronize(c.stream));
  prof_harvest(c);
  for (int k = 0; k < K_COUNT; ++k)
    for (int l = 0; l < kMaxLevels; ++l) {
      ms[k * kMaxLevels + l] = c.prof.ms[k][l];
      counts[k * kMaxLevels + l] = c.prof.count[k][l];
    }
  return PMG_OK;
}

pmg_status pmg_stage_history(pmg_ctx* h, double* norms, double* dtau, int max_count, int* count) {
  if (!h || !count) return fail(PMG_EINVAL, "null argument");
  Ctx& c = h->c;
  int n = (int)c.hist_norm.size();
  *count = n;
  for (int i = 0; i < n && i < max_count; ++i) {
    if (norms) norms[i] = c.hist_norm[i];
    if (dtau) dtau[i] = c.hist_dtau[i];
  }
  return PMG_OK;
}

pmg_status pmg_esdirk_step(pmg_ctx* h, double dt, pmg_step_stats* stats) {
  if (!h) return fail(PMG_EINVAL, "null argument");
  Ctx& c = h->c;
  if (!c.mesh_ready) return fail(PMG_ESTATE, "mesh not uploaded");
  if (!(dt > 0.0)) return fail(PMG_EINVAL, "dt must be positive");
  pmg_step_stats local;
  memset(&local, 0, sizeof(local));
  cudaEvent_t ev0, ev1;
  PMG_CK(cudaEventCreate(&ev0));
  PMG_CK(cudaEventCreate(&ev1));
  PMG_CK(cudaEventRecord(ev0, c.stream));
  LevelDev& L0 = c.lev[0];
  const int N0 = L0.N;
  c.hist_norm.clear();
  c.hist_dtau.clear();
  PMG_CK(cudaMemcpyAsync(c.qn, L0.q, L0.tot * 8, cudaMemcpyDeviceToDevice, c.stream));
  {
    ProfScope ps(c, K_FACE, 0);
    launch_face_flux(c, L0, L0.q, c.stream);
  }
  {
    ProfScope ps(c, K_VOLUME, 0);
    launch_volume(c, L0, 0, L0.q, c.Rst[0], RES_PURE, 0.0, nullptr, nullptr, nullptr, nullptr, nullptr, c.stream);
  }
  PMG_CK_LAUNCH();
  const double omega = c.A[1][1];
  c.omega_dt = omega * dt;
  c.stage_ready = true;
  c.split_stage = true;   // level-0 system uses q_c(q) - q_c(q^n) and src = sum_j a_ij R^j / omega
  pmg_status st = PMG_OK;
  for (int i = 1; i < c.stages; ++i) {
    double a[6];
    for (int j = 0; j < i; ++j) a[j] = c.A[i][j];
    {
      ProfScope ps(c, K_STAGE, 0);
      launch_stage_src(c, N0, nullptr, c.Rst, a, i, dt, 1.0 / c.omega_dt, c.src, c.stream);
    }
    c.F0_valid = false;
    int it = 0;
    double dr = 0.0;
    int vc = -1;
    st = stage_solve(c, &it, &dr, &local.n_refresh, &vc);
    local.pseudo_iters[i - 1] = it;
    local.res_drop[i - 1] = dr;
    local.n_vcycles += vc >= 0 ? vc : it;
    if (st) break;
    {
      ProfScope ps(c, K_FACE, 0);
      launch_face_flux(c, L0, L0.q, c.stream);
    }
    {
      ProfScope ps(c, K_VOLUME, 0);
      launch_volume(c, L0, 0, L0.q, c.Rst[i], RES_PURE, 0.0, nullptr, nullptr, nullptr, nullptr, nullptr, c.stream);
    }
  }
  if (st == PMG_OK) {
    ProfScope ps(c, K_STAGE, 0);
    launch_bsum_update(c, N0, c.qn, c.Rst, c.b, c.stages, dt, L0.q, c.stream);
    PMG_CK_LAUNCH();
  }
  c.F0_valid = false;
  PMG_CK(cudaEventRecord(ev1, c.stream));
  PMG_CK(cudaEventSynchronize(ev1));
  float ms = 0.f;
  cudaEventElapsedTime(&ms, ev0, ev1);
  local.ms_total = ms;
  if (c.prof.on) prof_harvest(c);
  cudaEventDestroy(ev0);
  cudaEventDestroy(ev1);
  if (stats) *stats = local;
  return st;
}

}  // extern "C"
