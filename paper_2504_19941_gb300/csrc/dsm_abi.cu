// dsm_abi.cu -- the extern "C" entry points declared in include/dsm.h.
// Host code only: argument checks, workspace carving, dispatch to the typed
// kernels, error latching.  No device memory is ever allocated here.
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <new>
#include <vector>

#include "dsm_em.cuh"
#include "dsm_lb_impl.cuh"
#include "dsm_tmap.cuh"
#include "dsm_trace.cuh"

using namespace dsm;

struct dsm_lattice {
  dsm_params prm;
  double kappa[3];
  LBTable tab;
  int kind, q;
  long long N, pitch;
  char *ws;
  size_t ws_bytes;
  void *f[2], *g[2];
  float *g0[2];
  void *Cb[2];   // Cb[cur]: C of the state's last collision; Cb[cur ^ 1]: moments output
  void *M;       // g held as g_eq: A, u_x, u_y, u_z planes
  void *C1;
  unsigned char *mask;
  double *partials, *obs;
  int *err;
  long long obs_blocks;
  int cur;
  cudaStream_t stream;
  long long step;
  bool has_solid, has_fluid, latched, moments_ready;
  int g_form;      // DSM_G_AUTO or DSM_G_POPULATIONS
  bool eq;         // the fused pass stores g as g_eq (tau_g = 1 and DSM_G_AUTO)
  bool g_implicit; // the current g are held as g_eq
  StepParams sp;
  // single-pass step (dsm_zstep.cuh): padded quads (A, C, u_x, u_y) and u_z,
  // two buffers, and padded C1; zc: the buffer holding the current state while
  // zpacked
  bool zok;        // the workspace has the padded buffers (D3Q19, nx % 32, ny % 8, tau_g = 1, periodic)
  bool zpacked;    // the current g_eq state lives in the padded buffers
  bool zmaps_ok;   // maps[] encoded
  int zc, nxp, nyp;
  void *Qz[2], *Uz[2], *C1z;
  ZMaps maps[2];   // maps[b]: read the padded state of buffer b (and C1)
  int step_form;   // DSM_STEP_AUTO or DSM_STEP_TWO_PASS
  int zrun;        // planes per block of the single-pass step (0: automatic)
  int zrun_auto;
  // step on moments (dsm_mom.cuh): mok, the parameters allow it; mom, the
  // current state is held as moments (buffer mc); mcp, Cb[0] holds the C of its
  // next step, mpk: the other buffer holds that step (made for reads); mstat, the
  // frozen solid's data is made; mfit, the canonical
  // state is the result of a step with every relaxation time 1, so moments
  // represent it; mstepped, mom and stepped since set_fluid
  bool mok, mom, mcp, mpk, mstat, mfit, mstepped;
  int mc, mzrun;
  // single-pass step of D2Q9 (dsm_tile2.cuh): tok, the parameters allow it; tp,
  // the state is f[cur] and the quads in g[cur ^ 1]; tcan, the canonical copy
  // of that state (made for reads, which leave the quads valid) is up to date
  bool tok, tp, tcan;
  // observables ring (dsm_set_observables_ring): caller-owned device records,
  // one appended by dsm_step after each step that is a multiple of ring_every
  double *ring = nullptr;
  int ring_cap = 0;
  long long ring_every = 0, ring_count = 0;
};

namespace {


dsm_status cuda_status(cudaError_t e) { return e == cudaSuccess ? DSM_OK : DSM_E_CUDA; }

// Polls of a bounded device wait before it gives up (dsm_set_wait_limit);
// 0: each kernel's default.
unsigned long long g_wait_limit = 0;

bool lb_table_for(int kind, int precision, LBTable *t) {
  switch (precision) {
    case DSM_F64: *t = lb_table_f64(kind); return true;
    case DSM_F32: *t = lb_table_f32(kind); return true;
    case DSM_BF16_STORE: *t = lb_table_bf16(kind); return true;
    case DSM_F16_STORE: *t = lb_table_f16(kind); return true;
    default: return false;
  }
}

// Tensions -> kappa (Sec. II.A, Eq. [frozen:kappa]); tension_mode 1 first
// applies Young's relation gamma_13 = gamma_12 + gamma_23 cos(theta).
dsm_status kappa_of(const dsm_params *p, double k[3]) {
  if (!(p->alpha > 0.0)) return DSM_E_INVAL;
  double g12 = p->g12, g23 = p->g23, g13 = p->g13;
  if (p->tension_mode == 1) g13 = g12 + g23 * cos(p->theta_deg * 3.14159265358979323846 / 180.0);
  else if (p->tension_mode != 0) return DSM_E_INVAL;
  k[0] = 3.0 / p->alpha * (g12 + g13 - g23);
  k[1] = 3.0 / p->alpha * (g12 - g13 + g23);
  k[2] = 3.0 / p->alpha * (-g12 + g13 + g23);
  if (!(k[1] > 0.0) || !(k[2] > 0.0)) return DSM_E_INVAL;
  return DSM_OK;
}

dsm_status check_params(const dsm_params *p) {
  if (!p) return DSM_E_INVAL;
  if (p->lattice != DSM_D2Q9 && p->lattice != DSM_D3Q19) return DSM_E_INVAL;
  if (p->nx < 1 || p->ny < 1 || p->nz < 1) return DSM_E_INVAL;
  if (p->lattice == DSM_D2Q9 && p->nz != 1) return DSM_E_INVAL;
  if ((long long)p->nx * p->ny * p->nz >= (1ll << 31)) return DSM_E_INVAL;
  if (p->precision < DSM_F64 || p->precision > DSM_F16_STORE) return DSM_E_INVAL;
  if (!(p->tau2 > 0.5) || !(p->tau3 > 0.5) || !(p->tau_g > 0.5)) return DSM_E_INVAL;
  if (!(p->rho2 > 0.0) || !(p->rho3 > 0.0)) return DSM_E_INVAL;
  if (p->alpha_s < 0.0) return DSM_E_INVAL;
  if (!faces_valid(p)) return DSM_E_INVAL;
  double k[3];
  return kappa_of(p, k);
}

struct Layout {
  size_t f[2], g[2], g0[2], C[2], M, C1, mask, partials, obs, err, Qz[2], Uz[2], C1z, total;
};

// The single-pass step applies to D3Q19 lattices at least one 32 x 8 tile wide
// (the last tiles may be ragged), with tau_g = 1 (g held as g_eq) and periodic
// faces.
bool z_eligible(const dsm_params *p) {
  if (p->lattice != DSM_D3Q19 || p->tau_g != 1.0 || has_walls(p)) return false;
  return z_tiles(p->nx, p->ny);
}
long long z_padded_nodes(const dsm_params *p) {
  return (long long)z_padded_x(p->nx) * z_padded_y(p->ny) * p->nz;
}

long long obs_blocks_of(int kind, int nx, int ny, int nz) {
  const dim3 g = lb_grid(kind, nx, ny, nz);
  return (long long)g.x * g.y * g.z;
}

Layout layout_of(const dsm_params *p, const LBTable &t, long long N, long long pitch) {
  Layout L;
  size_t o = 0;
  auto take = [&](size_t bytes) {
    size_t at = o;
    o += (size_t)round_up((long long)bytes, 256);
    return at;
  };
  const size_t pop = (size_t)t.q * pitch * t.store_bytes;
  L.f[0] = take(pop);
  L.f[1] = take(pop);
  L.g[0] = take(pop);
  L.g[1] = take(pop);
  L.g0[0] = take(t.k16 ? pitch * sizeof(float) : 0);
  L.g0[1] = take(t.k16 ? pitch * sizeof(float) : 0);
  L.C[0] = take(pitch * t.real_bytes);
  L.C[1] = take(pitch * t.real_bytes);
  L.M = take(4 * pitch * t.real_bytes);
  L.C1 = take(pitch * t.real_bytes);
  L.mask = take(pitch);
  L.partials = take(obs_blocks_of(p->lattice, p->nx, p->ny, p->nz) * OBS_K * sizeof(double));
  L.obs = take(8 * sizeof(double));
  L.err = take(sizeof(int) * 4);
  const long long P = z_eligible(p) ? z_padded_nodes(p) : 0;
  L.Qz[0] = take(4 * P * t.real_bytes);
  L.Qz[1] = take(4 * P * t.real_bytes);
  L.Uz[0] = take(P * t.real_bytes);
  L.Uz[1] = take(P * t.real_bytes);
  L.C1z = take(P * t.real_bytes);
  L.total = o;
  (void)N;
  return L;
}

StepParams step_params(const dsm_params *p, const double k[3]) {
  StepParams s;
  s.kappa1 = k[0];
  s.kappa2 = k[1];
  s.kappa3 = k[2];
  s.a2 = p->alpha * p->alpha;
  s.alpha_s = p->alpha_s > 0.0 ? p->alpha_s : p->alpha;
  s.rho2 = p->rho2;
  s.rho3 = p->rho3;
  s.tau2 = p->tau2;
  s.tau3 = p->tau3;
  s.tau_g = p->tau_g;
  for (int a = 0; a < 3; a++) s.body[a] = p->body_force[a];
  if (p->lattice == DSM_D2Q9) s.body[2] = 0.0;
  s.beta = p->beta;
  s.omega = p->omega;
  s.rho_contrast = p->rho2 != p->rho3;
  s.walls = 0;
  for (int f = 0; f < 6; f++) {
    s.face[f] = p->face[f];
    s.walls |= p->face[f] != DSM_FACE_PERIODIC;
  }
  return s;
}

LBRaw raw_of(const dsm_lattice *h, int src) {
  LBRaw r;
  memset(&r, 0, sizeof(r));
  r.nx = h->prm.nx;
  r.ny = h->prm.ny;
  r.nz = h->prm.nz;
  r.N = h->N;
  r.pitch = h->pitch;
  r.f_in = h->f[src];
  r.g_in = h->g[src];
  r.g0_in = h->g0[src];
  r.f_out = h->f[src ^ 1];
  r.g_out = h->g[src ^ 1];
  r.g0_out = h->g0[src ^ 1];
  r.C = h->Cb[src ^ 1];
  r.Cprev = h->Cb[src];
  r.M = h->M;
  r.nxp = h->nxp;
  r.nyp = h->nyp;
  r.eq = h->eq;
  r.implicit = h->g_implicit;
  r.C1 = h->C1;
  r.mask = h->mask;
  r.partials = h->partials;
  r.err = h->err;
  r.p = h->sp;
  return r;
}

// ---- single-pass step -------------------------------------------------------
bool z_maps(dsm_lattice *h) {
  if (h->zmaps_ok) return true;
  const int rb = h->tab.real_bytes, nz = h->prm.nz;
  for (int b = 0; b < 2; b++) {
    if (!encode_plane_map(&h->maps[b].Q, h->Qz[b], rb, 4, h->nxp, h->nyp, nz, ZB_Y) ||
        !encode_plane_map(&h->maps[b].U, h->Uz[b], rb, 1, h->nxp, h->nyp, nz, ZB_Y) ||
        !encode_plane_map(&h->maps[b].C1, h->C1z, rb, 1, h->nxp, h->nyp, nz, ZB1_Y))
      return false;
  }
  h->zmaps_ok = true;
  return true;
}

// The longest-lasting choice of planes per block: runs of zr planes give
// tiles * ceil(nz / zr) blocks, which run in waves of the resident blocks; a
// wave lasts about zr planes plus the run's prologue (this step's C of two
// extra planes and the first staged planes, about 0.7 of a plane).
//
// With a density contrast in FP32 arithmetic a node beside the solid takes a
// multiple of another's time, and a lattice that is one wave of long runs waits for
// the blocks that have most of them.  Runs of more than 12 planes become runs of 7,
// which the SMs take as they come free.  us per step (before) over pillars and over a
// flat wall: 250 x 130 x 101 210 (273) and 195 (211), 160 x 130 x 101 136 (186) and 128
// (132), 128 x 128 x 101 115 (142) and 103 (99), 144^3 196 (231) and 187 (181).  Two
// passes take 230 and 204, 151 and 134, 117 and 105, 214 and 191.
int z_auto_run(dsm_lattice *h) {
  if (h->zrun_auto) return h->zrun_auto;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const long long resident = (long long)(sms > 0 ? sms : 152) * (h->tab.zresident() > 0 ? h->tab.zresident() : 1);
  const long long tiles = (long long)z_tiles_x(h->prm.nx) * z_tiles_y(h->prm.ny);
  const int nz = h->prm.nz;
  double best = 1e300;
  int run = nz;
  for (int zr = 1; zr <= nz; zr++) {
    const long long blocks = tiles * ((nz + zr - 1) / zr);
    const double waves = (double)((blocks + resident - 1) / resident);
    const double cost = waves * (zr + 0.7);
    if (cost < best - 1e-9) {
      best = cost;
      run = zr;
    }
  }
  if (run > 12 && h->sp.rho_contrast && h->tab.real_bytes == 4) run = 7;
  h->zrun_auto = run;
  return run;
}

bool z_active(const dsm_lattice *h) {
  return h->zok && h->eq && h->step_form == DSM_STEP_AUTO;
}

// Canonical g_eq state -> padded buffers (buffer 0), and padded C1.
cudaError_t z_pack(dsm_lattice *h) {
  if (!z_maps(h)) return cudaErrorInvalidValue;
  LBRaw a = raw_of(h, h->cur);
  cudaError_t e = h->tab.zpack(a, h->Qz[0], h->Qz[1], h->Uz[0], h->Uz[1], h->C1z, h->stream);
  if (e != cudaSuccess) return e;
  h->zc = 0;
  h->zpacked = true;
  return cudaSuccess;
}

// Padded state -> canonical g_eq state (A, u planes and C of the last
// collision), before any call that reads the state in its canonical layout.
cudaError_t t_copy(dsm_lattice *h);
cudaError_t z_unpack(dsm_lattice *h) {
  if (h->tp) return t_copy(h);
  if (!h->zpacked) return cudaSuccess;
  LBRaw a = raw_of(h, h->cur);
  cudaError_t e = h->tab.zunpack(a, h->Qz[h->zc], h->Uz[h->zc], h->Cb[h->cur], h->stream);
  if (e != cudaSuccess) return e;
  h->zpacked = false;
  return cudaSuccess;
}

// FP64 lattices in 2D that are neither so small that at most two of their 64-node
// tiles fall to an SM nor large enough for tiles of 256 nodes on every SM stay with
// two passes over populations: the FP64 pipe is the bound there, and the halo of a
// tile costs it more sums of C.  One launch against two passes, us per step:
// 128 x 64 11.1 and 24.7, 160 x 121 22.1 and 26.7, 256 x 96 33.7 and 28.8 (34.9 with
// tiles of 256), 256 x 128 42.3 and 32.9 (40.0), 304 x 256 50 and 68, 400 x 320 53 and
// 86, 512 x 512 87 and 140; ragged tiles, 19 x 1000, 28 and 37, 5 x 2000 28 and 49.
bool f64_tiles(const dsm_params *p) {
  if (p->precision != DSM_F64 || p->lattice != DSM_D2Q9) return true;
  const long long n = (long long)p->nx * p->ny;
  return n <= 2ll * 152 * 64 || n >= 2ll * 152 * 256;
}
// tiles of 16 x 4 nodes, which small FP64 lattices in 2D take
long long small_tiles(const dsm_params *p) {
  return ((p->nx + 15ll) / 16) * ((p->ny + 3ll) / 4);
}
// The same for the single pass over populations, whose halo costs more: up to 256
// small tiles (tau contrast, 128 x 120, 240 tiles, 33.0 and 24.4 us per step; 160 x
// 120, 300 tiles, 33.0 and 31.8, with mirrors and a density contrast 39.2 and 40.6;
// 17 x 1100, 550 tiles, 37.3 and 44.4), and large ones with a density contrast
// (512 x 400 185 and 153; without one 115 and 120).
bool f64_quads(const dsm_params *p) {
  if (p->precision != DSM_F64) return true;
  return f64_tiles(p) &&
         (small_tiles(p) <= 256 ||
          (p->rho2 != p->rho3 && (long long)p->nx * p->ny >= 2ll * 152 * 256));
}
// And for the solid's relaxation, which has less to do per node: up to 360 small tiles
// (40 x 480, 360 tiles, 21.2 and 13.2; 33 x 550, 414, 21.2 and 30.3) and from 90000
// nodes up (340 x 240 48.0 and 51.1, 300 x 300 47.9 and 37.7).
bool f64_relax(const dsm_params *p) {
  if (p->precision != DSM_F64) return true;
  return f64_tiles(p) && (small_tiles(p) <= 360 || (long long)p->nx * p->ny >= 90000);
}

// ---- single-pass step of D2Q9 ---------------------------------------------------
// It applies with tau_g = 1 and faces that are periodic or mirrors (at a wall
// g would bounce back, which no image node gives), in the automatic forms of g
// and of the step, where the step on moments does not.
bool t_eligible(const dsm_params *p) {
  if (p->lattice != DSM_D2Q9 || p->tau_g != 1.0 || !f64_quads(p)) return false;
  const int n[2] = {p->nx, p->ny};
  for (int a = 0; a < 2; a++) {
    const int lo = p->face[2 * a], hi = p->face[2 * a + 1];
    if (lo == DSM_FACE_WALL || hi == DSM_FACE_WALL) return false;
    if (lo == DSM_FACE_MIRROR && n[a] < 2) return false;  // the halo has two images
  }
  return true;
}

// Canonical planes of a state held as quads: (A, u) in M, C in Cb[cur], and for
// lattices that keep g as populations (mirrors) those in g[cur].
cudaError_t t_copy(dsm_lattice *h) {
  if (h->tcan) return cudaSuccess;
  LBRaw a = raw_of(h, h->cur ^ 1);  // g_out = g[cur]
  cudaError_t e = h->tab.tpack(a, h->Cb[h->cur], h->g[h->cur ^ 1], 0, h->stream);
  if (e == cudaSuccess && !h->eq) {
    a.Cprev = h->Cb[h->cur];
    e = h->tab.materialize(a, h->stream);
  }
  if (e != cudaSuccess) return e;
  h->g_implicit = h->eq;
  h->tcan = true;
  return cudaSuccess;
}

// One step of a lattice in this form.  A state given as populations takes its
// first step in two passes, which leave (A, u) and C.
cudaError_t t_step(dsm_lattice *h) {
  LBRaw a = raw_of(h, h->cur);
  cudaError_t e = cudaSuccess;
  if (!h->tp && !h->g_implicit) {
    a.eq = 1;
    e = h->tab.moments(a, h->stream);
    if (e == cudaSuccess) e = h->tab.node(a, 2, MODE_STEP, h->stream);
    if (e == cudaSuccess) e = h->tab.tpack(a, h->Cb[h->cur ^ 1], h->g[h->cur], 1, h->stream);
  } else {
    if (!h->tp) e = h->tab.tpack(a, h->Cb[h->cur], h->g[h->cur ^ 1], 1, h->stream);
    a.Qz = h->g[h->cur];
    if (e == cudaSuccess) e = h->tab.tstep(a, h->g[h->cur ^ 1], h->stream);
  }
  if (e != cudaSuccess) return e;
  h->tp = true;
  h->tcan = false;
  return cudaSuccess;
}

// ---- step on moments ----------------------------------------------------------
// It applies to lattices with every relaxation time 1, equal densities and
// periodic faces in the automatic storage form of g: FP32 and FP64 ones of any
// size, and those with 16-bit populations where the padded buffers of the
// population form's single pass exist (3D, nx >= 32, ny >= 8), in whose place
// the solid's data goes.  dsm_set_step_form chooses one pass or two.  With
// 16-bit populations the moments are FP32 reals all the same: 36 B per node are
// fewer than the 38 B of the populations and the 20 B of (A, C, u) that they
// replace, and nothing is rounded to 16 bits any more.  FP32 lattices narrower than a
// tile gain most, two launches for four (8^3 16.5 -> 9.6 us per step, 24^3 20.6 -> 10.8,
// 31 x 100 x 100 28.9 -> 19.2, 1 x 1000 x 40 113 -> 54, 300 x 5 x 30 22.8 -> 15.2).
// FP64 lattices in 3D, which the FP64 pipe bounds, keep their populations where a
// run of planes has too much to sum beside its own nodes: small ones (16^3: 53 us per
// step in two passes, 87 on moments; 32^3: 104 and 92; 64^3: 360 and 245), and those
// narrower than a tile in x up to 80000 nodes (24 x 48 x 48 103 and 114, 31 x 64 x 64
// 166 and 157) or in y (128 x 4 x 100 95 and 136, 300 x 5 x 100 229 and 241).
bool m_f64_3d(const dsm_params *p) {
  const long long n = (long long)p->nx * p->ny * p->nz;
  return n >= 32768 && (z_tiles(p->nx, p->ny) || (n >= 80000 && p->ny >= 8));
}
bool m_eligible(const dsm_params *p) {
  if (p->precision == DSM_F64 && p->lattice == DSM_D3Q19 && !m_f64_3d(p)) return false;
  const bool k16 = p->precision != DSM_F32 && p->precision != DSM_F64;
  return (!k16 || z_eligible(p)) && f64_tiles(p) && p->tau2 == 1.0 && p->tau3 == 1.0 && p->tau_g == 1.0 &&
         p->rho2 == p->rho3 && !has_walls(p);
}
bool m_active(const dsm_lattice *h) {
  return h->mok && h->eq;
}

// The moments use buffers the g_eq form leaves idle: buffer b in g[b]; the
// solid's pairs and link bits behind them, its link fractions in f[0].  With
// 16-bit populations the fractions take f[0] and f[1] (72 of 76 B per node), the
// wall sums Qz[0], the solid's pairs, link bits and list Qz[1].  The canonical
// copy of a state held as moments goes to buffer 1 (and ends the solid's data).
MomRaw m_raw(const dsm_lattice *h, int src) {
  MomRaw r;
  memset(&r, 0, sizeof(r));
  r.nx = h->prm.nx;
  r.ny = h->prm.ny;
  r.nz = h->prm.nz;
  r.N = h->N;
  r.pitch = h->pitch;
  const size_t plane = (size_t)h->pitch * h->tab.real_bytes;
  const int nm = mom_reals(h->kind);
  for (int o = 0; o < 2; o++) {
    char *b = (char *)h->g[o ? src ^ 1 : src];
    void **d = o ? r.out : r.in;
    d[0] = b;
    d[1] = b + 4 * plane;
    d[2] = b + (nm - 1) * plane;
  }
  r.sol = (char *)h->g[0] + nm * plane;
  r.lk = (char *)h->g[1] + nm * plane;
  r.qpl = h->f[0];
  r.near = h->mask;
  r.count = (int *)(h->obs + 6);
  if (h->kind == DSM_D3Q19) {
    r.list = (char *)r.lk + plane;
    r.wall = (char *)r.sol + 2 * plane;
    if (h->tab.k16 && h->zok) {
      r.wall = h->Qz[0];
      r.sol = h->Qz[1];
      r.lk = (char *)h->Qz[1] + 2 * plane;
      r.list = (char *)h->Qz[1] + 3 * plane;
    }
  }
  r.c1 = h->C1;
  r.err = h->err;
  r.k[0] = h->sp.kappa2;
  r.ak[0] = h->sp.a2 * h->sp.kappa2;
  r.kl = h->sp.kappa3;
  r.akl = h->sp.a2 * h->sp.kappa3;
  r.rho = h->sp.rho3;
  for (int a = 0; a < 3; a++) r.body[a] = h->sp.body[a];
  r.alpha_s = h->sp.alpha_s;
  r.step = (unsigned)h->step;
  return r;
}

// For kernels that collide only for a read: what they find non-finite is the next
// step's, which may never come (another body force, another state), and goes to
// the error words' second one, of which only bounds faults count.
MomRaw m_read(const dsm_lattice *h, int src) {
  MomRaw r = m_raw(h, src);
  r.err = h->err + 1;
  return r;
}

// canonical planes of buffer b
MomPlanes m_planes(const dsm_lattice *h, int b) {
  const size_t plane = (size_t)h->pitch * h->tab.real_bytes;
  return {h->f[b], h->M, (char *)h->M + plane, h->Cb[b]};
}

cudaError_t m_statics(dsm_lattice *h) {
  if (h->mstat) return cudaSuccess;
  const cudaError_t e = h->tab.mom_solid(m_raw(h, 0), h->stream);
  if (e == cudaSuccess) h->mstat = true;
  return e;
}

// A state held as moments -> canonical form (buffer 1, g as g_eq).
cudaError_t m_leave(dsm_lattice *h) {
  if (!h->mom) return cudaSuccess;
  const cudaError_t e = h->tab.mom_expand(m_raw(h, h->mc), m_planes(h, 1), 1, h->stream);
  if (e != cudaSuccess) return e;
  h->cur = 1;
  h->g_implicit = true;
  h->mom = h->mcp = h->mpk = h->mstat = false;
  h->mfit = true;
  return cudaSuccess;
}

// A new state arrives by other means.
void m_drop(dsm_lattice *h) { h->mom = h->mcp = h->mpk = h->mstat = h->mfit = h->tp = h->tcan = false; }

// C of the next step of a state held as moments, into Cb[0].
cudaError_t m_c(dsm_lattice *h) {
  if (h->mcp) return cudaSuccess;
  const cudaError_t e = h->tab.mom_c(m_raw(h, h->mc), h->Cb[0], 0, h->stream);
  if (e == cudaSuccess) h->mcp = true;
  return e;
}

// Canonical state (mfit) -> moments, buffer 0.
cudaError_t m_enter(dsm_lattice *h) {
  MomRaw r = m_raw(h, 1);  // out = buffer 0
  cudaError_t e = h->tab.mom_enter(r, m_planes(h, h->cur), h->stream);
  if (e == cudaSuccess) e = m_statics(h);
  if (e != cudaSuccess) return e;
  h->mc = 0;
  h->mom = true;
  h->mstepped = true;
  h->mcp = h->mpk = h->tp = h->tcan = false;
  return cudaSuccess;
}

bool t_active(const dsm_lattice *h) {
  return h->tok && !m_active(h) && h->g_form == DSM_G_AUTO && h->step_form == DSM_STEP_AUTO;
}

int m_zrun(dsm_lattice *h) {
  if (h->zrun > 0) return h->zrun;
  if (h->mzrun) return h->mzrun;
  h->mzrun = 1;
  if (h->kind != DSM_D3Q19) return 1;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int per_sm = h->tab.mom_resident();
  h->mzrun = mom_zrun(h->prm.nx, h->prm.ny, h->prm.nz, sms > 0 ? sms : 152, per_sm,
                      h->prm.precision == DSM_F64);
  return h->mzrun;
}

// Whether dsm_relax_solid runs on moments: D2Q9 in FP32 or FP64, each axis
// periodic, or a mirror on both sides (a wall's bounce-back has no image node).
bool m_relax_of(const dsm_lattice *h, MomRelax *m) {
  if (h->kind != DSM_D2Q9 || !h->tab.mom_relax || !f64_relax(&h->prm)) return false;
  const int n[2] = {h->prm.nx, h->prm.ny};
  for (int a = 0; a < 2; a++) {
    const int lo = h->prm.face[2 * a], hi = h->prm.face[2 * a + 1];
    if (lo == DSM_FACE_WALL || hi == DSM_FACE_WALL) return false;
    m->mirror[a] = lo == DSM_FACE_MIRROR;
    if (m->mirror[a] && n[a] < 2) return false;
  }
  m->mask = h->mask;
  m->beta2 = 2.0 * h->sp.beta;
  m->omega2 = 2.0 * h->sp.omega;
  return true;
}

// The second pass of a step of a state held as moments (C in Cb[0]).
cudaError_t m_collide(dsm_lattice *h) {
  cudaError_t e = m_statics(h);
  if (e == cudaSuccess)
    e = h->tab.mom_node(m_raw(h, h->mc), h->Cb[0], 0, MODE_STEP, 0, 0, nullptr, nullptr,
                        h->stream);
  if (e != cudaSuccess) return e;
  h->mc ^= 1;
  h->mcp = h->mpk = false;
  h->mstepped = true;
  return cudaSuccess;
}

// One step of a state held as moments, in one pass or two.
cudaError_t m_step(dsm_lattice *h) {
  cudaError_t e = m_statics(h);
  if (h->step_form == DSM_STEP_TWO_PASS) {
    if (e == cudaSuccess) e = m_c(h);
    return e == cudaSuccess ? m_collide(h) : e;
  }
  if (e == cudaSuccess) e = h->tab.mom_step(m_raw(h, h->mc), m_zrun(h), h->stream);
  if (e != cudaSuccess) return e;
  h->mc ^= 1;
  h->mcp = h->mpk = false;
  h->mstepped = true;
  return cudaSuccess;
}

// The next step of a state held as moments, into the other buffer, for the reads
// that take their values from it: in 3D, where the automatic form steps.
bool m_peeks(const dsm_lattice *h) {
  return h->kind == DSM_D3Q19 && h->step_form == DSM_STEP_AUTO;
}
cudaError_t m_peek(dsm_lattice *h) {
  if (h->mpk) return cudaSuccess;
  cudaError_t e = m_statics(h);
  if (e == cudaSuccess) e = h->tab.mom_step(m_read(h, h->mc), m_zrun(h), h->stream);
  if (e == cudaSuccess) h->mpk = true;
  return e;
}

// Read and clear nothing: report the latched device error word.
dsm_status read_err(dsm_lattice *h, int *word) {
  int w[2] = {0, 0};
  cudaError_t e = cudaMemcpyAsync(w, h->err, sizeof(w), cudaMemcpyDeviceToHost, h->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) return DSM_E_CUDA;
  *word = w[0] | (w[1] & ERR_BOUNDS);
  return DSM_OK;
}

}  // namespace

// Final deterministic reduction of the observables' block partials.
__global__ void obs_finalize_kernel(const double *partials, long long nb, double *out) {
  __shared__ double sh[OBS_K][256];
  double s[OBS_K] = {0, 0, 0, 0, 0};
  for (long long b = threadIdx.x; b < nb; b += blockDim.x)
    for (int k = 0; k < OBS_K; k++) {
      const double v = partials[b * OBS_K + k];
      s[k] = (k >= 3) ? fmax(s[k], v) : s[k] + v;
    }
  for (int k = 0; k < OBS_K; k++) sh[k][threadIdx.x] = s[k];
  __syncthreads();
  for (int st = blockDim.x / 2; st > 0; st >>= 1) {
    if (threadIdx.x < st)
      for (int k = 0; k < OBS_K; k++)
        sh[k][threadIdx.x] = (k >= 3) ? fmax(sh[k][threadIdx.x], sh[k][threadIdx.x + st])
                                      : sh[k][threadIdx.x] + sh[k][threadIdx.x + st];
    __syncthreads();
  }
  if (threadIdx.x < OBS_K) out[threadIdx.x] = sh[threadIdx.x][0];
}

// One observables record (step, then the OBS_K values) into the ring.
__global__ void obs_record_kernel(const double *obs, double *rec, long long step) {
  if (threadIdx.x == 0) rec[0] = (double)step;
  if (threadIdx.x < OBS_K) rec[1 + threadIdx.x] = obs[threadIdx.x];
}

namespace {

// The observables of the current state into h->obs, on the lattice's stream,
// without synchronising: the moments and observables passes over the
// canonical state, then the deterministic final reduction.
cudaError_t obs_launch(dsm_lattice *h) {
  cudaError_t e;
  if (h->mom && m_peeks(h)) {
    e = m_peek(h);
    if (e == cudaSuccess)
      e = h->tab.mom_peek(m_raw(h, h->mc ^ 1), MODE_OBS, 0, nullptr, h->partials, h->stream);
    if (e != cudaSuccess) return e;
    obs_finalize_kernel<<<1, 256, 0, h->stream>>>(h->partials, h->obs_blocks, h->obs);
    return cudaGetLastError();
  }
  if (h->mom) {
    e = m_statics(h);
    if (e == cudaSuccess) e = m_c(h);
    if (e == cudaSuccess)
      e = h->tab.mom_node(m_read(h, h->mc), h->Cb[0], 0, MODE_OBS, 0, 0, nullptr, h->partials,
                          h->stream);
    if (e != cudaSuccess) return e;
    obs_finalize_kernel<<<1, 256, 0, h->stream>>>(h->partials, h->obs_blocks, h->obs);
    return cudaGetLastError();
  }
  e = z_unpack(h);
  if (e != cudaSuccess) return e;
  LBRaw a = raw_of(h, h->cur);
  e = h->tab.moments(a, h->stream);
  if (e == cudaSuccess) e = h->tab.node(a, 2, MODE_OBS, h->stream);
  if (e != cudaSuccess) return e;
  obs_finalize_kernel<<<1, 256, 0, h->stream>>>(h->partials, h->obs_blocks, h->obs);
  return cudaGetLastError();
}

}  // namespace

// S = {C1 > 1/2} (dsm_solid_region)
template <class T>
__global__ void __launch_bounds__(256) solid_region_kernel(const T *c1, unsigned char *mask,
                                                           long long n) {
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
       k += (long long)gridDim.x * blockDim.x)
    mask[k] = c1[k] > T(0.5) ? 1 : 0;
}

extern "C" {

int dsm_checked_build(void) {
#ifdef DSM_CHECKED
  return 1;
#else
  return 0;
#endif
}

const char *dsm_status_string(dsm_status s) {
  switch (s) {
    case DSM_OK: return "ok";
    case DSM_E_INVAL: return "invalid argument";
    case DSM_E_WORKSPACE: return "workspace too small or misaligned";
    case DSM_E_CUDA: return "CUDA error";
    case DSM_E_NONFINITE: return "non-finite population";
    case DSM_E_TIMEOUT: return "device wait timed out";
    case DSM_E_STATE: return "call out of order or handle latched in error";
    case DSM_E_UNSUPPORTED: return "unsupported";
    case DSM_E_BOUNDS: return "index out of bounds (checked build)";
  }
  return "unknown status";
}

dsm_status dsm_lattice_table(int lattice, int *q_out, int *c_out, double *w_out) {
  if (!q_out || !c_out || !w_out) return DSM_E_INVAL;
  if (lattice == DSM_D2Q9) {
    *q_out = 9;
    for (int i = 0; i < 9; i++) {
      c_out[3 * i] = Lat<0>::cx(i);
      c_out[3 * i + 1] = Lat<0>::cy(i);
      c_out[3 * i + 2] = 0;
      w_out[i] = Lat<0>::w(i);
    }
    return DSM_OK;
  }
  if (lattice == DSM_D3Q19) {
    *q_out = 19;
    for (int i = 0; i < 19; i++) {
      c_out[3 * i] = Lat<1>::cx(i);
      c_out[3 * i + 1] = Lat<1>::cy(i);
      c_out[3 * i + 2] = Lat<1>::cz(i);
      w_out[i] = Lat<1>::w(i);
    }
    return DSM_OK;
  }
  return DSM_E_INVAL;
}

dsm_status dsm_kappa(const dsm_params *p, double kappa_out[3]) {
  if (!p || !kappa_out) return DSM_E_INVAL;
  return kappa_of(p, kappa_out);
}

dsm_status dsm_workspace_bytes(const dsm_params *p, size_t *bytes) {
  dsm_status s = check_params(p);
  if (s != DSM_OK) return s;
  if (!bytes) return DSM_E_INVAL;
  LBTable t;
  lb_table_for(p->lattice, p->precision, &t);
  const long long N = (long long)p->nx * p->ny * p->nz;
  *bytes = layout_of(p, t, N, round_up(N, 64)).total;
  return DSM_OK;
}

dsm_status dsm_create(const dsm_params *p, void *d_workspace, size_t bytes, void *cuda_stream,
                      dsm_lattice **out) {
  if (!out) return DSM_E_INVAL;
  *out = nullptr;
  dsm_status s = check_params(p);
  if (s != DSM_OK) return s;
  LBTable t;
  lb_table_for(p->lattice, p->precision, &t);
  const long long N = (long long)p->nx * p->ny * p->nz;
  const long long pitch = round_up(N, 64);
  Layout L = layout_of(p, t, N, pitch);
  if (!d_workspace || bytes < L.total || ((uintptr_t)d_workspace & 255u)) return DSM_E_WORKSPACE;
  dsm_lattice *h = new (std::nothrow) dsm_lattice;
  if (!h) return DSM_E_INVAL;
  memset(h, 0, sizeof(*h));
  h->prm = *p;
  kappa_of(p, h->kappa);
  h->tab = t;
  h->kind = p->lattice;
  h->q = t.q;
  h->N = N;
  h->pitch = pitch;
  h->ws = (char *)d_workspace;
  h->ws_bytes = bytes;
  for (int b = 0; b < 2; b++) {
    h->f[b] = h->ws + L.f[b];
    h->g[b] = h->ws + L.g[b];
    h->g0[b] = t.k16 ? (float *)(h->ws + L.g0[b]) : nullptr;
  }
  h->Cb[0] = h->ws + L.C[0];
  h->Cb[1] = h->ws + L.C[1];
  h->M = h->ws + L.M;
  h->C1 = h->ws + L.C1;
  h->mask = (unsigned char *)(h->ws + L.mask);
  h->partials = (double *)(h->ws + L.partials);
  h->obs = (double *)(h->ws + L.obs);
  h->err = (int *)(h->ws + L.err);
  h->obs_blocks = obs_blocks_of(p->lattice, p->nx, p->ny, p->nz);
  h->zok = z_eligible(p);
  h->nxp = z_padded_x(p->nx);
  h->nyp = z_padded_y(p->ny);
  for (int b = 0; b < 2; b++) {
    h->Qz[b] = h->zok ? h->ws + L.Qz[b] : nullptr;
    h->Uz[b] = h->zok ? h->ws + L.Uz[b] : nullptr;
  }
  h->C1z = h->zok ? h->ws + L.C1z : nullptr;
  h->step_form = DSM_STEP_AUTO;
  h->stream = (cudaStream_t)cuda_stream;
  h->sp = step_params(p, h->kappa);
  h->g_form = DSM_G_AUTO;
  h->eq = p->tau_g == 1.0 && !has_walls(p);
  h->mok = m_eligible(p) && t.mom_step;
  h->tok = t_eligible(p) && t.tstep;
  // no solid yet: C1 = 0 everywhere; clear the error word and the mask
  cudaError_t e = cudaMemsetAsync(h->C1, 0, pitch * t.real_bytes, h->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(h->mask, 0, pitch, h->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(h->err, 0, sizeof(int) * 4, h->stream);
  if (e != cudaSuccess) {
    delete h;
    return DSM_E_CUDA;
  }
  *out = h;
  return DSM_OK;
}

dsm_status dsm_set_solid(dsm_lattice *h, const void *d_field, int kind) {
  if (!h || !d_field) return DSM_E_INVAL;
  cudaError_t e;
  if (kind == 0) e = h->tab.solid(d_field, h->C1, h->N, h->sp.alpha_s, h->stream);
  else if (kind == 1)
    e = cudaMemcpyAsync(h->C1, d_field, h->N * h->tab.real_bytes, cudaMemcpyDeviceToDevice, h->stream);
  else return DSM_E_INVAL;
  if (e != cudaSuccess) return DSM_E_CUDA;
  h->has_solid = true;
  h->has_fluid = false;
  h->zpacked = false;
  m_drop(h);
  return DSM_OK;
}

dsm_status dsm_relax_solid(dsm_lattice *h, const unsigned char *d_mask, int steps, double beta,
                           double omega) {
  TraceRange trace_range("dsm_relax_solid (stage 1)");
  if (!h || !d_mask || steps < 0 || beta < 0.0 || omega < 0.0) return DSM_E_INVAL;
  cudaError_t e = cudaMemcpyAsync(h->mask, d_mask, h->N, cudaMemcpyDeviceToDevice, h->stream);
  if (e != cudaSuccess) return DSM_E_CUDA;
  h->sp.beta = beta;
  h->sp.omega = omega;
  // initial state of stage 1 from the current C1, written into buffer 0
  // (stage 1 keeps g as populations)
  h->cur = 0;
  h->g_implicit = false;
  h->has_fluid = false;
  h->zpacked = false;
  m_drop(h);
  MomRelax mr;
  if (m_relax_of(h, &mr)) {
    // every relaxation time is 1 here, so moments carry the state (dsm_mom.cuh)
    MomRaw a[2] = {m_raw(h, 0), m_raw(h, 1)};
    for (MomRaw &r : a) {
      r.k[0] = h->sp.kappa1 + h->sp.kappa3;
      r.ak[0] = h->sp.a2 * r.k[0];
      r.rho = 1.0;
    }
    e = h->tab.mom_relax(a[1], mr, 0, h->C1, h->stream);
    for (int t = 0; t < steps && e == cudaSuccess; t++) {
      a[t & 1].step = (unsigned)t;
      e = h->tab.mom_relax(a[t & 1], mr, 1, nullptr, h->stream);
    }
    a[steps & 1].step = (unsigned)steps;
    if (e == cudaSuccess) e = h->tab.mom_relax(a[steps & 1], mr, 2, h->C1, h->stream);
    h->sp.beta = h->prm.beta;
    h->sp.omega = h->prm.omega;
    if (e != cudaSuccess) return DSM_E_CUDA;
    h->has_solid = true;
    return DSM_OK;
  }
  LBRaw r = raw_of(h, 1);  // out = buffer 0
  r.eq = 0;
  if ((e = h->tab.init(r, h->C1, 1, h->stream)) != cudaSuccess) return DSM_E_CUDA;
  for (int t = 0; t < steps; t++) {
    LBRaw a = raw_of(h, h->cur);
    a.eq = 0;
    if ((e = h->tab.moments(a, h->stream)) != cudaSuccess) return DSM_E_CUDA;
    if ((e = h->tab.node(a, 1, MODE_STEP, h->stream)) != cudaSuccess) return DSM_E_CUDA;
    h->cur ^= 1;
  }
  // relaxed C1 = the concentration the next step would see
  LBRaw a = raw_of(h, h->cur);
  if ((e = h->tab.moments(a, h->stream)) != cudaSuccess) return DSM_E_CUDA;
  e = cudaMemcpyAsync(h->C1, a.C, h->N * h->tab.real_bytes, cudaMemcpyDeviceToDevice, h->stream);
  if (e != cudaSuccess) return DSM_E_CUDA;
  h->sp.beta = h->prm.beta;
  h->sp.omega = h->prm.omega;
  h->has_solid = true;
  h->has_fluid = false;
  return DSM_OK;
}

dsm_status dsm_solid_region(dsm_lattice *h, unsigned char *d_mask) {
  if (!h || !d_mask) return DSM_E_INVAL;
  if (!h->has_solid) return DSM_E_STATE;
  long long blocks = (h->N + 255) / 256;
  if (blocks > 152 * 16) blocks = 152 * 16;
  if (h->tab.real_bytes == 8)
    solid_region_kernel<double><<<(int)blocks, 256, 0, h->stream>>>((const double *)h->C1, d_mask,
                                                                    h->N);
  else
    solid_region_kernel<float><<<(int)blocks, 256, 0, h->stream>>>((const float *)h->C1, d_mask,
                                                                   h->N);
  return cuda_status(cudaGetLastError());
}

dsm_status dsm_set_fluid(dsm_lattice *h, const void *d_c2) {
  if (!h || !d_c2) return DSM_E_INVAL;
  h->cur = 0;
  cudaError_t e;
  if (m_active(h)) {  // the rest state as moments
    if (!h->mom) h->mstat = false;  // (its buffers held another form)
    e = m_statics(h);
    if (e == cudaSuccess) e = h->tab.mom_init(m_raw(h, 1), d_c2, 0, h->stream);  // writes buffer 0
    h->mc = 0;
    h->mom = true;
    h->mcp = h->mpk = h->mfit = h->mstepped = h->tp = h->tcan = false;
  } else {
    m_drop(h);
    LBRaw r = raw_of(h, 1);  // writes buffer 0
    e = h->tab.init(r, d_c2, 2, h->stream);
  }
  if (e == cudaSuccess) e = cudaMemsetAsync(h->err, 0, sizeof(int) * 4, h->stream);
  if (e != cudaSuccess) return DSM_E_CUDA;
  h->step = 0;
  h->has_fluid = true;
  h->latched = false;
  h->moments_ready = false;
  h->g_implicit = false;  // the initial g are written as populations
  h->zpacked = false;
  return DSM_OK;
}

dsm_status dsm_step(dsm_lattice *h, long long nsteps) {
  TraceRange trace_range("dsm_step");
  if (!h || nsteps < 0) return DSM_E_INVAL;
  if (!h->has_fluid || h->latched) return DSM_E_STATE;
  const bool mom = m_active(h), single = !mom && z_active(h), tile = t_active(h);
  if (!single && !tile && z_unpack(h) != cudaSuccess) return DSM_E_CUDA;
  if (!mom && m_leave(h) != cudaSuccess) return DSM_E_CUDA;
  for (long long t = 0; t < nsteps; t++) {
    cudaError_t e;
    if (mom && (h->mom || (h->mfit && h->g_implicit))) {
      if (!h->mom && m_enter(h) != cudaSuccess) return DSM_E_CUDA;
      e = m_step(h);
      if (e != cudaSuccess) return DSM_E_CUDA;
    } else if (single && h->g_implicit) {
      // one pass per step over the padded g_eq state
      if (!h->zpacked && (e = z_pack(h)) != cudaSuccess) return DSM_E_CUDA;
      LBRaw a = raw_of(h, h->cur);
      a.Qz = h->Qz[h->zc ^ 1];
      a.Uz = h->Uz[h->zc ^ 1];
      e = h->tab.zstep(a, h->maps[h->zc], h->zrun > 0 ? h->zrun : z_auto_run(h), h->stream);
      if (e != cudaSuccess) return DSM_E_CUDA;
      h->zc ^= 1;
    } else if (tile) {
      if (t_step(h) != cudaSuccess) return DSM_E_CUDA;
    } else {
      h->tp = h->tcan = false;
      // moments pass, then the fused pass (also the first step of a state given
      // as populations)
      LBRaw a = raw_of(h, h->cur);
      e = h->tab.moments(a, h->stream);
      if (e == cudaSuccess) e = h->tab.node(a, 2, MODE_STEP, h->stream);
      if (e != cudaSuccess) return DSM_E_CUDA;
      h->mfit = h->mok && h->eq;
    }
    if (!h->mom) {
      h->cur ^= 1;
      h->g_implicit = h->eq;
    }
    h->step++;
    if (h->ring && h->step % h->ring_every == 0) {
      // observables record into the ring: device work only, no synchronisation
      if ((e = obs_launch(h)) != cudaSuccess) return DSM_E_CUDA;
      double *rec = h->ring + (h->ring_count % h->ring_cap) * DSM_OBS_RECORD;
      obs_record_kernel<<<1, 32, 0, h->stream>>>(h->obs, rec, h->step);
      if ((e = cudaGetLastError()) != cudaSuccess) return DSM_E_CUDA;
      h->ring_count++;
    }
  }
  h->moments_ready = false;
  return DSM_OK;
}

dsm_status dsm_set_observables_ring(dsm_lattice *h, double *d_ring, int capacity,
                                    long long every) {
  if (!h) return DSM_E_INVAL;
  if (!d_ring || every == 0) {
    h->ring = nullptr;
    h->ring_cap = 0;
    h->ring_every = 0;
    h->ring_count = 0;
    return DSM_OK;
  }
  if (capacity < 1 || every < 0 || ((uintptr_t)d_ring & 7u)) return DSM_E_INVAL;
  h->ring = d_ring;
  h->ring_cap = capacity;
  h->ring_every = every;
  h->ring_count = 0;
  return DSM_OK;
}

dsm_status dsm_observables_ring_count(const dsm_lattice *h, long long *written) {
  if (!h || !written) return DSM_E_INVAL;
  *written = h->ring_count;
  return DSM_OK;
}

dsm_status dsm_set_body_force(dsm_lattice *h, const double *body) {
  if (!h || !body) return DSM_E_INVAL;
  for (int a = 0; a < 3; a++)
    if (!isfinite(body[a])) return DSM_E_INVAL;
  for (int a = 0; a < 3; a++) h->prm.body_force[a] = body[a];
  h->mpk = false;
  h->sp.body[0] = body[0];
  h->sp.body[1] = body[1];
  h->sp.body[2] = h->kind == DSM_D2Q9 ? 0.0 : body[2];
  return DSM_OK;
}

dsm_status dsm_set_step_form(dsm_lattice *h, int form, int zrun) {
  if (!h || (form != DSM_STEP_AUTO && form != DSM_STEP_TWO_PASS) || zrun < 0) return DSM_E_INVAL;
  if (form == DSM_STEP_TWO_PASS && z_unpack(h) != cudaSuccess) return DSM_E_CUDA;
  h->step_form = form;
  h->zrun = zrun;
  return DSM_OK;
}

dsm_status dsm_step_info(dsm_lattice *h, int *single_pass, int *zrun) {
  if (!h) return DSM_E_INVAL;
  const bool single = z_active(h);
  if (single_pass) *single_pass = single ? 1 : 0;
  if (zrun) *zrun = single ? (h->zrun > 0 ? h->zrun : m_active(h) ? m_zrun(h) : z_auto_run(h)) : 0;
  return DSM_OK;
}

dsm_status dsm_step_moments(dsm_lattice *h) {
  TraceRange trace_range("moments pass (K1)");
  if (!h) return DSM_E_INVAL;
  if (!h->has_fluid || h->latched) return DSM_E_STATE;
  if (z_unpack(h) != cudaSuccess) return DSM_E_CUDA;
  if (m_active(h) && !h->mom && h->mfit && h->g_implicit && m_enter(h) != cudaSuccess)
    return DSM_E_CUDA;
  if (h->mom) {
    if (m_c(h) != cudaSuccess) return DSM_E_CUDA;
    h->moments_ready = true;
    return DSM_OK;
  }
  LBRaw a = raw_of(h, h->cur);
  if (h->tab.moments(a, h->stream) != cudaSuccess) return DSM_E_CUDA;
  h->moments_ready = true;
  return DSM_OK;
}

dsm_status dsm_step_collide(dsm_lattice *h) {
  TraceRange trace_range("fused pass (K2)");
  if (!h) return DSM_E_INVAL;
  if (!h->has_fluid || h->latched || !h->moments_ready) return DSM_E_STATE;
  if (z_unpack(h) != cudaSuccess) return DSM_E_CUDA;
  if (h->mom) {
    if (m_c(h) != cudaSuccess || m_collide(h) != cudaSuccess) return DSM_E_CUDA;
    h->step++;
    h->moments_ready = false;
    return DSM_OK;
  }
  LBRaw a = raw_of(h, h->cur);
  if (h->tab.node(a, 2, MODE_STEP, h->stream) != cudaSuccess) return DSM_E_CUDA;
  h->tp = h->tcan = false;
  h->cur ^= 1;
  h->step++;
  h->g_implicit = h->eq;
  h->mfit = h->mok && h->eq;
  h->moments_ready = false;
  return DSM_OK;
}

dsm_status dsm_get_observables(dsm_lattice *h, dsm_observables *out) {
  if (!h || !out) return DSM_E_INVAL;
  if (!h->has_fluid) return DSM_E_STATE;
  cudaError_t e = obs_launch(h);
  if (e != cudaSuccess) return DSM_E_CUDA;
  double v[OBS_K];
  e = cudaMemcpyAsync(v, h->obs, sizeof(v), cudaMemcpyDeviceToHost, h->stream);
  if (e != cudaSuccess) return DSM_E_CUDA;
  int word = 0;
  dsm_status s = read_err(h, &word);  // synchronises
  if (s != DSM_OK) return s;
  out->mass_c2 = v[0];
  out->mass_c1 = v[1];
  out->kinetic = v[2];
  out->max_u = v[3];
  out->step = h->step;
  out->nonfinite = (v[4] > 0.0 || (word & ERR_NONFINITE)) ? 1 : 0;
  if (word & ERR_TIMEOUT) {
    h->latched = true;
    return DSM_E_TIMEOUT;
  }
  if (word & ERR_BOUNDS) {
    h->latched = true;
    return DSM_E_BOUNDS;
  }
  if (out->nonfinite) {
    h->latched = true;
    return DSM_E_NONFINITE;
  }
  return DSM_OK;
}

dsm_status dsm_get_field(dsm_lattice *h, int field, void *d_dst) {
  if (!h || !d_dst || field < DSM_FIELD_C1 || field > DSM_FIELD_TAU) return DSM_E_INVAL;
  cudaError_t e;
  if (field == DSM_FIELD_C1) {
    e = cudaMemcpyAsync(d_dst, h->C1, h->N * h->tab.real_bytes, cudaMemcpyDeviceToDevice, h->stream);
    return cuda_status(e);
  }
  if (!h->has_fluid) return DSM_E_STATE;
  if (h->mom && m_peeks(h)) {
    e = field == DSM_FIELD_RHO || field == DSM_FIELD_TAU ? m_statics(h) : m_peek(h);
    if (e == cudaSuccess)
      e = h->tab.mom_peek(m_raw(h, h->mc ^ 1), MODE_FIELDS, field, d_dst, nullptr, h->stream);
    return cuda_status(e);
  }
  if (h->mom) {
    if (field == DSM_FIELD_C2 && !h->mcp)
      return cuda_status(h->tab.mom_c(m_raw(h, h->mc), d_dst, 0, h->stream));
    if (field == DSM_FIELD_C2)
      return cuda_status(cudaMemcpyAsync(d_dst, h->Cb[0], h->N * h->tab.real_bytes,
                                         cudaMemcpyDeviceToDevice, h->stream));
    e = m_statics(h);
    if (e == cudaSuccess) e = m_c(h);
    if (e == cudaSuccess)
      e = h->tab.mom_node(m_read(h, h->mc), h->Cb[0], 0, MODE_FIELDS, field, 0, d_dst, nullptr,
                          h->stream);
    return cuda_status(e);
  }
  if (z_unpack(h) != cudaSuccess) return DSM_E_CUDA;
  LBRaw a = raw_of(h, h->cur);
  a.out = d_dst;
  a.field_sel = field;
  e = h->tab.moments(a, h->stream);
  if (e == cudaSuccess) e = h->tab.node(a, 2, MODE_FIELDS, h->stream);
  return cuda_status(e);
}

dsm_status dsm_get_populations(dsm_lattice *h, void *d_f, void *d_g) {
  if (!h || !d_f || !d_g) return DSM_E_INVAL;
  if (!h->has_fluid) return DSM_E_STATE;
  if (h->mom)
    return cuda_status(h->tab.mom_expand(m_raw(h, h->mc), {d_f, nullptr, nullptr, d_g}, 2,
                                         h->stream));
  if (z_unpack(h) != cudaSuccess) return DSM_E_CUDA;
  LBRaw a = raw_of(h, h->cur);
  return cuda_status(h->tab.get_pops(a, d_f, d_g, h->stream));
}

dsm_status dsm_set_populations(dsm_lattice *h, const void *d_f, const void *d_g) {
  if (!h || !d_f || !d_g) return DSM_E_INVAL;
  m_drop(h);
  LBRaw a = raw_of(h, h->cur ^ 1);  // out = current buffer
  cudaError_t e = h->tab.set_pops(a, d_f, d_g, h->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(h->err, 0, sizeof(int) * 4, h->stream);
  if (e != cudaSuccess) return DSM_E_CUDA;
  h->has_fluid = true;
  h->latched = false;
  h->moments_ready = false;
  h->g_implicit = false;
  h->zpacked = false;
  return DSM_OK;
}

dsm_status dsm_set_g_storage(dsm_lattice *h, int form) {
  if (!h || (form != DSM_G_AUTO && form != DSM_G_POPULATIONS)) return DSM_E_INVAL;
  const bool eq = form == DSM_G_AUTO && h->prm.tau_g == 1.0 && !has_walls(&h->prm);
  if (z_unpack(h) != cudaSuccess) return DSM_E_CUDA;
  if (!eq && m_leave(h) != cudaSuccess) return DSM_E_CUDA;
  if (form == DSM_G_POPULATIONS) h->tp = h->tcan = false;  // (the canonical copy is the state)
  if (h->g_implicit && !eq) {
    // write the current g_eq out as populations of the current buffer
    LBRaw a = raw_of(h, h->cur ^ 1);  // g_out = current buffer
    a.Cprev = h->Cb[h->cur];
    if (h->tab.materialize(a, h->stream) != cudaSuccess) return DSM_E_CUDA;
    h->g_implicit = false;
    h->mfit = false;
    h->moments_ready = false;
  }
  h->g_form = form;
  h->eq = eq;
  return DSM_OK;
}

dsm_status dsm_get_g_storage(dsm_lattice *h, int *form, int *implicit_now) {
  if (!h) return DSM_E_INVAL;
  if (form) *form = h->g_form;
  if (implicit_now) *implicit_now = (h->mom ? h->mstepped : h->g_implicit) ? 1 : 0;
  return DSM_OK;
}

// Raw state (checkpoint): a 256-byte header, then the current buffer's f, g,
// 16-bit g_0, C of the last collision and the g_eq planes, each region
// 256-byte aligned; a state held as moments (implicit = 2) has them in the
// place of f, and the density they belong to in the header; one held as f and
// quads (implicit = 3) has the quads in the place of g.  Restoring it continues
// the run bitwise.
namespace {
constexpr unsigned kStateMagic = 0x53534d44u;  // "DSMS"
struct StateHeader {
  unsigned magic, version;
  int lattice, precision, nx, ny, nz, implicit;
  long long step, pitch;
  double rho;
  int rest;  // implicit = 2: not stepped since dsm_set_fluid
};
struct StateLayout {
  size_t f, g, g0, C, M, total;
};
StateLayout state_layout(const dsm_lattice *h) {
  StateLayout L;
  size_t o = 256;
  auto take = [&](size_t bytes) {
    size_t at = o;
    o += (size_t)round_up((long long)bytes, 256);
    return at;
  };
  const size_t pop = (size_t)h->q * h->pitch * h->tab.store_bytes;
  L.f = take(pop);
  L.g = take(pop);
  L.g0 = take(h->tab.k16 ? h->pitch * sizeof(float) : 0);
  L.C = take(h->pitch * h->tab.real_bytes);
  L.M = take(4 * h->pitch * h->tab.real_bytes);
  L.total = o;
  return L;
}
}  // namespace

dsm_status dsm_state_bytes(dsm_lattice *h, size_t *bytes) {
  if (!h || !bytes) return DSM_E_INVAL;
  *bytes = state_layout(h).total;
  return DSM_OK;
}

dsm_status dsm_get_state(dsm_lattice *h, void *d_dst, size_t bytes) {
  if (!h || !d_dst) return DSM_E_INVAL;
  if (!h->has_fluid) return DSM_E_STATE;
  const StateLayout L = state_layout(h);
  if (bytes < L.total || ((uintptr_t)d_dst & 255u)) return DSM_E_WORKSPACE;
  if (!h->tp && z_unpack(h) != cudaSuccess) return DSM_E_CUDA;
  StateHeader hd;
  memset(&hd, 0, sizeof(hd));
  hd.magic = kStateMagic;
  hd.version = 1;
  hd.lattice = h->kind;
  hd.precision = h->prm.precision;
  hd.nx = h->prm.nx;
  hd.ny = h->prm.ny;
  hd.nz = h->prm.nz;
  hd.implicit = h->mom ? 2 : h->tp ? 3 : h->g_implicit ? 1 : 0;
  hd.rho = h->sp.rho3;
  hd.rest = h->mom && !h->mstepped;
  hd.step = h->step;
  hd.pitch = h->pitch;
  char *d = (char *)d_dst;
  const size_t pop = (size_t)h->q * h->pitch * h->tab.store_bytes;
  const size_t real = h->pitch * h->tab.real_bytes;
  cudaStream_t st = h->stream;
  cudaError_t e = cudaMemcpyAsync(d, &hd, sizeof(hd), cudaMemcpyHostToDevice, st);
  if (h->mom) {
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(d + L.f, h->g[h->mc], mom_reals(h->kind) * real,
                          cudaMemcpyDeviceToDevice, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    return cuda_status(e);
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(d + L.f, h->f[h->cur], pop, cudaMemcpyDeviceToDevice, st);
  if (h->tp) {
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(d + L.g, h->g[h->cur ^ 1], 4 * real, cudaMemcpyDeviceToDevice, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    return cuda_status(e);
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(d + L.g, h->g[h->cur], pop, cudaMemcpyDeviceToDevice, st);
  if (e == cudaSuccess && h->tab.k16)
    e = cudaMemcpyAsync(d + L.g0, h->g0[h->cur], h->pitch * sizeof(float), cudaMemcpyDeviceToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(d + L.C, h->Cb[h->cur], real, cudaMemcpyDeviceToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(d + L.M, h->M, 4 * real, cudaMemcpyDeviceToDevice, st);
  // the header copy reads host stack memory
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  return cuda_status(e);
}

dsm_status dsm_set_state(dsm_lattice *h, const void *d_src, size_t bytes) {
  if (!h || !d_src) return DSM_E_INVAL;
  const StateLayout L = state_layout(h);
  if (bytes < L.total || ((uintptr_t)d_src & 255u)) return DSM_E_WORKSPACE;
  StateHeader hd;
  cudaStream_t st = h->stream;
  cudaError_t e = cudaMemcpyAsync(&hd, d_src, sizeof(hd), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return DSM_E_CUDA;
  if (hd.magic != kStateMagic || hd.version != 1 || hd.lattice != h->kind ||
      hd.precision != h->prm.precision || hd.nx != h->prm.nx || hd.ny != h->prm.ny ||
      hd.nz != h->prm.nz || hd.pitch != h->pitch || hd.implicit < 0 || hd.implicit > 3 ||
      (hd.implicit == 3 && h->kind != DSM_D2Q9) ||
      (hd.implicit == 2 && (!h->tab.mom_expand || !(hd.rho > 0.0))) || hd.step < 0)
    return DSM_E_INVAL;
  const char *d = (const char *)d_src;
  const size_t pop = (size_t)h->q * h->pitch * h->tab.store_bytes;
  const size_t real = h->pitch * h->tab.real_bytes;
  m_drop(h);
  h->cur = 0;
  if (hd.implicit == 2) {
    e = cudaMemcpyAsync(h->g[0], d + L.f, mom_reals(h->kind) * real, cudaMemcpyDeviceToDevice, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(h->err, 0, sizeof(int) * 4, st);
    h->mc = 0;
    h->mom = true;
    h->mstepped = !hd.rest;
    if (e == cudaSuccess && (!m_active(h) || hd.rho != h->sp.rho3)) {
      // a handle that holds its state otherwise: expanded with the density the
      // moments belong to
      MomRaw r = m_raw(h, 0);
      r.rho = hd.rho;
      e = h->tab.mom_expand(r, m_planes(h, 1), 1, st);
      h->cur = 1;
      h->mom = false;
    }
    if (e != cudaSuccess) return DSM_E_CUDA;
    h->step = hd.step;
    h->g_implicit = true;
    h->zpacked = false;
    h->has_fluid = true;
    h->latched = false;
    h->moments_ready = false;
    if (!h->mom && !h->eq) return dsm_set_g_storage(h, h->g_form);
    return DSM_OK;
  }
  e = cudaMemcpyAsync(h->f[0], d + L.f, pop, cudaMemcpyDeviceToDevice, st);
  if (hd.implicit == 3) {
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(h->g[1], d + L.g, 4 * real, cudaMemcpyDeviceToDevice, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(h->err, 0, sizeof(int) * 4, st);
    if (e != cudaSuccess) return DSM_E_CUDA;
    h->tp = true;
    h->step = hd.step;
    h->g_implicit = h->eq;
    h->zpacked = false;
    h->has_fluid = true;
    h->latched = false;
    h->moments_ready = false;
    if (!h->tok) {  // a handle that never steps from quads: the canonical planes
      if (t_copy(h) != cudaSuccess) return DSM_E_CUDA;
      h->tp = h->tcan = false;
    }
    return DSM_OK;
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(h->g[0], d + L.g, pop, cudaMemcpyDeviceToDevice, st);
  if (e == cudaSuccess && h->tab.k16)
    e = cudaMemcpyAsync(h->g0[0], d + L.g0, h->pitch * sizeof(float), cudaMemcpyDeviceToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(h->Cb[0], d + L.C, real, cudaMemcpyDeviceToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(h->M, d + L.M, 4 * real, cudaMemcpyDeviceToDevice, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(h->err, 0, sizeof(int) * 4, st);
  if (e != cudaSuccess) return DSM_E_CUDA;
  h->step = hd.step;
  h->g_implicit = hd.implicit != 0;
  h->zpacked = false;
  h->has_fluid = true;
  h->latched = false;
  h->moments_ready = false;
  // a state holding g as g_eq, restored into a handle that keeps populations
  if (h->g_implicit && !h->eq) return dsm_set_g_storage(h, h->g_form);
  return DSM_OK;
}

dsm_status dsm_fe_scratch_bytes(int lattice, int nx, int ny, int nz, size_t *bytes) {
  if (!bytes || (lattice != DSM_D2Q9 && lattice != DSM_D3Q19) || nx < 1 || ny < 1 || nz < 1)
    return DSM_E_INVAL;
  if (lattice == DSM_D2Q9 && nz != 1) return DSM_E_INVAL;
  *bytes = fe_scratch_bytes(lattice, nx, ny, nz);
  return DSM_OK;
}

dsm_status dsm_fe_energy_grad(const dsm_params *p, const float *d_c1, const float *d_c2,
                              const unsigned char *d_mask, int active, double dP, double kcs,
                              double V0, double fg, double *d_energy, float *d_grad,
                              double *d_terms, void *d_scratch, size_t scratch_bytes,
                              void *cuda_stream) {
  TraceRange trace_range("energy and gradient (K4)");
  if (!p || !d_c1 || !d_c2 || !d_grad || !d_scratch) return DSM_E_INVAL;
  if (active != 1 && active != 2) return DSM_E_INVAL;
  if (active == 1 && !d_mask) return DSM_E_INVAL;
  if (p->lattice != DSM_D2Q9 && p->lattice != DSM_D3Q19) return DSM_E_INVAL;
  if (p->nx < 1 || p->ny < 1 || p->nz < 1 || (p->lattice == DSM_D2Q9 && p->nz != 1))
    return DSM_E_INVAL;
  if ((long long)p->nx * p->ny * p->nz >= (1ll << 31)) return DSM_E_INVAL;
  if (kcs < 0.0) return DSM_E_INVAL;
  double k[3];
  dsm_status s = kappa_of(p, k);
  if (s != DSM_OK) return s;
  if (scratch_bytes < fe_scratch_bytes(p->lattice, p->nx, p->ny, p->nz) ||
      ((uintptr_t)d_scratch & 255u))
    return DSM_E_WORKSPACE;
  FEArgs a;
  s = fe_args_of(p, k, active, fg, &a);
  if (s != DSM_OK) return s;
  a.c1 = d_c1;
  a.c2 = d_c2;
  a.mask = d_mask;
  a.grad = d_grad;
  return cuda_status(fe_launch(p->lattice, a, dP, kcs, V0, d_energy, d_terms, d_scratch,
                               (cudaStream_t)cuda_stream));
}

dsm_status dsm_fe_multi_scratch_bytes(int lattice, int nx, int ny, int nz, int nfluid,
                                      size_t *bytes) {
  if (!bytes || (lattice != DSM_D2Q9 && lattice != DSM_D3Q19) || nx < 1 || ny < 1 || nz < 1)
    return DSM_E_INVAL;
  if (nfluid < 2 || nfluid > FEM_MAX_NF + 1) return DSM_E_INVAL;
  *bytes = fe_multi_scratch_bytes(lattice, nx, ny, nz, nfluid - 1);
  return DSM_OK;
}

dsm_status dsm_fe_energy_grad_multi(const dsm_params *p, int nfluid, const double *kappa,
                                    const float *d_c1, const float *d_c, const double *dP,
                                    const double *kcs, const double *V0, double *d_energy,
                                    float *d_grad, double *d_terms, void *d_scratch,
                                    size_t scratch_bytes, void *cuda_stream) {
  TraceRange trace_range("N-fluid energy and gradient");
  if (!d_c1 || !d_c || !d_grad || !d_scratch) return DSM_E_INVAL;
  FEMArgs a;
  FEMCons cons;
  dsm_status s = fem_args_of(p, nfluid, kappa, dP, kcs, V0, &a, &cons);
  if (s != DSM_OK) return s;
  if (scratch_bytes < fe_multi_scratch_bytes(p->lattice, p->nx, p->ny, p->nz, a.nf) ||
      ((uintptr_t)d_scratch & 255u))
    return DSM_E_WORKSPACE;
  a.c1 = d_c1;
  a.c = d_c;
  a.grad = d_grad;
  return cuda_status(fe_multi_launch(p->lattice, a, cons, d_energy, d_terms, d_scratch,
                                     (cudaStream_t)cuda_stream));
}

dsm_status dsm_vec_scratch_bytes(long long n, size_t *bytes) {
  if (!bytes || n < 0) return DSM_E_INVAL;
  *bytes = vec_scratch_bytes(n);
  return DSM_OK;
}

dsm_status dsm_vec_dot(long long n, const float *d_x, const float *d_y, double *d_out,
                       void *d_scratch, size_t scratch_bytes, void *cuda_stream) {
  if (n < 0 || !d_x || !d_y || !d_out || !d_scratch) return DSM_E_INVAL;
  if (scratch_bytes < vec_scratch_bytes(n)) return DSM_E_WORKSPACE;
  return cuda_status(vec_dot(n, d_x, d_y, d_out, nullptr, d_scratch, (cudaStream_t)cuda_stream));
}

dsm_status dsm_vec_axpy_dev(long long n, double sign, const double *d_a, const double *d_b,
                            const float *d_x, float *d_y, void *cuda_stream) {
  if (n < 0 || !d_a || !d_x || !d_y) return DSM_E_INVAL;
  return cuda_status(vec_axpy_dev(n, sign, d_a, d_b, d_x, d_y, (cudaStream_t)cuda_stream));
}

dsm_status dsm_vec_scale_dev(long long n, const double *d_a, const float *d_x, float *d_y,
                             void *cuda_stream) {
  if (n < 0 || !d_a || !d_x || !d_y) return DSM_E_INVAL;
  return cuda_status(vec_scale_dev(n, d_a, d_x, d_y, (cudaStream_t)cuda_stream));
}

dsm_status dsm_vec_axpby(long long n, double a, const float *d_x, double b, float *d_y,
                         void *cuda_stream) {
  if (n < 0 || !d_x || !d_y) return DSM_E_INVAL;
  return cuda_status(vec_axpby(n, a, d_x, b, d_y, (cudaStream_t)cuda_stream));
}

dsm_status dsm_lbfgs_direction(long long n, int m, const int *order, const float *d_S,
                               const float *d_Y, const double *d_rho, const double *d_gamma,
                               const float *d_g, float *d_r, double *d_alpha, void *d_scratch,
                               size_t scratch_bytes, void *cuda_stream) {
  if (n < 0 || m < 0 || (m > 0 && (!order || !d_S || !d_Y || !d_rho || !d_alpha)) || !d_gamma ||
      !d_g || !d_r || !d_scratch)
    return DSM_E_INVAL;
  if (scratch_bytes < vec_scratch_bytes(n)) return DSM_E_WORKSPACE;
  return cuda_status(lbfgs_direction(n, m, order, d_S, d_Y, d_rho, d_gamma, d_g, d_r, d_alpha,
                                     d_scratch, (cudaStream_t)cuda_stream));
}

dsm_status dsm_vec_dots_scratch_bytes(long long n, int nv, size_t *bytes) {
  if (!bytes || n < 0 || nv < 0) return DSM_E_INVAL;
  *bytes = vec_dots_scratch_bytes(n, nv);
  return DSM_OK;
}

dsm_status dsm_vec_dots(long long n, int nv, const float *d_V, long long stride,
                        const float *d_x, double *d_out, void *d_scratch, size_t scratch_bytes,
                        void *cuda_stream) {
  if (n < 0 || nv < 0 || stride < 0 || (nv > 0 && (!d_V || !d_x || !d_out || !d_scratch)))
    return DSM_E_INVAL;
  if (nv > 1 && stride < n) return DSM_E_INVAL;
  if (scratch_bytes < vec_dots_scratch_bytes(n, nv)) return DSM_E_WORKSPACE;
  return cuda_status(vec_dots(n, nv, d_V, stride, d_x, d_out, d_scratch, (cudaStream_t)cuda_stream));
}

dsm_status dsm_vec_lincomb(long long n, int nv, const float *d_V, long long stride,
                           const double *coef, const float *d_x, double cx, float *d_y,
                           void *cuda_stream) {
  if (n < 0 || nv < 0 || nv > LINCOMB_MAX || stride < 0 || !d_x || !d_y ||
      (nv > 0 && (!d_V || !coef)))
    return DSM_E_INVAL;
  if (nv > 1 && stride < n) return DSM_E_INVAL;
  return cuda_status(vec_lincomb(n, nv, d_V, stride, coef, d_x, cx, d_y, (cudaStream_t)cuda_stream));
}

// Batch admission: common kind, precision, stream and density-contrast flag.
static dsm_status batch_items(dsm_lattice *const *hs, int n, const long long *nsteps,
                              std::vector<BatchRaw> &items) {
  if (!hs || n < 1) return DSM_E_INVAL;
  const dsm_lattice *h0 = hs[0];
  if (!h0) return DSM_E_INVAL;
  items.resize(n);
  for (int i = 0; i < n; i++) {
    const dsm_lattice *h = hs[i];
    if (!h) return DSM_E_INVAL;
    if (has_walls(&h->prm)) return DSM_E_UNSUPPORTED;  // the batched step is periodic
    if (h->kind != h0->kind || h->prm.precision != h0->prm.precision ||
        h->stream != h0->stream || h->sp.rho_contrast != h0->sp.rho_contrast || h->eq != h0->eq)
      return DSM_E_INVAL;
    if (nsteps && (nsteps[i] < 0 || nsteps[i] > (1ll << 30))) return DSM_E_INVAL;
    items[i].r[0] = raw_of(h, 0);
    items[i].r[1] = raw_of(h, 1);
    items[i].nsteps = nsteps ? nsteps[i] : 0;
    items[i].cur0 = h->cur;
  }
  return DSM_OK;
}

// Scratch of a batched call: of the population form's launch over all handles,
// and of the launch on moments over those that can take it.
static size_t batch_need(dsm_lattice *const *hs, int n, const std::vector<BatchRaw> &items) {
  int m = 0;
  for (int i = 0; i < n; i++) m += hs[i]->mok;
  size_t b = (size_t)round_up((long long)hs[0]->tab.batch_bytes(items.data(), n), 256);
  if (m) b += hs[0]->tab.mom_batch_bytes(m);
  return b;
}

dsm_status dsm_batch_scratch_bytes(dsm_lattice *const *hs, int n, size_t *bytes) {
  if (!bytes) return DSM_E_INVAL;
  std::vector<BatchRaw> items;
  dsm_status s = batch_items(hs, n, nullptr, items);
  if (s != DSM_OK) return s;
  *bytes = batch_need(hs, n, items);
  return DSM_OK;
}

dsm_status dsm_batch_step(dsm_lattice *const *hs, int n, const long long *nsteps, void *d_scratch,
                          size_t scratch_bytes) {
  TraceRange trace_range("batched step (K9)");
  if (!nsteps || !d_scratch) return DSM_E_INVAL;
  std::vector<BatchRaw> items;
  dsm_status s = batch_items(hs, n, nsteps, items);
  if (s != DSM_OK) return s;
  for (int i = 0; i < n; i++)
    if (!hs[i]->has_fluid || hs[i]->latched) return DSM_E_STATE;
  if (scratch_bytes < batch_need(hs, n, items) || ((uintptr_t)d_scratch & 255u))
    return DSM_E_WORKSPACE;
  const LBTable &tab = hs[0]->tab;
  cudaStream_t st = hs[0]->stream;
  // lattices stepped on moments, and the others: a launch of each kind
  std::vector<MomBatchRaw> mi;
  std::vector<BatchRaw> pi;
  std::vector<long long> left(nsteps, nsteps + n);
  for (int i = 0; i < n; i++) {
    dsm_lattice *h = hs[i];
    if (z_unpack(h) != cudaSuccess) return DSM_E_CUDA;
    if (!m_active(h)) {
      if (m_leave(h) != cudaSuccess) return DSM_E_CUDA;
      BatchRaw b = items[i];  // (leaving may have moved the current buffer)
      b.r[0] = raw_of(h, 0);
      b.r[1] = raw_of(h, 1);
      b.cur0 = h->cur;
      pi.push_back(b);
      continue;
    }
    if (left[i] > 0 && !h->mom && !(h->mfit && h->g_implicit)) {
      // a state given as populations: its first step as dsm_step takes it
      LBRaw a = raw_of(h, h->cur);
      if (tab.moments(a, st) != cudaSuccess || tab.node(a, 2, MODE_STEP, st) != cudaSuccess)
        return DSM_E_CUDA;
      h->cur ^= 1;
      h->step++;
      h->g_implicit = h->mfit = true;
      h->moments_ready = h->tp = h->tcan = false;
      left[i]--;
    }
    if (left[i] == 0) continue;
    if (!h->mom && m_enter(h) != cudaSuccess) return DSM_E_CUDA;
    if (m_statics(h) != cudaSuccess) return DSM_E_CUDA;
    MomBatchRaw b;
    b.r[0] = m_raw(h, 0);
    b.r[1] = m_raw(h, 1);
    b.nsteps = left[i];
    b.cur0 = h->mc;
    mi.push_back(b);
  }
  size_t used = 0;
  if (!pi.empty()) {
    used = (size_t)round_up((long long)tab.batch_bytes(pi.data(), (int)pi.size()), 256);
    if (tab.batch(pi.data(), (int)pi.size(), d_scratch, scratch_bytes, hs[0]->sp.rho_contrast != 0,
                  hs[0]->eq, g_wait_limit, st) != cudaSuccess)
      return DSM_E_CUDA;
  }
  if (!mi.empty() && tab.mom_batch(mi.data(), (int)mi.size(), (char *)d_scratch + used,
                                   scratch_bytes - used, g_wait_limit, st) != cudaSuccess)
    return DSM_E_CUDA;
  for (int i = 0; i < n; i++) {
    dsm_lattice *h = hs[i];
    h->moments_ready = false;
    h->step += left[i];
    if (left[i] == 0) continue;
    if (m_active(h)) {
      h->mc ^= (int)(left[i] & 1);
      h->mcp = h->mpk = false;
      h->mstepped = true;
    } else {
      h->tp = h->tcan = false;
      h->cur ^= (int)(left[i] & 1);
      h->g_implicit = h->eq;
      h->mfit = h->mok && h->eq;
    }
  }
  return DSM_OK;
}

dsm_status dsm_set_wait_limit(unsigned long long polls) {
  g_wait_limit = polls;
  return DSM_OK;
}

dsm_status dsm_destroy(dsm_lattice *h) {
  if (!h) return DSM_E_INVAL;
  delete h;
  return DSM_OK;
}

}  // extern "C"
