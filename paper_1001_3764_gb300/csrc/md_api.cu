// md_api.cu -- host runtime and C ABI of the GB300 MD engine (include/md.h).
//
// One md_system owns: a replica table, tile tables, every device buffer (one
// allocation, or a caller workspace), a stream, and a CUDA graph holding one
// rebin cycle (rebin + neighbour list + rebin_every steps).  Kernels are in
// k_bin.cu (binning), k_lj.cu (neighbour list and Lennard-Jones), k_step.cu
// (bonded forces and update of a step), k_force.cu (bonded terms of the
// read-outs), k_integrate.cu (opening update, kinetic energy, energy
// reductions, chain observables, state transfer), k_observe.cu (RDF, ACF) and
// md_adjoint.cu (the adjoint); md_static.cu holds the allocation-free binning
// entry point.  bonded.cuh, integrate.cuh and cell_order.cuh hold what several
// of them share.
#include <algorithm>
#include <array>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <tuple>
#include <cstring>
#include <string>
#include <vector>
#include <cuda.h>

#include "../../include/md.h"
#include "md_kernels.cuh"

using namespace mdg;

namespace {

constexpr int kIntTile = 224;    // atoms per integrator / bonded block (original order)
constexpr int kNumProf = 5;      // rebin, neighbour build, integrate, lj, bonded
constexpr double kKB = 0.0083144626;

thread_local std::string g_create_error;

size_t align256(size_t b) { return (b + 255) & ~size_t(255); }

}  // namespace

struct md_system {
  // configuration
  int n_reps = 0, S = 0, R = 10;
  int64_t N = 0;
  int C = 0, Npad = 0, cap = 0;
  bool mixed = false;
  int thermo = 0;                 // MD_NVE, MD_VRESCALE or MD_NOSE_HOOVER
  double dt = 0, rc = 0, skin = 0, tau = 0.1;
  md_params params{};
  ForceParams fp{};
  std::vector<RepDev> reps_h;
  std::vector<Tile> t_int;                   // kIntTile atoms each
  std::vector<Tile> t_chain;                 // whole chains or molecules (fused step kernels)
  std::vector<double> T0;
  // memory
  char* base = nullptr;
  size_t bytes = 0;
  bool own_mem = false;
  RepDev* reps = nullptr;
  Tile *tiles_int = nullptr, *tiles_chain = nullptr;
  void *x = nullptr, *v = nullptr, *F = nullptr;
  long long* flj[2] = {nullptr, nullptr};    // LJ force, int64 SoA [3][Npad], sorted order: a step adds to one
                                             // while the other is cleared for the next
  int* img = nullptr;
  uint16_t* site = nullptr;
  int *cellc = nullptr, *inv_perm = nullptr, *tag = nullptr, *perm = nullptr;
  float4 *ref = nullptr, *pos = nullptr;
  unsigned* list = nullptr;                  // cluster lists [n_cl_max][cap]
  int* ncl = nullptr;                        // entries per cluster
  int* cl_start = nullptr;                   // first cluster of each cell [C + 1]
  int64_t n_cl_max = 0;
  int n_regions = 0;
  std::vector<RegionShape> shapes_h;
  int* region_cells = nullptr;
  RegionShape* shapes = nullptr;
  std::vector<ItemRun> runs_h;               // what the items are made from (launch_plan)
  ItemRun* runs = nullptr;
  WorkItem* items = nullptr;                 // blocks of the LJ kernel, then those of the list build
  int n_lj_items = 0, n_build_items = 0;
  ClusterTask* tasks = nullptr;              // each LJ item's clusters in task order, from task_base[item] on
  int *task_base = nullptr, *n_tasks = nullptr, *big = nullptr;
  int tile_cap = 0, lj_cap = 0;              // atoms of a tile: list build, first force launch
  int lj_block = 256, persistent_grid = 0;   // persistent_grid > 0: fixed grid for the LJ kernel
  int lj_lanes = 8;                          // lanes per 4-atom cluster in the LJ kernel
  int lj_region = 3;                         // cells per side (x, y) of an LJ / list region
  bool lj_pair_exact = false;                // each LJ pair force converted once, +q to i and -q to j
  int* work = nullptr;                       // LJ work counters (persistent schedule)
  int *count = nullptr, *cell_start = nullptr, *cell_of = nullptr, *scan_seg = nullptr;
  int *slot = nullptr, *tmp = nullptr;
  double *lj_part = nullptr, *b_part = nullptr, *kepart = nullptr, *ke_out = nullptr, *lam = nullptr;
  double* e_out = nullptr;
  double* e_slices = nullptr;   // first-pass energy sums, n_reps * max_slices * 11
  int max_slices = 1;
  double* stage = nullptr;                   // input staging (6N doubles)
  unsigned* flags = nullptr;
  // end-to-end vector ACF (allocated by md_acf_reset)
  double *acf_ring = nullptr, *acf_acc = nullptr;
  int acf_lag = -1;
  int64_t acf_n = 0;
  // execution
  cudaStream_t st = nullptr;
  bool own_stream = false;
  cudaGraphExec_t cycle = nullptr;
  cudaGraphExec_t cycle_fresh = nullptr;     // the same cycle without its leading rebin + list
  std::vector<cudaGraphExec_t> rem_graphs;   // blocks of k < R steps (remainders), captured on first use
  cudaStream_t side = nullptr;               // captures the bodies of the conditional rebins
  unsigned long long* early = nullptr;       // early rebins (displacement beyond skin/2) so far
  int* ctl = nullptr;                        // early rebin within a block of steps (StepGate)
  // a general molecule type (md_desc.topology), or linear chains
  bool generic = false;
  int disp = MD_DISP_REBUILD;                // what a displacement beyond skin/2 does
  std::vector<unsigned char> mtype_h;        // type of each atom of the molecule
  std::vector<int> t_boff, t_bat, t_aoff, t_aat, t_doff, t_dat, t_xoff, t_xat;   // term and exclusion lists
  std::vector<ushort4> t_terms;
  unsigned char* mtype = nullptr;            // device copies
  TopoDev topo{};
  bool fresh = false;                        // bins, list and forces are those of the current positions
  bool profile = false;
  std::vector<cudaEvent_t> ev;
  int ev_used = 0;
  double prof_ms[kNumProf] = {0, 0, 0, 0, 0};
  int64_t prof_n[kNumProf] = {0, 0, 0, 0, 0};
  std::string err;
};

void md_set_global_error(const char* msg) { g_create_error = msg; }

// ------------------------------------------------------------------ helpers
static int fail(md_system* s, int code, const std::string& msg) {
  if (s) s->err = msg; else g_create_error = msg;
  if (code == MD_ECUDA || code == MD_ENOMEM) cudaGetLastError();   // reported: not left to the next call
  return code;
}
#define CU(call)                                                                                      \
  do {                                                                                                \
    cudaError_t e_ = (call);                                                                          \
    if (e_ != cudaSuccess) return fail(s, MD_ECUDA, std::string(#call ": ") + cudaGetErrorString(e_)); \
  } while (0)

// constants of the replicas' thermostats (T0, dt, tau, masses)
static void fill_thermostats(md_system* s) {
  for (RepDev& q : s->reps_h) {
    const double m0 = s->params.mass[0], Qm = s->tau * s->tau * q.T0 / (4.0 * M_PI * M_PI);
    q.t_scale = m0 / (q.dof * kKB);
    q.vr_num = s->dt / s->tau * q.T0 * q.dof * kKB / m0;
    q.nh_rate = s->dt / Qm;
    q.com_scale = m0 / ((double)q.n_chains * s->fp.mol_mass);
  }
}

static void fill_force_params(md_system* s) {
  const md_params& p = s->params;
  ForceParams& f = s->fp;
  for (RepDev& q : s->reps_h)
    for (int t = 0; t < 3; ++t) {
      const int a = t >= 1 ? 1 : 0, b = t >= 2 ? 1 : 0;
      const int ta = (t == 1) ? 0 : a;   // pair (0,1) for t = 1
      const int tb = (t == 1) ? 1 : b;
      double eps = std::sqrt(p.eps[ta] * p.eps[tb]);
      double sig = std::sqrt(p.sigma[ta] * p.sigma[tb]) * q.inv_h;   // sigma in cell units
      double s6 = sig * sig * sig * sig * sig * sig;
      q.C6u[t] = (float)(4.0 * eps * s6);
      q.C12u[t] = (float)(4.0 * eps * s6 * s6);
    }
  for (int a = 0; a < 2; ++a)
    for (int b = 0; b < 2; ++b) {
      double eps = std::sqrt(p.eps[a] * p.eps[b]);
      double sig = std::sqrt(p.sigma[a] * p.sigma[b]);
      double s6 = sig * sig * sig * sig * sig * sig;
      double c6 = 4.0 * eps * s6, c12 = 4.0 * eps * s6 * s6;
      double ir6 = 1.0 / (s->rc * s->rc * s->rc * s->rc * s->rc * s->rc);
      f.c6[a][b] = (float)c6;
      f.c12[a][b] = (float)c12;
      f.erc[a][b] = (float)(c12 * ir6 * ir6 - c6 * ir6);
    }
  f.rc2 = (float)(s->rc * s->rc);
  f.rlist2 = (float)((s->rc + s->skin) * (s->rc + s->skin));
  f.kb = (float)p.kb; f.b0 = (float)p.b0; f.ka = (float)p.ka; f.theta0 = (float)p.theta0;
  f.kphi = (float)p.kphi; f.phis = (float)p.phis; f.n_mult = p.n_mult;
  f.sites = s->S;
  f.half_skin2 = (float)(0.25 * s->skin * s->skin);
  f.b0sq = p.b0 * p.b0;
  f.b0sq_hi = (float)f.b0sq;
  f.b0sq_lo = (float)(f.b0sq - (double)f.b0sq_hi);
  for (int a = 0; a < 2; ++a) {
    f.mass[a] = p.mass[a];
    f.inv_mass[a] = 1.0 / p.mass[a];
    f.mass_ratio = p.mass[1] / p.mass[0];
    f.hdt_m[a] = 0.5 * s->dt / p.mass[a];
    f.hdt_m_fix[a] = f.hdt_m[a] * kFixInv;
    f.hdt_m_f[a] = (float)f.hdt_m[a];
  }
  f.dt_f = (float)s->dt;
  f.dt = s->dt;
  if (s->generic) {
    double mm = 0.0;
    for (unsigned char t : s->mtype_h) mm += p.mass[t];
    f.mol_mass = mm;
  } else {
    f.mol_mass = (double)(s->S - 2) * p.mass[0] + 2.0 * p.mass[1];
  }
  f.mtype = s->generic ? s->mtype : nullptr;
  fill_thermostats(s);
}

// Region shapes: sx x sy x 1 home cells (sx, sy in 1 .. G; shape id
// (sx - 1) + G (sy - 1)).  The tile lists the cells that the home cells and
// their 13 forward offsets take up, rows of x one after another: the layer above,
// then the home layer.  So a home cell's forward cells are five runs of
// consecutive tile cells.  nb[h] gives home cell h's own tile cell and its 13
// forward tile cells, in the offset order (dz = +1 layer: dy = +1, 0, -1, each
// dx = -1, 0, 1; then dz = 0, dy = +1; then (+1, 0, 0)).
static RegionShape make_shape(int sx, int sy) {
  RegionShape S{};
  std::vector<std::array<int, 3>> tile;
  for (int y = -1; y <= sy; ++y)
    for (int x = -1; x <= sx; ++x) tile.push_back({x, y, 1});
  for (int y = 0; y <= sy; ++y)
    for (int x = y == 0 ? 0 : -1; x <= sx; ++x) tile.push_back({x, y, 0});
  S.n_home = sx * sy;
  std::vector<std::array<int, 3>> fw;
  for (int dz = -1; dz <= 1; ++dz)
    for (int dy = -1; dy <= 1; ++dy)
      for (int dx = -1; dx <= 1; ++dx)
        if (dz > 0 || (dz == 0 && dy > 0) || (dz == 0 && dy == 0 && dx > 0)) fw.push_back({dx, dy, dz});
  std::sort(fw.begin(), fw.end(), [](const std::array<int, 3>& a, const std::array<int, 3>& b) {
    return std::make_tuple(-a[2], -a[1], a[0]) < std::make_tuple(-b[2], -b[1], b[0]);
  });
  for (int h = 0; h < S.n_home; ++h) {
    const std::array<int, 3> home = {h % sx, h / sx, 0};
    auto index = [&](const std::array<int, 3>& c) {
      return (unsigned char)(std::find(tile.begin(), tile.end(), c) - tile.begin());
    };
    S.nb[h][0] = index(home);
    for (int q = 0; q < 13; ++q) S.nb[h][q + 1] = index({home[0] + fw[q][0], home[1] + fw[q][1], home[2] + fw[q][2]});
  }
  S.n_tile = (int)tile.size();
  for (int k = 0; k < S.n_tile; ++k)
    for (int a = 0; a < 3; ++a) S.off[k][a] = (signed char)tile[k][a];
  S.cx = 0.5f * (float)(sx - 1);
  S.cy = 0.5f * (float)(sy - 1);
  S.cz = 0.f;
  return S;
}

// Regions of G x G x 1 cells over every replica (narrower at the high faces
// when G does not divide M) and the runs of their work items.
static void plan_regions(md_system* s, bool grid_schedule) {
  const int G = s->lj_region;
  // Where two of the largest tiles do not fit an SM's shared memory (cells
  // above 1.22 nm) but two of the usual ones do: the force kernel's tile is
  // the one that fits twice, and items of larger tiles are left to a second
  // launch: those of the replicas whose mean tile is within 12% of it (a melt's
  // tiles differ by 3%), at most half of the atoms, and dense parts of an
  // uneven box.  For systems of more rows than resident blocks; smaller ones
  // are split.  Else one block of 24 warps an SM.  64 replicas, 1.5M sites,
  // skin 0.12 nm: LJ 484 us with one block an SM, 357 + 19 now.
  s->lj_cap = s->tile_cap;
  std::vector<char> large(s->n_reps, 0);
  if (G == 3 && (!s->lj_block || s->lj_block == 384) && grid_schedule && lj_tiles_per_sm(s->tile_cap) == 1) {
    const int two = lj_tile_cap_for(2);
    int64_t rows = 0, large_atoms = 0;
    for (int r = 0; r < s->n_reps; ++r) {
      const RepDev& q = s->reps_h[r];
      const double cell = std::max(q.n_atoms / (q.L * q.L * q.L), 33.0) * q.h * q.h * q.h;
      large[r] = 1.12 * s->shapes_h.back().n_tile * cell + 64.0 > two;
      if (large[r]) large_atoms += q.n_atoms;
      rows += (int64_t)q.M * q.M * ((q.M + G - 1) / G);
    }
    if (rows > 2 * kSMs && 2 * large_atoms <= s->N) s->lj_cap = two;
    else large.assign(s->n_reps, 0);
  }
  int n_rows = 0, n_cells = 0, R = 0;
  for (RepDev& q : s->reps_h) {
    const int nx = (q.M + G - 1) / G;
    q.region_off = R;
    R += nx * nx * q.M;
    n_rows += nx * q.M * q.M;
    n_cells += q.M * q.M * q.M;
  }
  s->n_regions = R;
  // regions of a shape in a replica
  const int n_shapes = (int)s->shapes_h.size();
  auto regions_of = [&](int r, int shape) {
    auto along = [&](int side) { return side == G ? s->reps_h[r].M / G : s->reps_h[r].M % G == side ? 1 : 0; };
    return along(shape % G + 1) * along(shape / G + 1) * s->reps_h[r].M;
  };
  // Work items, the regions with most cells first (narrow regions fill the
  // tail: LJ 137.6 -> 128.1 us at 506k sites, M = 22, 47.8 -> 37.6 at 120k).
  // A system of few regions is split, since a block spends 6 us on set-up
  // and tail and 1.5 us per home cell, and two fit an SM.  LJ, us per launch:
  //   cells while all are resident at once: 24.6 -> 14.2 at 1,500 sites, 27.8 -> 16.2 at 12,000
  //   rows likewise (else whole): 25.6 -> 16.3 at 18,750, 24.8 -> 21.2 at 35,100; whole 47.7, rows 65.3 at 150k
  //   between 1 and 2 regions per SM: rows from the second on (35.9 -> 27.4 at 84,000, M = 12)
  std::vector<int> order(n_shapes);
  for (int k = 0; k < n_shapes; ++k) order[k] = k;
  std::stable_sort(order.begin(), order.end(),
                   [s](int a, int b) { return s->shapes_h[a].n_home > s->shapes_h[b].n_home; });
  s->runs_h.clear();
  int n_items = 0;
  // rows of home cells a block takes (0: a single cell)
  auto add_run = [&](int r, int shape, int region0, int count, int rows, int parts) {
    if (count <= 0) return;
    const int n_home = s->shapes_h[shape].n_home;
    const int step = std::min(n_home, rows > 0 ? rows * (shape % G + 1) : 1);
    s->runs_h.push_back(ItemRun{n_items, r, shape, region0, step, parts});
    n_items += count * ((n_home + step - 1) / step) * parts;
  };
  constexpr int kWhole = 255;
  const int per_sm = lj_tiles_per_sm(s->lj_cap), slots = per_sm * kSMs;
  const int lj_rows = n_cells <= slots ? 0 : n_rows <= slots ? 1 : kWhole;
  // default block: 24 warps an SM, as two resident blocks where two tiles fit
  // the shared memory of an SM, else as one (cells above 1.22 nm: LJ 565 ->
  // 478 us for 64 replicas at skin 0.12 nm); three of 8 warps for 2 x 2 regions
  if (!s->lj_block) s->lj_block = G == 2 ? 256 : per_sm >= 2 || lj_rows != kWhole ? 384 : 768;
  // the second launch takes one block of 24 warps an SM: its items are whole
  // regions, rows or cells, by how many there are
  int n_large = 0;
  for (int r = 0; r < s->n_reps; ++r)
    if (large[r]) n_large += regions_of(r, n_shapes - 1);
  const int large_rows = 9 * n_large <= kSMs ? 0 : 3 * n_large <= kSMs ? 1 : kWhole;
  int q = 0;   // regions so far
  for (int shape : order)
    for (int r = 0; r < s->n_reps; ++r) {
      const int n = regions_of(r, shape);
      if (large[r] && shape == n_shapes - 1) {
        add_run(r, shape, 0, n, large_rows, 1);
      } else if (lj_rows == kWhole && per_sm >= 2 && R <= slots) {
        const int whole = std::max(0, std::min(n, kSMs - q));
        add_run(r, shape, 0, whole, kWhole, 1);
        add_run(r, shape, whole, n - whole, 1, 1);
      } else {
        add_run(r, shape, 0, n, lj_rows, 1);
      }
      q += n;
    }
  s->n_lj_items = n_items;
  // The list build gives a warp a cluster at a time (7 us alone), 32 warps an
  // SM.  With the task order, us (whole regions / rows / cells / cells in 3 parts):
  //   - / 31 / 21 / 18.6 at 1,500 sites, 67 / 35 / 23 / 18.8 at 6,000, 62 / 33 / 26 / 31 at 12,000 (216 cells),
  //   82 / 56 / 54 at 64,800 (176 regions), 102 / 89 / 94 at 150k (375), 232 / 213 / 243 at 444k (1,029),
  //   236 / 243 / 272 at 506k (1,408), 317 / 336 / 388 at 737k (2,025), 609 / 639 / 774 at 1.5M;
  // between 600 and 1,800 regions the last wave decides, by up to 8% either way
  const int parts = n_cells <= 128 ? 3 : 1;
  for (int shape : order)
    for (int r = 0; r < s->n_reps; ++r)
      add_run(r, shape, 0, regions_of(r, shape), R >= 12 * kSMs ? kWhole : R >= 2 * kSMs ? 1 : 0, parts);
  s->n_build_items = n_items - s->n_lj_items;
}

// The per-type lists of Sec. 3.3 from a molecule's bond graph: each atom's
// neighbours (ascending); exclusions = 1-2 and 1-3 neighbours; angles = every
// path a-b-c (vertex b, a < c), listed under a; dihedrals = every path
// a-b-c-d around each bond b-c (in bond order, b < c), listed under a; bonds
// listed under their first atom as given.
static int build_topology(md_system* s, const md_topology* t) {
  const int n = t->naom;
  if (n < 4 || n > 1023) return fail(s, MD_EINVAL, "topology: naom must be 4 .. 1023");
  if (t->n_bonds < 1 || t->n_bonds > 4 * n || !t->bonds || !t->types)
    return fail(s, MD_EINVAL, "topology: 1 .. 4 naom bonds, bonds and types required");
  std::vector<std::vector<int>> nb(n);
  std::vector<std::pair<int, int>> bl;
  for (int k = 0; k < t->n_bonds; ++k) {
    const int a = t->bonds[2 * k], b = t->bonds[2 * k + 1];
    if (a < 0 || b < 0 || a >= n || b >= n || a == b) return fail(s, MD_EINVAL, "topology: bond atom out of range");
    for (int c : nb[a])
      if (c == b) return fail(s, MD_EINVAL, "topology: repeated bond");
    nb[a].push_back(b);
    nb[b].push_back(a);
    bl.push_back({a, b});
  }
  for (auto& v : nb) std::sort(v.begin(), v.end());
  s->mtype_h.assign(n, 0);
  for (int a = 0; a < n; ++a) {
    if (t->types[a] != 0 && t->types[a] != 1) return fail(s, MD_EINVAL, "topology: types must be 0 or 1");
    s->mtype_h[a] = (unsigned char)t->types[a];
  }
  std::vector<std::vector<int>> ob(n), oa(n), od(n), ex(n);
  for (auto& e : bl) ob[e.first].push_back(e.second);
  for (int b = 0; b < n; ++b)
    for (size_t p = 0; p < nb[b].size(); ++p)
      for (size_t q = p + 1; q < nb[b].size(); ++q) {
        oa[nb[b][p]].push_back(b);
        oa[nb[b][p]].push_back(nb[b][q]);
      }
  for (auto& e : bl) {
    const int b = std::min(e.first, e.second), c = std::max(e.first, e.second);
    for (int a : nb[b]) {
      if (a == c) continue;
      for (int d : nb[c]) {
        if (d == b || d == a) continue;
        od[a].push_back(b); od[a].push_back(c); od[a].push_back(d);
      }
    }
  }
  for (int a = 0; a < n; ++a) {
    for (int b : nb[a]) {
      ex[a].push_back(b);
      for (int c : nb[b])
        if (c != a) ex[a].push_back(c);
    }
    std::sort(ex[a].begin(), ex[a].end());
    ex[a].erase(std::unique(ex[a].begin(), ex[a].end()), ex[a].end());
  }
  auto csr = [n](const std::vector<std::vector<int>>& v, std::vector<int>& off, std::vector<int>& at) {
    off.assign(n + 1, 0);
    at.clear();
    for (int a = 0; a < n; ++a) { at.insert(at.end(), v[a].begin(), v[a].end()); off[a + 1] = (int)at.size(); }
    if (at.empty()) at.push_back(0);
  };
  csr(ob, s->t_boff, s->t_bat);
  csr(oa, s->t_aoff, s->t_aat);
  csr(od, s->t_doff, s->t_dat);
  csr(ex, s->t_xoff, s->t_xat);
  // the CSR offsets of angles and dihedrals count ints; the kernels index terms
  for (int& o : s->t_aoff) o /= 2;
  for (int& o : s->t_doff) o /= 3;
  auto terms = [&](const std::vector<std::vector<int>>& v, size_t m) {
    for (int a = 0; a < n; ++a)
      for (size_t q = 0; q < v[a].size(); q += m)
        s->t_terms.push_back({(unsigned short)a, (unsigned short)v[a][q], (unsigned short)(m > 1 ? v[a][q + 1] : 0),
                              (unsigned short)(m > 2 ? v[a][q + 2] : 0)});
  };
  s->t_terms.clear();
  terms(ob, 1);
  terms(oa, 2);
  terms(od, 3);
  return MD_OK;
}

// Validate the descriptor and fill geometry, tiles and sizes (no device work).
static int configure(md_system* s, const md_desc* d) {
  if (!d) return fail(s, MD_EINVAL, "null descriptor");
  if (d->n_replicas < 1 || d->n_replicas > kMaxReplicas) return fail(s, MD_EINVAL, "n_replicas out of range");
  // chains: the packed tags keep the site in 10 bits, and the last site of one
  // chain must stay more than 2 away from the next chain's first (1024 - S + 1 > 2)
  if (d->sites_per_chain < 4 || d->sites_per_chain > (d->topology ? 1023 : 1022))
    return fail(s, MD_EINVAL, "sites_per_chain must be 4..1022 (4..1023 with a topology)");
  s->generic = d->topology != nullptr;
  if (s->generic) {
    if (d->topology->naom != d->sites_per_chain) return fail(s, MD_EINVAL, "sites_per_chain must equal topology->naom");
    if (d->precision != MD_MIXED) return fail(s, MD_EINVAL, "a molecule topology needs the mixed precision form");
    const int rc = build_topology(s, d->topology);
    if (rc) return rc;
  } else {
    s->mtype_h.assign(d->sites_per_chain, 0);
    s->mtype_h[0] = s->mtype_h[d->sites_per_chain - 1] = 1;
  }
  if (!d->n_chains || !d->box) return fail(s, MD_EINVAL, "n_chains and box are required");
  if (!(d->dt > 0) || !(d->rc > 0) || !(d->skin >= 0) || d->rebin_every < 1)
    return fail(s, MD_EINVAL, "dt, rc must be > 0, skin >= 0, rebin_every >= 1");
  if (d->precision != MD_PLAIN_FP32 && d->precision != MD_MIXED) return fail(s, MD_EINVAL, "unknown precision");
  if (d->thermostat != MD_NVE && d->thermostat != MD_VRESCALE && d->thermostat != MD_NOSE_HOOVER)
    return fail(s, MD_EINVAL, "unknown thermostat");
  if (d->thermostat != MD_NVE && (!d->T_target || !(d->tau_t > 0)))
    return fail(s, MD_EINVAL, "thermostat needs T_target and tau_t > 0");
  for (int a = 0; a < 2; ++a)
    if (!(d->params.mass[a] > 0) || !(d->params.sigma[a] > 0) || !(d->params.eps[a] >= 0))
      return fail(s, MD_EINVAL, "masses and sigmas must be > 0, eps >= 0");
  if (d->params.n_mult < 0 || d->params.n_mult > 12) return fail(s, MD_EINVAL, "n_mult out of range");
  s->n_reps = d->n_replicas;
  s->S = d->sites_per_chain;
  s->R = d->rebin_every;
  s->mixed = d->precision == MD_MIXED;
  s->thermo = d->thermostat;
  s->dt = d->dt; s->rc = d->rc; s->skin = d->skin; s->tau = d->thermostat ? d->tau_t : 0.1;
  if (d->lj_block != 0 && d->lj_block != 128 && d->lj_block != 256 && d->lj_block != 384)
    return fail(s, MD_EINVAL, "lj_block must be 0, 128, 256 or 384");
  if (d->schedule != MD_SCHED_GRID && d->schedule != MD_SCHED_PERSISTENT) return fail(s, MD_EINVAL, "unknown schedule");
  if (d->lj_lanes != 0 && d->lj_lanes != 8 && d->lj_lanes != 16 && d->lj_lanes != 32)
    return fail(s, MD_EINVAL, "lj_lanes must be 0, 8, 16 or 32");
  s->lj_lanes = d->lj_lanes ? d->lj_lanes : 8;
  if (d->lj_region != 0 && d->lj_region != 2 && d->lj_region != 3)
    return fail(s, MD_EINVAL, "lj_region must be 0, 2 or 3");
  s->lj_region = d->lj_region ? d->lj_region : 3;
  if (d->lj_pair_exact != 0 && d->lj_pair_exact != 1) return fail(s, MD_EINVAL, "lj_pair_exact must be 0 or 1");
  s->lj_pair_exact = d->lj_pair_exact == 1;
  s->lj_block = d->lj_block;   // 0: set with the regions
  if (d->displacement != MD_DISP_REBUILD && d->displacement != MD_DISP_ERROR)
    return fail(s, MD_EINVAL, "displacement must be MD_DISP_REBUILD or MD_DISP_ERROR");
  s->disp = d->displacement;
  s->params = d->params;
  const double rl = d->rc + d->skin;
  s->reps_h.assign(s->n_reps, RepDev{});
  s->T0.assign(s->n_reps, 0.0);
  int64_t atoms = 0, cells = 0, chains = 0;
  double max_expected = 0.0, max_tile = 0.0;
  // regions of G x G x 1 cells (narrower at the high faces when G does not divide M)
  const int G = s->lj_region;
  s->shapes_h.clear();
  for (int sy = 1; sy <= G; ++sy)
    for (int sx = 1; sx <= G; ++sx) s->shapes_h.push_back(make_shape(sx, sy));
  const double tile_cells = (double)s->shapes_h.back().n_tile;
  s->t_int.clear();
  s->t_chain.clear();
  for (int r = 0; r < s->n_reps; ++r) {
    const int nc = d->n_chains[r];
    const double L = d->box[r];
    if (nc < 1) return fail(s, MD_EINVAL, "every replica needs at least one chain");
    if (!(L > 0) || !std::isfinite(L)) return fail(s, MD_EINVAL, "box sides must be positive");
    const int M = (int)std::floor(L / rl);
    if (M < 3) return fail(s, MD_EINVAL, "box side must be at least 3 (rc + skin)");
    if (M > 1023) return fail(s, MD_EINVAL, "more than 1023 cells per side");
    RepDev& q = s->reps_h[r];
    q.L = L; q.M = M; q.h = L / M; q.inv_h = (double)M / L; q.half_L = 0.5 * L;
    q.Lf = (float)L; q.hf = (float)q.h; q.half_Lf = (float)(0.5 * L); q.Mf = (float)M;
    q.ih_hi = (float)q.inv_h; q.ih_lo = (float)(q.inv_h - (double)q.ih_hi);
    q.rc2u = (float)(d->rc * d->rc * q.inv_h * q.inv_h);
    q.rlist2u = (float)(rl * rl * q.inv_h * q.inv_h);
    q.hs2u = (float)(0.25 * d->skin * d->skin * q.inv_h * q.inv_h);
    q.cell_base = (int)cells; q.atom_off = (int)atoms;
    q.n_atoms = nc * s->S; q.n_chains = nc; q.chain_off = (int)chains;
    q.T0 = d->T_target ? d->T_target[r] : 0.0;
    q.dof = 3.0 * q.n_atoms - 3.0;
    s->T0[r] = q.T0;
    q.tile_off = (int)s->t_int.size();
    for (int o = 0; o < q.n_atoms; o += kIntTile) s->t_int.push_back(Tile{q.atom_off + o, std::min(kIntTile, q.n_atoms - o), r, 0});
    q.n_tiles = (int)s->t_int.size() - q.tile_off;
    q.ctile_off = (int)s->t_chain.size();
    const int per = step_chains_per_block(s->S, s->generic) * s->S;
    for (int o = 0; o < q.n_atoms; o += per)
      s->t_chain.push_back(Tile{q.atom_off + o, std::min(per, q.n_atoms - o), r, 0});
    q.n_ctiles = (int)s->t_chain.size() - q.ctile_off;
    // chains are locally as dense as a melt even in a sparse box, so the
    // density used for the capacity is at least that of a dense melt
    const double rho = std::max(q.n_atoms / (L * L * L), 40.0);
    max_expected = std::max(max_expected, 4.0 / 3.0 * M_PI * rl * rl * rl * rho);
    max_tile = std::max(max_tile, tile_cells * std::max(q.n_atoms / (L * L * L), 33.0) * q.h * q.h * q.h);
    atoms += q.n_atoms; cells += (int64_t)M * M * M; chains += nc;
    s->max_slices = std::max(s->max_slices, energy_slice_count(M * M * M));
    if (atoms >= (int64_t)kNbrIndexMask) return fail(s, MD_EINVAL, "too many atoms (limit 2^26)");
    if (chains >= (1 << 20)) return fail(s, MD_EINVAL, "too many chains (limit 2^20)");
    if (cells >= (1 << 26)) return fail(s, MD_EINVAL, "too many cells");
  }
  s->N = atoms; s->C = (int)cells;
  // tile capacity (shared memory per block): 1.4x the mean tile of
  // the densest replica (at least melt density, 33 sites/nm^3) plus 64, in
  // multiples of 128 atoms; a larger tile is reported as MD_EOVERFLOW
  s->tile_cap = std::min(tile_capacity_max(), ((int)std::ceil(1.4 * max_tile + 64.0) + 127) / 128 * 128);
  plan_regions(s, d->schedule == MD_SCHED_GRID);
  s->n_cl_max = (atoms + 3 * cells) / 4 + 1;   // sum of ceil(n_c / 4) over the cells
  s->Npad = (int)((atoms + 31) / 32 * 32);
  // default list capacity (entries per 4-atom cluster): a cluster's list holds
  // about 0.75 x the atoms within rc + skin of one atom at melt density
  // (~135 in the benchmark melt, at most ~350); 2.5 x that plus 64
  s->cap = d->nbr_capacity > 0 ? d->nbr_capacity : (int)std::ceil(2.5 * 0.75 * max_expected + 64.0);
  s->cap = (s->cap + 31) / 32 * 32;
  if (s->cap > 4096) return fail(s, MD_EINVAL, "neighbour capacity above 4096");
  fill_force_params(s);
  return MD_OK;
}

// Lay out every buffer; with base == nullptr only the size is computed.
static size_t plan(md_system* s, char* base) {
  size_t off = 0;
  auto take = [&](size_t b) -> char* { char* p = base ? base + off : nullptr; off += align256(b); return p; };
  const size_t N = (size_t)s->N, C = (size_t)s->C;
  const size_t fsz = s->mixed ? sizeof(double) : sizeof(float);
  s->reps = (RepDev*)take(sizeof(RepDev) * s->n_reps);
  s->tiles_int = (Tile*)take(sizeof(Tile) * s->t_int.size());
  s->tiles_chain = (Tile*)take(sizeof(Tile) * s->t_chain.size());
  s->x = take(3 * N * fsz);
  s->v = take(3 * N * fsz);
  s->img = (int*)take(3 * N * sizeof(int));
  s->F = take(N * (s->mixed ? sizeof(F4i) : sizeof(float4)));
  for (long long*& f : s->flj) f = (long long*)take(3 * (size_t)s->Npad * sizeof(long long));
  s->site = (uint16_t*)take(N * sizeof(uint16_t));
  s->cellc = (int*)take(N * sizeof(int));
  s->ref = (float4*)take(N * sizeof(float4));
  s->inv_perm = (int*)take(N * sizeof(int));
  s->pos = (float4*)take(N * sizeof(float4));
  s->tag = (int*)take(N * sizeof(int));
  s->perm = (int*)take(N * sizeof(int));
  s->region_cells = (int*)take(sizeof(int) * (size_t)kRegionCells * s->n_regions);
  s->shapes = (RegionShape*)take(sizeof(RegionShape) * s->shapes_h.size());
  s->runs = (ItemRun*)take(sizeof(ItemRun) * s->runs_h.size());
  s->items = (WorkItem*)take(sizeof(WorkItem) * (size_t)(s->n_lj_items + s->n_build_items));
  s->tasks = (ClusterTask*)take(sizeof(ClusterTask) * (size_t)s->n_cl_max);
  s->task_base = (int*)take(sizeof(int) * (size_t)s->n_lj_items);
  s->n_tasks = (int*)take(2 * sizeof(int));
  s->big = (int*)take(sizeof(int) * (size_t)s->n_lj_items);
  s->list = (unsigned*)take((size_t)s->n_cl_max * s->cap * sizeof(unsigned));
  s->ncl = (int*)take((size_t)s->n_cl_max * sizeof(int));
  s->cl_start = (int*)take((C + 1) * sizeof(int));
  s->count = (int*)take(C * sizeof(int));
  s->scan_seg = (int*)take(scan_seg_ints(s->C) * sizeof(int));
  s->cell_start = (int*)take((C + 1) * sizeof(int));
  s->cell_of = (int*)take(N * sizeof(int));
  s->slot = (int*)take(N * sizeof(int));
  s->tmp = (int*)take(N * sizeof(int));
  s->lj_part = (double*)take(C * 8 * sizeof(double));
  s->b_part = (double*)take(s->t_int.size() * 9 * sizeof(double));
  // kinetic energy (and momentum) per tile of either kind
  s->kepart = (double*)take(4 * std::max(s->t_int.size(), s->t_chain.size()) * sizeof(double));
  s->ke_out = (double*)take(s->n_reps * sizeof(double));
  s->lam = (double*)take((size_t)kNhDoubles * s->n_reps * sizeof(double));   // rescale factor, or the Nose-Hoover state
  s->e_out = (double*)take((size_t)s->n_reps * 16 * sizeof(double));
  s->e_slices = (double*)take((size_t)s->n_reps * s->max_slices * 11 * sizeof(double));
  s->work = (int*)take(2 * sizeof(int));
  s->flags = (unsigned*)take(sizeof(unsigned));
  s->ctl = (int*)take(2 * sizeof(int));
  s->early = (unsigned long long*)take(sizeof(unsigned long long));
  s->stage = (double*)take(6 * N * sizeof(double) + 3 * N * sizeof(int));   // staging: x, v (FP64), images
  if (s->generic) {
    s->mtype = (unsigned char*)take(s->mtype_h.size());
    auto ti = [&](const std::vector<int>& v) { return (const int*)take(v.size() * sizeof(int)); };
    s->topo.b_off = ti(s->t_boff); s->topo.b_at = ti(s->t_bat);
    s->topo.a_off = ti(s->t_aoff); s->topo.a_at = ti(s->t_aat);
    s->topo.d_off = ti(s->t_doff); s->topo.d_at = ti(s->t_dat);
    s->topo.x_off = ti(s->t_xoff); s->topo.x_at = ti(s->t_xat);
    s->topo.terms = (const ushort4*)take(s->t_terms.size() * sizeof(ushort4));
    s->topo.naom = s->S;
    s->topo.n_bonds = s->t_boff[s->S];
    s->topo.n_angles = s->t_aoff[s->S];
    s->topo.n_dihedrals = s->t_doff[s->S];
  }
  return off;
}

// ------------------------------------------------------------------ enqueue helpers
static void prof_mark(md_system* s) {
  if (!s->profile || s->ev_used >= (int)s->ev.size()) return;
  // inside a stream capture an external record becomes an event-record node;
  // outside one (a remainder block launched directly) a plain record
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  cudaStreamIsCapturing(s->st, &cs);
  if (cs == cudaStreamCaptureStatusActive)
    cudaEventRecordWithFlags(s->ev[s->ev_used++], s->st, cudaEventRecordExternal);
  else
    cudaEventRecord(s->ev[s->ev_used++], s->st);
}

// dep: the launch before is the sort's (launch_dependent)
static void enqueue_build(md_system* s, bool dep = false) {
  launch_cl_build(s->pos, s->tag, s->cell_start, s->cl_start, s->region_cells, s->items + s->n_lj_items,
                  s->n_build_items, s->shapes, s->reps, s->list, s->ncl, s->cap, s->tile_cap, s->flags,
                  s->n_tasks, s->generic ? &s->topo : nullptr, dep, s->st);
  launch_cl_rank(s->pos, s->cell_start, s->cl_start, s->region_cells, s->items, s->n_lj_items, s->shapes, s->ncl,
                 s->tasks, s->task_base, s->n_tasks, s->lj_cap, s->big, true, s->st);
}

static void enqueue_rebin(md_system* s) {
  constexpr bool dep = true;
  cudaMemsetAsync(s->count, 0, sizeof(int) * s->C, s->st);
  launch_bin_count(s->mixed, s->x, (int)s->N, s->tiles_int, (int)s->t_int.size(), s->reps, s->cell_of, s->cellc,
                   s->count, s->slot, s->st);
  launch_scan2(s->count, s->cell_start, s->cl_start, s->C, s->scan_seg, dep, s->st);
  launch_bin_scatter(s->cell_of, s->slot, s->cell_start, s->tmp, (int)s->N, dep, s->st);
  launch_cell_sort(s->mixed, s->x, (int)s->N, s->cell_start, s->tmp, s->fp.mtype, s->cellc, s->site, s->reps, s->n_reps, s->C,
                   s->S, s->perm, s->inv_perm, s->pos, s->tag, s->ref, s->flags, dep, s->st);
  prof_mark(s);
  enqueue_build(s, !s->profile);
  prof_mark(s);
}
// memset counted as a launch; the scan of many cells takes two
static int rebin_launches(const md_system* s) { return 7 + (scan_seg_ints(s->C) > 0 ? 1 : 0); }

static void enqueue_lj(md_system* s, bool energy, long long* flj, const StepGate& gate = StepGate{},
                       const ThermoArgs& thermo = ThermoArgs{}) {
  auto launch = [&](int tile_cap, int block, const BigTiles& big, const StepGate& g, const ThermoArgs& t) {
    launch_cl_force(energy, s->pos, s->cell_start, s->cl_start, s->region_cells, s->items, s->n_lj_items, s->shapes,
                    s->reps, s->list, s->tasks, s->task_base, s->cap, tile_cap, s->fp, flj, s->Npad, s->lj_part,
                    s->flags, block, s->lj_lanes, s->persistent_grid, s->work, s->lj_pair_exact, big, g, t, s->st);
  };
  launch(s->lj_cap, s->lj_block, BigTiles{nullptr, nullptr, s->tile_cap}, gate, thermo);
  if (s->lj_cap < s->tile_cap) {
    // not a dependent: the kernel after it may read what the update before the
    // first launch left while this one runs, not while that one does
    StepGate g = gate;
    g.dep = false;
    launch(s->tile_cap, 768, BigTiles{s->big, s->n_tasks + 1, s->tile_cap}, g, ThermoArgs{});
  }
}

static void enqueue_bonded(md_system* s, bool energy, const long long* flj, void* F_out) {
  if (s->generic)
    launch_bonded_generic(energy, (const double*)s->x, s->inv_perm, flj, s->Npad, (int)s->N, s->tiles_int,
                          (int)s->t_int.size(), s->reps, s->fp, s->topo, F_out, s->b_part, s->flags, s->st);
  else
    launch_bonded(s->mixed, energy, s->x, s->site, s->inv_perm, flj, s->Npad, (int)s->N, s->tiles_int,
                  (int)s->t_int.size(), s->reps, s->fp, F_out, s->b_part, s->flags, s->st);
}

// the total force into s->F
static void enqueue_forces(md_system* s) {
  cudaMemsetAsync(s->flj[0], 0, 3 * (size_t)s->Npad * sizeof(long long), s->st);
  enqueue_lj(s, false, s->flj[0]);
  enqueue_bonded(s, false, s->flj[0], s->F);
}

// energies and virial into lj_part and b_part; the force form's kernels and
// buffers are left alone (the energy kernels' LJ form accumulates no forces,
// the general molecules' bonded form leaves its own in scratch memory)
static void enqueue_energy(md_system* s) {
  enqueue_lj(s, true, s->flj[1]);
  enqueue_bonded(s, true, s->flj[1], s->generic ? s->stage : nullptr);
}

static StepArgs step_args(md_system* s, bool chain_tiles, const long long* flj, long long* flj_next) {
  return StepArgs{s->x, s->v, s->img, s->F, s->site, s->cellc, s->inv_perm, s->ref, s->pos, flj, flj_next, s->Npad,
                  (int)s->N, chain_tiles ? s->tiles_chain : s->tiles_int,
                  (int)(chain_tiles ? s->t_chain.size() : s->t_int.size()), s->reps, s->kepart, s->lam, s->flags};
}

// Steps first .. last - 1 of a block of k and, with the last, the closing
// kick; repeat: from LJ launch `first` on.  The opening drift clears an LJ
// buffer, and between LJ launches one kernel does the bonded forces, the
// update and the clearing of the other buffer; the last one closes the step
// and leaves the force.
static void enqueue_steps(md_system* s, int first, int last, int k, bool repeat, const MoveReport& mr) {
  const TopoDev* topo = s->generic ? &s->topo : nullptr;
  for (int j = first; j < last; ++j) {
    long long* flj = s->flj[j & 1];
    // launched as dependents of the kernel before, but where the profile's event
    // records or a WHILE node come in between, and a repeat's first LJ launch: what
    // that reads before its wait is the list build's, its predecessor's
    const StepGate gate{mr.ctl, j, repeat ? 1 : 0, !s->profile && (j > first || (j == 0 && !repeat))};
    if (j == first && repeat) {
      // a repeat resumes at an LJ launch
    } else if (j == 0) {
      launch_integrate(s->mixed, kKickDrift, s->thermo, step_args(s, false, nullptr, flj), s->fp, gate, mr, s->st);
    } else {
      launch_step(s->mixed, kKickKickDrift, s->thermo, s->S, step_args(s, true, s->flj[(j - 1) & 1], flj), s->fp, topo,
                  gate, mr, s->st);
      prof_mark(s);   // closes the bonded group (bonded forces and update)
    }
    ThermoArgs thermo{};
    if (s->thermo != MD_NVE)
      thermo = ThermoArgs{s->n_reps, s->thermo, j > 0, s->kepart, s->lam, 1.0 - s->dt / s->tau, s->dt};
    prof_mark(s);   // closes the integrate group
    StepGate lj_gate = gate;
    lj_gate.dep = !s->profile && !(repeat && j == first);
    enqueue_lj(s, false, flj, lj_gate, thermo);
    prof_mark(s);
  }
  if (last < k) return;
  const StepGate gate{mr.ctl, k - 1, repeat ? 1 : 0, !s->profile};
  launch_step(s->mixed, kKickOnly, s->thermo, s->S, step_args(s, true, s->flj[(k - 1) & 1], nullptr), s->fp, topo, gate,
              mr, s->st);
  prof_mark(s);
}

// Steps that share a WHILE node.  A report leaves the rest of its group without
// effect, and its repeat the launches before, so an early rebin costs a group
// of launches that are off, and a node that is not taken 20 us at 1,500 sites (a
// node per step and a kernel to set its condition: 9 us of a 33 us step).  506k
// sites, us a step, with a node per step / one per block whose launches worked
// before they read the gate / now: 211 / 238 / 177 with 2 early rebins a block of
// 50 steps, 286 / 766 / 272 with 16, 518 / 2,073 / 528 with one every step; 213 /
// 174 / 174 without, in blocks of 10.
constexpr int kGroupSteps = 10, kOneGroup = 16;

// A group of steps inside a capture and the WHILE node after it, whose
// condition the drifts' kernels set when an atom has moved more than skin/2
// since the last rebin: its body rebins and repeats the group from that step's
// LJ launch (StepGate), so such a step computes its forces from fresh bins (and
// is counted), instead of the run stopping.
static cudaError_t enqueue_group(md_system* s, int first, int last, int k) {
  MoveReport mr{};
  const cudaGraphNode_t* deps = nullptr;
  const cudaGraphEdgeData* ed = nullptr;
  size_t nd = 0;
  cudaGraph_t g = nullptr;
  // the graph being captured and where it ends (there is none once a launch, or
  // another thread's call, has invalidated the capture)
  auto captured = [&] {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    const cudaError_t q = cudaStreamGetCaptureInfo(s->st, &cs, nullptr, &g, &deps, &ed, &nd);
    return q != cudaSuccess ? q : cs == cudaStreamCaptureStatusActive && g ? cudaSuccess : cudaErrorStreamCaptureInvalidated;
  };
  cudaError_t e = captured();
  if (e != cudaSuccess) return e;
  if ((e = cudaGraphConditionalHandleCreate(&mr.handle, g, 0, cudaGraphCondAssignDefault)) != cudaSuccess) return e;
  mr.ctl = s->ctl;
  mr.events = s->early;
  enqueue_steps(s, first, last, k, false, mr);
  if ((e = captured()) != cudaSuccess) return e;
  cudaGraphNodeParams p{};
  p.type = cudaGraphNodeTypeConditional;
  p.conditional.handle = mr.handle;
  p.conditional.type = cudaGraphCondTypeWhile;
  p.conditional.size = 1;
  cudaGraphNode_t node;
  if ((e = cudaGraphAddNode(&node, g, deps, ed, nd, &p)) != cudaSuccess) return e;
  cudaGraph_t body = p.conditional.phGraph_out[0];
  e = cudaStreamUpdateCaptureDependencies(s->st, &node, nullptr, 1, cudaStreamSetCaptureDependencies);
  if (e != cudaSuccess) return e;
  // the body, captured on the side stream
  e = cudaStreamBeginCaptureToGraph(s->side, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
  if (e != cudaSuccess) return e;
  cudaStream_t main = s->st;
  const bool prof = s->profile;
  s->st = s->side;
  s->profile = false;
  launch_resume(mr.handle, s->ctl, s->st);
  enqueue_rebin(s);
  enqueue_steps(s, first, last, k, true, mr);
  s->st = main;
  s->profile = prof;
  cudaGraph_t out = nullptr;
  return cudaStreamEndCapture(s->side, &out);
}

// One block of k steps, inside a capture: rebin + list (unless the bins and
// list are already those of the current positions), k velocity-Verlet steps,
// with MD_DISP_REBUILD in groups.  The error of a graph call is returned; a
// refused launch is the runtime's last error.
static cudaError_t enqueue_block(md_system* s, int k, bool rebin) {
  s->ev_used = 0;
  prof_mark(s);
  if (rebin) enqueue_rebin(s);
  if (s->disp != MD_DISP_REBUILD) {
    enqueue_steps(s, 0, k, k, false, MoveReport{});
    return cudaSuccess;
  }
  const int groups = k <= kOneGroup ? 1 : (k + kGroupSteps - 1) / kGroupSteps;
  for (int q = 0; q < groups; ++q) {
    const cudaError_t e = enqueue_group(s, (int)((int64_t)k * q / groups), (int)((int64_t)k * (q + 1) / groups), k);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}
// per step: LJ (two launches where tiles are large) and one update; a closing update (an early rebin adds rebin_launches
// and the launches of the steps it repeats)
static int64_t block_launches(const md_system* s, int k) {
  return rebin_launches(s) + (s->lj_cap < s->tile_cap ? 3LL : 2LL) * k + 1;
}

// accumulate the event timings of the last block (requires a finished stream)
static void prof_collect(md_system* s, int k) {
  if (!s->profile || s->ev_used < 3 + 3 * k) return;
  float ms;
  cudaEventElapsedTime(&ms, s->ev[0], s->ev[1]); s->prof_ms[0] += ms; s->prof_n[0] += 5;
  cudaEventElapsedTime(&ms, s->ev[1], s->ev[2]); s->prof_ms[1] += ms; s->prof_n[1] += 1;
  // per step: the opening update (later steps have none: two records in a row), LJ, bonded and update
  for (int j = 0, e = 2; j < k; ++j, e += 3) {
    if (j == 0) { cudaEventElapsedTime(&ms, s->ev[e], s->ev[e + 1]); s->prof_ms[2] += ms; s->prof_n[2] += 1; }
    cudaEventElapsedTime(&ms, s->ev[e + 1], s->ev[e + 2]); s->prof_ms[3] += ms; s->prof_n[3] += 1;
    cudaEventElapsedTime(&ms, s->ev[e + 2], s->ev[e + 3]); s->prof_ms[4] += ms; s->prof_n[4] += 1;
  }
}

// the rebin cycle as a graph, and the same without its leading rebin + list
// (used for the first cycle after md_set_state / md_rebin, which just did
// them; never while profiling, so that the event layout stays fixed)
static void drop_rem_graphs(md_system* s) {
  for (cudaGraphExec_t& e : s->rem_graphs)
    if (e) { cudaGraphExecDestroy(e); e = nullptr; }
}

// a block of k steps as a graph; rebin: with its leading rebin + list
static int capture_block(md_system* s, int k, bool rebin, cudaGraphExec_t* out) {
  cudaGraph_t g = nullptr;
  CU(cudaStreamBeginCapture(s->st, cudaStreamCaptureModeThreadLocal));
  cudaError_t e = enqueue_block(s, k, rebin);
  const cudaError_t refused = cudaGetLastError();   // a launch, or the graph call that e tells of
  const cudaError_t end = cudaStreamEndCapture(s->st, &g);
  if (e == cudaSuccess) e = refused != cudaSuccess ? refused : end;
  if (e != cudaSuccess) {
    if (g) cudaGraphDestroy(g);
    return fail(s, MD_ECUDA, std::string("graph capture: ") + cudaGetErrorString(e));
  }
  e = cudaGraphInstantiate(out, g, 0);
  cudaGraphDestroy(g);
  if (e != cudaSuccess) {
    *out = nullptr;
    return fail(s, MD_ECUDA, std::string("graph instantiate: ") + cudaGetErrorString(e));
  }
  return MD_OK;
}

static int capture_cycle(md_system* s) {
  if (s->cycle) { cudaGraphExecDestroy(s->cycle); s->cycle = nullptr; }
  if (s->cycle_fresh) { cudaGraphExecDestroy(s->cycle_fresh); s->cycle_fresh = nullptr; }
  drop_rem_graphs(s);
  s->rem_graphs.assign(s->R, nullptr);
  const int rc = capture_block(s, s->R, true, &s->cycle);
  if (rc) return rc;
  const bool prof = s->profile;
  s->profile = false;
  const int rc_fresh = capture_block(s, s->R, false, &s->cycle_fresh);
  s->profile = prof;
  return rc_fresh;
}

static int check_flags(md_system* s) {
  unsigned f = 0;
  CU(cudaGetLastError());   // a launch that was refused
  CU(cudaStreamSynchronize(s->st));
  CU(cudaMemcpy(&f, s->flags, sizeof f, cudaMemcpyDeviceToHost));
  if (!f) return MD_OK;
  CU(cudaMemset(s->flags, 0, sizeof(unsigned)));
  // a non-finite value is the first thing to report: it usually comes with
  // huge finite forces nearby
  if (f & kFlagNaN) return fail(s, MD_EUNSTABLE, "non-finite position, velocity or force");
  if (f & kFlagNbrOverflow) return fail(s, MD_EOVERFLOW, "neighbour list capacity exceeded (raise nbr_capacity)");
  if (f & kFlagFixOverflow) return fail(s, MD_EOVERFLOW, "force beyond the fixed-point range (a part >= 2^17 kJ/mol/nm)");
  if (f & kFlagDisplacement) return fail(s, MD_EUNSTABLE, "an atom moved more than skin/2 between rebins (raise skin or lower rebin_every)");
  if (f & kFlagBadInput) return fail(s, MD_EINVAL, "non-finite input position or velocity");
  if (f & kFlagTimeout) return fail(s, MD_ETIMEOUT, "a bounded device wait gave up");
  return fail(s, MD_ECUDA, "unknown device flag");
}

// Can kernels read or write the caller's n elements at ptr where they lie?  Device
// memory of the current device, aligned to its type, wholly inside its
// allocation (a copy refuses what is not, and a kernel would fault) and apart
// from the system's own workspace; anything else goes through the staging
// buffer by a copy.  A copy of 3 N doubles each way and the gap before it cost
// 3 us at 65k sites, 14 us at 1.5M.
template <class T>
static bool usable_in_place(const md_system* s, const T* ptr, size_t n) {
  using Fn = CUresult (*)(unsigned, CUpointer_attribute*, void**, CUdeviceptr);
  static const Fn fn = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q{};
    const bool ok =
        cudaGetDriverEntryPointByVersion("cuPointerGetAttributes", &f, 12000, cudaEnableDefault, &q) == cudaSuccess;
    return ok && q == cudaDriverEntryPointSuccess ? (Fn)f : nullptr;
  }();
  if (!fn || !ptr || (uintptr_t)ptr % sizeof(T)) return false;
  unsigned type = 0, managed = 1;
  int device = -1, current = -2;
  CUdeviceptr start = 0;
  size_t size = 0;
  CUpointer_attribute what[] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_IS_MANAGED,
                                CU_POINTER_ATTRIBUTE_DEVICE_ORDINAL, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR,
                                CU_POINTER_ATTRIBUTE_RANGE_SIZE};
  void* where[] = {&type, &managed, &device, &start, &size};
  if (fn(5, what, where, (CUdeviceptr)ptr) != CUDA_SUCCESS || type != CU_MEMORYTYPE_DEVICE || managed) return false;
  if (cudaGetDevice(&current) != cudaSuccess || current != device) return false;
  const uintptr_t a = (uintptr_t)ptr, e = a + n * sizeof(T), w = (uintptr_t)s->base;
  return a >= start && e <= start + size && (e <= w || a >= w + s->bytes);
}

// upload positions (wrapped) and velocities, reset images
// Caller's arrays (host or device, x,y,z per atom): k_ingest checks, wraps and
// transposes them on the GPU, from where they lie or from the staging buffer.  A
// non-finite value raises kFlagBadInput, reported by the next check_flags
// (refresh() runs one before md_create / md_set_state return).
static int upload_state(md_system* s, const double* pos, const double* vel) {
  const size_t N = (size_t)s->N;
  auto input = [&](const double*& p, double* stage) {
    if (usable_in_place(s, p, 3 * N)) return cudaSuccess;
    const cudaError_t e = cudaMemcpyAsync(stage, p, 3 * N * sizeof(double), cudaMemcpyDefault, s->st);
    p = stage;
    return e;
  };
  CU(input(pos, s->stage));
  CU(input(vel, s->stage + 3 * N));
  launch_ingest(s->mixed, pos, vel, (int)N, s->tiles_int, (int)s->t_int.size(), s->reps, s->x, s->v, s->img, s->flags,
                s->st);
  CU(cudaGetLastError());
  return MD_OK;
}

static int refresh(md_system* s) {
  const bool p = s->profile;
  s->profile = false;
  enqueue_rebin(s);
  enqueue_forces(s);
  s->profile = p;
  const int rc = check_flags(s);
  s->fresh = rc == MD_OK;
  return rc;
}

// The paper's CBIN binning (Sec. 3.1) done here as a comparison arm: the
// cell of every atom, histogram, exclusive scans and the stable order by atom
// index, on the host from a copy of the positions, with the device's
// formulas (host code is compiled without contraction, so the FP64 cell
// coordinates agree bit for bit).
template <class T>
static void host_bins(const T* x, const md_system* s, std::vector<int>& cell_of, std::vector<int>& cellc,
                      std::vector<int>& cell_start, std::vector<int>& cl_start, std::vector<int>& perm) {
  const int64_t N = s->N;
  std::vector<int> count(s->C, 0);
  for (const RepDev& q : s->reps_h) {
    for (int i = q.atom_off; i < q.atom_off + q.n_atoms; ++i) {
      int k[3];
      for (int a = 0; a < 3; ++a) {
        const double xv = (double)x[a * N + i];
        double sv = xv;
        if (!(xv >= 0.0 && xv < q.L)) sv = xv - q.L * std::floor(xv / q.L);
        int c = (int)std::floor(sv * q.inv_h);
        k[a] = c < 0 ? 0 : (c > q.M - 1 ? q.M - 1 : c);
      }
      const int c = q.cell_base + (k[2] * q.M + k[1]) * q.M + k[0];
      cell_of[i] = c;
      cellc[i] = k[0] | (k[1] << 10) | (k[2] << 20);
      ++count[c];
    }
  }
  cell_start[0] = 0;
  cl_start[0] = 0;
  for (int c = 0; c < s->C; ++c) {
    cell_start[c + 1] = cell_start[c] + count[c];
    cl_start[c + 1] = cl_start[c] + (count[c] + 3) / 4;
  }
  std::vector<int> fill(cell_start.begin(), cell_start.end() - 1);
  for (int64_t i = 0; i < N; ++i) perm[fill[cell_of[i]]++] = (int)i;
}

// ------------------------------------------------------------------ C ABI
extern "C" {

int md_workspace_size(const md_desc* desc, size_t* bytes) {
  md_system tmp;
  md_system* s = &tmp;
  int rc = configure(s, desc);
  if (rc) { g_create_error = s->err; return rc; }
  if (!bytes) return fail(nullptr, MD_EINVAL, "null output");
  *bytes = plan(s, nullptr);
  return MD_OK;
}

int md_create(const md_desc* d, md_system** out) {
  if (!out) return fail(nullptr, MD_EINVAL, "null output pointer");
  *out = nullptr;
  md_system* s = new md_system();
  int rc = configure(s, d);
  if (rc) { g_create_error = s->err; delete s; return rc; }
  if (!d->pos || !d->vel) { delete s; return fail(nullptr, MD_EINVAL, "pos and vel are required"); }
  auto bail = [&](int code) { g_create_error = s->err; md_destroy(s); return code; };
  s->bytes = plan(s, nullptr);
  if (d->workspace) {
    if (d->workspace_bytes < s->bytes) {
      fail(s, MD_ENOMEM, "workspace too small: need " + std::to_string(s->bytes) + " bytes");
      return bail(MD_ENOMEM);
    }
    if (((uintptr_t)d->workspace & 255) != 0) { fail(s, MD_EINVAL, "workspace must be 256-byte aligned"); return bail(MD_EINVAL); }
    s->base = (char*)d->workspace;
  } else {
    if (cudaMalloc(&s->base, s->bytes) != cudaSuccess) {
      cudaGetLastError();
      s->base = nullptr;
      fail(s, MD_ENOMEM, "cudaMalloc of " + std::to_string(s->bytes) + " bytes failed");
      return bail(MD_ENOMEM);
    }
    s->own_mem = true;
  }
  plan(s, s->base);
  s->fp.mtype = s->generic ? s->mtype : nullptr;
  if (d->cuda_stream) {
    s->st = (cudaStream_t)d->cuda_stream;
  } else {
    if (cudaStreamCreateWithFlags(&s->st, cudaStreamNonBlocking) != cudaSuccess) {
      fail(s, MD_ECUDA, "stream creation failed");
      return bail(MD_ECUDA);
    }
    s->own_stream = true;
  }
  if (cudaStreamCreateWithFlags(&s->side, cudaStreamNonBlocking) != cudaSuccess) {
    fail(s, MD_ECUDA, "stream creation failed");
    return bail(MD_ECUDA);
  }
  if (tile_kernels_init() != cudaSuccess || step_kernels_init() != cudaSuccess) {
    cudaGetLastError();
    fail(s, MD_ECUDA, "cannot reserve shared memory for the neighbour-tile kernels");
    return bail(MD_ECUDA);
  }
  if (d->schedule == MD_SCHED_PERSISTENT) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int per_sm = lj_blocks_per_sm(s->lj_block, s->lj_lanes, s->tile_cap);
    s->persistent_grid = std::max(1, std::min(s->n_lj_items, sms * std::max(per_sm, 1)));
  }
  // static tables
  std::vector<uint16_t> site(s->N);
  for (int64_t i = 0; i < s->N; ++i) site[i] = 0;
  for (int r = 0; r < s->n_reps; ++r) {
    const RepDev& q = s->reps_h[r];
    for (int i = 0; i < q.n_atoms; ++i) site[q.atom_off + i] = (uint16_t)(i % s->S);
  }
  // thermostat state: the weak-coupling factor lam[r] = 1, or per replica the
  // Nose-Hoover state at rest (xi = 0, V_com = 0)
  std::vector<double> lam0((size_t)kNhDoubles * s->n_reps, 1.0);
  if (s->thermo == MD_NOSE_HOOVER)
    for (int r = 0; r < s->n_reps; ++r) {
      double* nh = lam0.data() + (size_t)kNhDoubles * r;
      const double rest[12] = {0.0, 1.0, 1.0, 0.0, 0.0, 0.0, 1.0, 2.0, 0.0, 0.0, 0.0, 0.0};
      float* nf = reinterpret_cast<float*>(nh + 12);
      for (int k = 0; k < 12; ++k) { nh[k] = rest[k]; nf[k] = (float)rest[k]; }
    }
  auto up = [&](void* dst, const void* src, size_t b) {
    return cudaMemcpyAsync(dst, src, b, cudaMemcpyHostToDevice, s->st) == cudaSuccess;
  };
  const int ctl0[2] = {kNoMove, 0};
  bool ok = up(s->reps, s->reps_h.data(), sizeof(RepDev) * s->n_reps) &&
            up(s->tiles_int, s->t_int.data(), sizeof(Tile) * s->t_int.size()) &&
            up(s->site, site.data(), sizeof(uint16_t) * s->N) &&
            up(s->lam, lam0.data(), sizeof(double) * lam0.size()) &&
            (!s->generic || (up(s->mtype, s->mtype_h.data(), s->mtype_h.size()) &&
                             up((void*)s->topo.b_off, s->t_boff.data(), s->t_boff.size() * sizeof(int)) &&
                             up((void*)s->topo.b_at, s->t_bat.data(), s->t_bat.size() * sizeof(int)) &&
                             up((void*)s->topo.a_off, s->t_aoff.data(), s->t_aoff.size() * sizeof(int)) &&
                             up((void*)s->topo.a_at, s->t_aat.data(), s->t_aat.size() * sizeof(int)) &&
                             up((void*)s->topo.d_off, s->t_doff.data(), s->t_doff.size() * sizeof(int)) &&
                             up((void*)s->topo.d_at, s->t_dat.data(), s->t_dat.size() * sizeof(int)) &&
                             up((void*)s->topo.x_off, s->t_xoff.data(), s->t_xoff.size() * sizeof(int)) &&
                             up((void*)s->topo.x_at, s->t_xat.data(), s->t_xat.size() * sizeof(int)) &&
                             up((void*)s->topo.terms, s->t_terms.data(), s->t_terms.size() * sizeof(ushort4)))) &&
            up(s->shapes, s->shapes_h.data(), sizeof(RegionShape) * s->shapes_h.size()) &&
            up(s->runs, s->runs_h.data(), sizeof(ItemRun) * s->runs_h.size()) &&
            up(s->tiles_chain, s->t_chain.data(), sizeof(Tile) * s->t_chain.size()) &&
            cudaMemsetAsync(s->flj[0], 0, 3 * (size_t)s->Npad * sizeof(long long), s->st) == cudaSuccess &&
            cudaMemsetAsync(s->flj[1], 0, 3 * (size_t)s->Npad * sizeof(long long), s->st) == cudaSuccess &&
            cudaMemsetAsync(s->work, 0, 2 * sizeof(int), s->st) == cudaSuccess &&
            cudaMemsetAsync(s->flags, 0, sizeof(unsigned), s->st) == cudaSuccess &&
            up(s->ctl, ctl0, sizeof ctl0) &&
            cudaMemsetAsync(s->early, 0, sizeof(unsigned long long), s->st) == cudaSuccess;
  if (ok) {
    launch_plan(s->reps, s->n_reps, s->shapes, s->lj_region, s->n_regions, s->region_cells, s->runs,
                (int)s->runs_h.size(), s->n_lj_items + s->n_build_items, s->items, s->st);
    ok = cudaGetLastError() == cudaSuccess && cudaStreamSynchronize(s->st) == cudaSuccess;
  }
  if (!ok) { fail(s, MD_ECUDA, "initial upload failed"); return bail(MD_ECUDA); }
  rc = upload_state(s, d->pos, d->vel);
  if (rc) return bail(rc);
  rc = refresh(s);
  if (rc) return bail(rc);
  rc = capture_cycle(s);
  if (rc) return bail(rc);
  *out = s;
  return MD_OK;
}

int md_step_async(md_system* s, int64_t n) {
  if (!s || n < 0) return fail(s, MD_EINVAL, "bad arguments");
  const int64_t full = n / s->R, rem = n % s->R;
  if (full && (!s->cycle || !s->cycle_fresh)) {   // a capture failed in an earlier call, which said so
    const int rc = capture_cycle(s);
    if (rc) return rc;
  }
  for (int64_t c = 0; c < full; ++c) {
    const bool skip_rebin = c == 0 && s->fresh && !s->profile;
    s->fresh = false;
    CU(cudaGraphLaunch(skip_rebin ? s->cycle_fresh : s->cycle, s->st));
    if (s->profile) {
      s->ev_used = (int)std::min<int64_t>(s->ev.size(), 3 + 3 * s->R);
      CU(cudaStreamSynchronize(s->st));
      prof_collect(s, s->R);
    }
  }
  if (rem) {
    s->fresh = false;
    cudaGraphExec_t& gr = s->rem_graphs[rem];
    if (!gr) {
      const int rc = capture_block(s, (int)rem, true, &gr);
      if (rc) return rc;
    }
    if (s->profile) s->ev_used = (int)std::min<int64_t>(s->ev.size(), 3 + 3 * rem);
    CU(cudaGraphLaunch(gr, s->st));
    if (s->profile) { CU(cudaStreamSynchronize(s->st)); prof_collect(s, (int)rem); }
  }
  return MD_OK;
}

int md_step(md_system* s, int64_t n) {
  int rc = md_step_async(s, n);
  if (rc) return rc;
  return check_flags(s);
}

int md_sync(md_system* s) {
  if (!s) return fail(s, MD_EINVAL, "null system");
  return check_flags(s);
}

int md_forces(md_system* s, double* f_out) {
  if (!s || !f_out) return fail(s, MD_EINVAL, "bad arguments");
  const size_t N = (size_t)s->N;
  const bool in_place = usable_in_place(s, f_out, 3 * N);
  launch_egress_forces(s->mixed, s->F, (int)N, kFixInv, in_place ? f_out : s->stage, s->st);
  CU(cudaGetLastError());
  if (!in_place) CU(cudaMemcpyAsync(f_out, s->stage, 3 * N * sizeof(double), cudaMemcpyDefault, s->st));
  CU(cudaStreamSynchronize(s->st));
  return MD_OK;
}

int md_energy(md_system* s, md_energy_t* out) {
  if (!s || !out) return fail(s, MD_EINVAL, "bad arguments");
  const bool p = s->profile;
  s->profile = false;
  // energies and virial of the current state
  enqueue_energy(s);
  launch_energy_reduce(s->lj_part, s->b_part, s->reps, s->n_reps, s->max_slices, s->e_slices, s->e_out, s->st);
  // kinetic energy of the current velocities (a pass that only reads v)
  launch_integrate(s->mixed, kKineticOnly, MD_NVE, step_args(s, false, nullptr, nullptr), s->fp, StepGate{},
                   MoveReport{}, s->st);
  launch_kinetic(s->kepart, s->reps, s->n_reps, s->fp, s->ke_out, s->st);
  s->profile = p;
  CU(cudaGetLastError());
  std::vector<double> e((size_t)s->n_reps * 16), ke(s->n_reps);
  CU(cudaMemcpyAsync(e.data(), s->e_out, e.size() * sizeof(double), cudaMemcpyDeviceToHost, s->st));
  CU(cudaMemcpyAsync(ke.data(), s->ke_out, ke.size() * sizeof(double), cudaMemcpyDeviceToHost, s->st));
  int rc = check_flags(s);
  if (rc) return rc;
  for (int r = 0; r < s->n_reps; ++r) {
    md_energy_t& o = out[r];
    const double* q = e.data() + 16 * r;
    o.lj = q[0]; o.lj_shifted = q[1]; o.bond = q[2]; o.angle = q[3]; o.dihedral = q[4];
    for (int k = 0; k < 6; ++k) o.virial[k] = q[5 + k];
    o.kinetic = ke[r];
    o.temperature = 2.0 * ke[r] / (s->reps_h[r].dof * kKB);
    o.total = o.lj_shifted + o.bond + o.angle + o.dihedral + o.kinetic;
    const double V = s->reps_h[r].L * s->reps_h[r].L * s->reps_h[r].L;
    o.pressure = (2.0 * o.kinetic + o.virial[0] + o.virial[1] + o.virial[2]) / (3.0 * V);
  }
  return MD_OK;
}

int md_rebin(md_system* s) {
  if (!s) return fail(s, MD_EINVAL, "null system");
  const bool p = s->profile;
  s->profile = false;
  enqueue_rebin(s);
  s->profile = p;
  const int rc = check_flags(s);
  s->fresh = rc == MD_OK;   // the forces already belong to these positions
  return rc;
}

int md_get_state(md_system* s, double* pos, double* vel, int32_t* images) {
  if (!s) return fail(s, MD_EINVAL, "null system");
  const size_t N = (size_t)s->N, n = 3 * N;
  // the caller's arrays, or where they overlap (copied one after another then)
  // or cannot be written in place the staging buffer
  auto apart = [](const void* a, size_t na, const void* b, size_t nb) {
    return !a || !b || (uintptr_t)a + na <= (uintptr_t)b || (uintptr_t)b + nb <= (uintptr_t)a;
  };
  const bool split = apart(pos, n * 8, vel, n * 8) && apart(pos, n * 8, images, n * 4) && apart(vel, n * 8, images, n * 4);
  const bool px = split && usable_in_place(s, pos, n), pv = split && usable_in_place(s, vel, n),
             pi = split && usable_in_place(s, images, n);
  double* sp = px ? pos : pos ? s->stage : nullptr;
  double* sv = pv ? vel : vel ? s->stage + n : nullptr;
  int* si = pi ? images : images ? reinterpret_cast<int*>(s->stage + 2 * n) : nullptr;
  launch_egress_state(s->mixed, s->x, s->v, s->img, (int)N, sp, sv, si, s->st);
  CU(cudaGetLastError());
  if (pos && !px) CU(cudaMemcpyAsync(pos, sp, n * sizeof(double), cudaMemcpyDefault, s->st));
  if (vel && !pv) CU(cudaMemcpyAsync(vel, sv, n * sizeof(double), cudaMemcpyDefault, s->st));
  if (images && !pi) CU(cudaMemcpyAsync(images, si, n * sizeof(int), cudaMemcpyDefault, s->st));
  CU(cudaStreamSynchronize(s->st));
  return MD_OK;
}

int md_set_state(md_system* s, const double* pos, const double* vel) {
  if (!s || !pos || !vel) return fail(s, MD_EINVAL, "bad arguments");
  CU(cudaStreamSynchronize(s->st));
  int rc = upload_state(s, pos, vel);
  if (rc) return rc;
  return refresh(s);
}

int md_set_params(md_system* s, const md_params* p) {
  if (!s || !p) return fail(s, MD_EINVAL, "bad arguments");
  for (int a = 0; a < 2; ++a)
    if (!(p->mass[a] > 0) || !(p->sigma[a] > 0) || !(p->eps[a] >= 0))
      return fail(s, MD_EINVAL, "masses and sigmas must be > 0, eps >= 0");
  CU(cudaStreamSynchronize(s->st));
  s->params = *p;
  fill_force_params(s);
  CU(cudaMemcpy(s->reps, s->reps_h.data(), sizeof(RepDev) * s->n_reps, cudaMemcpyHostToDevice));
  int rc = capture_cycle(s);
  if (rc) return rc;
  const bool pf = s->profile;
  s->profile = false;
  enqueue_forces(s);
  s->profile = pf;
  return check_flags(s);
}

int md_set_temperature(md_system* s, const double* T) {
  if (!s || !T) return fail(s, MD_EINVAL, "bad arguments");
  CU(cudaStreamSynchronize(s->st));
  for (int r = 0; r < s->n_reps; ++r) { s->reps_h[r].T0 = T[r]; s->T0[r] = T[r]; }
  fill_thermostats(s);
  CU(cudaMemcpy(s->reps, s->reps_h.data(), sizeof(RepDev) * s->n_reps, cudaMemcpyHostToDevice));
  return MD_OK;
}

int md_observables(md_system* s, double* r_ee, double* rg2, double* trans_fraction) {
  if (!s) return fail(s, MD_EINVAL, "null system");
  if (s->generic) return fail(s, MD_EINVAL, "chain observables need linear chains");
  int chains = 0;
  for (int r = 0; r < s->n_reps; ++r) chains += s->reps_h[r].n_chains;
  // scratch in the staging buffer (6N doubles + 3N ints >= 4 doubles per chain + counts)
  double* ree_d = s->stage;
  double* rg_d = s->stage + 3 * (size_t)chains;
  unsigned long long* tr_d = reinterpret_cast<unsigned long long*>(s->stage + 4 * (size_t)chains);
  CU(cudaMemsetAsync(tr_d, 0, sizeof(unsigned long long) * s->n_reps, s->st));
  launch_chain_observables(s->mixed, s->x, (int)s->N, s->reps, s->n_reps, s->fp, chains, ree_d, rg_d, tr_d, s->st);
  CU(cudaGetLastError());
  std::vector<unsigned long long> tr(s->n_reps);
  if (r_ee) CU(cudaMemcpyAsync(r_ee, ree_d, 3 * (size_t)chains * sizeof(double), cudaMemcpyDefault, s->st));
  if (rg2) CU(cudaMemcpyAsync(rg2, rg_d, (size_t)chains * sizeof(double), cudaMemcpyDefault, s->st));
  CU(cudaMemcpyAsync(tr.data(), tr_d, sizeof(unsigned long long) * s->n_reps, cudaMemcpyDeviceToHost, s->st));
  CU(cudaStreamSynchronize(s->st));
  if (trans_fraction)
    for (int r = 0; r < s->n_reps; ++r) {
      const double nd = (double)s->reps_h[r].n_chains * (double)(s->S > 3 ? s->S - 3 : 0);
      trans_fraction[r] = nd > 0 ? (double)tr[r] / nd : 0.0;
    }
  return MD_OK;
}

int md_rdf(md_system* s, int32_t n_bins, const double* edges, int64_t* counts) {
  if (!s || !edges || !counts || n_bins < 1 || n_bins > kRdfMaxBins) return fail(s, MD_EINVAL, "bad arguments (1 <= n_bins <= 16384)");
  if (s->generic) return fail(s, MD_EINVAL, "the RDF's exclusions are those of linear chains");
  if (!(edges[0] >= 0.0)) return fail(s, MD_EINVAL, "edges[0] must be >= 0");
  for (int k = 0; k < n_bins; ++k)
    if (!(edges[k + 1] > edges[k])) return fail(s, MD_EINVAL, "edges must increase");
  for (const RepDev& q : s->reps_h)
    if (edges[n_bins] > q.h) return fail(s, MD_EINVAL, "r_max beyond the cell side of a replica");
  double* ed = nullptr;          // the edges, then the inner part of each bin (two floats)
  unsigned long long* cnt = nullptr;
  const size_t nc = (size_t)s->n_reps * n_bins;
  double h_max = 0.0;
  for (const RepDev& q : s->reps_h) h_max = std::max(h_max, q.h);
  std::vector<double> table(2 * (size_t)n_bins + 1);
  std::copy(edges, edges + n_bins + 1, table.begin());
  rdf_inner_edges(edges, n_bins, h_max, reinterpret_cast<float2*>(table.data() + n_bins + 1));
  // table and counts in the staging buffer (6 N doubles) where
  // they fit, else allocated for the call (allocating and freeing takes longer than the histogram)
  const bool own = table.size() + nc > 6 * (size_t)s->N;
  if (!own) {
    ed = s->stage;
    cnt = reinterpret_cast<unsigned long long*>(s->stage + table.size());
  } else if (cudaMalloc(&ed, sizeof(double) * table.size()) != cudaSuccess ||
             cudaMalloc(&cnt, sizeof(unsigned long long) * nc) != cudaSuccess) {
    cudaGetLastError();
    if (ed) cudaFree(ed);
    return fail(s, MD_ENOMEM, "device memory for the histogram");
  }
  int rc = MD_OK;
  // bins of the current positions (the last rebin's may be up to skin/2 old)
  const bool p = s->profile;
  s->profile = false;
  enqueue_rebin(s);
  s->profile = p;
  if (cudaMemcpyAsync(ed, table.data(), sizeof(double) * table.size(), cudaMemcpyHostToDevice, s->st) != cudaSuccess ||
      cudaMemsetAsync(cnt, 0, sizeof(unsigned long long) * nc, s->st) != cudaSuccess) {
    rc = fail(s, MD_ECUDA, "histogram set-up failed");
  } else {
    const double norm = (double)n_bins / (edges[n_bins] - edges[0]);
    launch_rdf(s->mixed, s->x, (int)s->N, s->cell_start, s->perm, s->pos, s->tag, s->reps, s->n_reps, s->C, ed,
               reinterpret_cast<const float2*>(ed + n_bins + 1), n_bins, norm, cnt, s->st);
    if (cudaGetLastError() != cudaSuccess ||
        cudaMemcpyAsync(counts, cnt, sizeof(unsigned long long) * nc, cudaMemcpyDefault, s->st) != cudaSuccess)
      rc = fail(s, MD_ECUDA, "histogram kernel failed");
  }
  if (rc == MD_OK) {
    rc = check_flags(s);
    s->fresh = rc == MD_OK;
  } else {
    cudaStreamSynchronize(s->st);
  }
  if (own) {
    cudaFree(ed);
    cudaFree(cnt);
  }
  return rc;
}

int md_acf_reset(md_system* s, int32_t max_lag) {
  if (!s || max_lag < 0 || max_lag > 100000) return fail(s, MD_EINVAL, "max_lag must be 0 .. 100000");
  CU(cudaStreamSynchronize(s->st));
  int chains = 0;
  for (const RepDev& q : s->reps_h) chains += q.n_chains;
  if (max_lag != s->acf_lag) {
    if (s->acf_ring) cudaFree(s->acf_ring);
    if (s->acf_acc) cudaFree(s->acf_acc);
    s->acf_ring = s->acf_acc = nullptr;
    s->acf_lag = -1;
    if (cudaMalloc(&s->acf_ring, sizeof(double) * 3 * (size_t)chains * (max_lag + 1)) != cudaSuccess ||
        cudaMalloc(&s->acf_acc, sizeof(double) * (size_t)s->n_reps * (max_lag + 1)) != cudaSuccess) {
      cudaGetLastError();
      return fail(s, MD_ENOMEM, "device memory for the ACF ring");
    }
    s->acf_lag = max_lag;
  }
  CU(cudaMemset(s->acf_acc, 0, sizeof(double) * (size_t)s->n_reps * (max_lag + 1)));
  s->acf_n = 0;
  return MD_OK;
}

static int acf_add(md_system* s, int chains) {
  launch_acf_add(s->acf_ring, chains, s->reps, s->n_reps, s->acf_n, s->acf_lag, s->acf_acc, s->st);
  CU(cudaGetLastError());
  ++s->acf_n;
  return MD_OK;
}

int md_acf_push(md_system* s, const double* r_ee) {
  if (!s || !r_ee) return fail(s, MD_EINVAL, "bad arguments");
  if (s->acf_lag < 0) return fail(s, MD_EINVAL, "md_acf_reset first");
  int chains = 0;
  for (const RepDev& q : s->reps_h) chains += q.n_chains;
  double* slot = s->acf_ring + (size_t)(s->acf_n % (s->acf_lag + 1)) * 3 * chains;
  CU(cudaMemcpyAsync(slot, r_ee, sizeof(double) * 3 * chains, cudaMemcpyDefault, s->st));
  int rc = acf_add(s, chains);
  if (rc) return rc;
  CU(cudaStreamSynchronize(s->st));
  return MD_OK;
}

int md_acf_sample(md_system* s) {
  if (!s) return fail(s, MD_EINVAL, "null system");
  if (s->generic) return fail(s, MD_EINVAL, "end-to-end vectors need linear chains");
  if (s->acf_lag < 0) return fail(s, MD_EINVAL, "md_acf_reset first");
  int chains = 0;
  for (const RepDev& q : s->reps_h) chains += q.n_chains;
  double* slot = s->acf_ring + (size_t)(s->acf_n % (s->acf_lag + 1)) * 3 * chains;
  // end-to-end vectors straight into the ring; R_g^2 and trans counts to scratch
  double* rg_d = s->stage;
  unsigned long long* tr_d = reinterpret_cast<unsigned long long*>(s->stage + chains);
  CU(cudaMemsetAsync(tr_d, 0, sizeof(unsigned long long) * s->n_reps, s->st));
  launch_chain_observables(s->mixed, s->x, (int)s->N, s->reps, s->n_reps, s->fp, chains, slot, rg_d, tr_d, s->st);
  CU(cudaGetLastError());
  return acf_add(s, chains);
}

int md_acf_read(md_system* s, double* C, int64_t* n_samples) {
  if (!s) return fail(s, MD_EINVAL, "null system");
  if (s->acf_lag < 0) return fail(s, MD_EINVAL, "md_acf_reset first");
  const int slots = s->acf_lag + 1;
  std::vector<double> acc((size_t)s->n_reps * slots);
  CU(cudaMemcpyAsync(acc.data(), s->acf_acc, acc.size() * sizeof(double), cudaMemcpyDeviceToHost, s->st));
  CU(cudaStreamSynchronize(s->st));
  const int64_t n = s->acf_n;
  if (n_samples) *n_samples = n;
  if (C)
    for (int r = 0; r < s->n_reps; ++r) {
      const double nc = (double)s->reps_h[r].n_chains;
      const double norm = n > 0 ? acc[(size_t)r * slots] / ((double)n * nc) : 0.0;
      for (int t = 0; t < slots; ++t)
        C[(size_t)r * slots + t] = t < n ? (acc[(size_t)r * slots + t] / ((double)(n - t) * nc)) / norm : NAN;
    }
  return MD_OK;
}

int md_bin_study(md_system* s, int32_t reps, double* ms) {
  if (!s || !ms || reps < 1 || reps > 1000) return fail(s, MD_EINVAL, "bad arguments (1 <= reps <= 1000)");
  CU(cudaStreamSynchronize(s->st));
  const size_t N = (size_t)s->N, C = (size_t)s->C;
  const size_t xb = 3 * N * (s->mixed ? sizeof(double) : sizeof(float));
  void* hx = nullptr;
  CU(cudaMallocHost(&hx, xb));
  std::vector<int> cell_of(N), cellc(N), cell_start(C + 1), cl_start(C + 1), perm(N);
  cudaEvent_t ev[6];
  for (cudaEvent_t& e : ev) cudaEventCreate(&e);
  double acc[6] = {0, 0, 0, 0, 0, 0};
  constexpr bool dep = false;   // event records and copies between the launches
  const bool prof = s->profile;
  s->profile = false;
  int rc = MD_OK;
  for (int k = 0; k < reps && rc == MD_OK; ++k) {
    // GPU arm: on-GPU counting sort and sorted arrays, then the list build
    cudaEventRecord(ev[0], s->st);
    cudaMemsetAsync(s->count, 0, sizeof(int) * C, s->st);
    launch_bin_count(s->mixed, s->x, (int)N, s->tiles_int, (int)s->t_int.size(), s->reps, s->cell_of, s->cellc,
                     s->count, s->slot, s->st);
    launch_scan2(s->count, s->cell_start, s->cl_start, s->C, s->scan_seg, dep, s->st);
    launch_bin_scatter(s->cell_of, s->slot, s->cell_start, s->tmp, (int)N, dep, s->st);
    launch_cell_sort(s->mixed, s->x, (int)N, s->cell_start, s->tmp, s->fp.mtype, s->cellc, s->site, s->reps, s->n_reps, s->C,
                     s->S, s->perm, s->inv_perm, s->pos, s->tag, s->ref, s->flags, dep, s->st);
    cudaEventRecord(ev[1], s->st);
    enqueue_build(s);
    cudaEventRecord(ev[2], s->st);
    // host arm: positions to the host, bins there, binned data back, sorted arrays
    if (cudaMemcpyAsync(hx, s->x, xb, cudaMemcpyDeviceToHost, s->st) != cudaSuccess) { rc = fail(s, MD_ECUDA, "copy"); break; }
    cudaEventRecord(ev[3], s->st);
    if (cudaStreamSynchronize(s->st) != cudaSuccess) { rc = fail(s, MD_ECUDA, "sync"); break; }
    const auto t0 = std::chrono::steady_clock::now();
    if (s->mixed) host_bins((const double*)hx, s, cell_of, cellc, cell_start, cl_start, perm);
    else host_bins((const float*)hx, s, cell_of, cellc, cell_start, cl_start, perm);
    const auto t1 = std::chrono::steady_clock::now();
    cudaEventRecord(ev[4], s->st);
    bool ok = cudaMemcpyAsync(s->cell_of, cell_of.data(), N * sizeof(int), cudaMemcpyHostToDevice, s->st) == cudaSuccess &&
              cudaMemcpyAsync(s->cellc, cellc.data(), N * sizeof(int), cudaMemcpyHostToDevice, s->st) == cudaSuccess &&
              cudaMemcpyAsync(s->cell_start, cell_start.data(), (C + 1) * sizeof(int), cudaMemcpyHostToDevice, s->st) == cudaSuccess &&
              cudaMemcpyAsync(s->cl_start, cl_start.data(), (C + 1) * sizeof(int), cudaMemcpyHostToDevice, s->st) == cudaSuccess &&
              cudaMemcpyAsync(s->tmp, perm.data(), N * sizeof(int), cudaMemcpyHostToDevice, s->st) == cudaSuccess;
    if (!ok) { rc = fail(s, MD_ECUDA, "copy"); break; }
    launch_cell_sort(s->mixed, s->x, (int)N, s->cell_start, s->tmp, s->fp.mtype, s->cellc, s->site, s->reps, s->n_reps, s->C,
                     s->S, s->perm, s->inv_perm, s->pos, s->tag, s->ref, s->flags, dep, s->st);
    cudaEventRecord(ev[5], s->st);
    if (cudaStreamSynchronize(s->st) != cudaSuccess) { rc = fail(s, MD_ECUDA, "sync"); break; }
    float a, b, c, d;
    cudaEventElapsedTime(&a, ev[0], ev[1]);
    cudaEventElapsedTime(&b, ev[1], ev[2]);
    cudaEventElapsedTime(&c, ev[2], ev[3]);
    cudaEventElapsedTime(&d, ev[4], ev[5]);
    const double hb = std::chrono::duration<double, std::milli>(t1 - t0).count();
    acc[0] += a; acc[1] += b; acc[2] += c; acc[3] += hb; acc[4] += d; acc[5] += c + hb + d;
  }
  s->profile = prof;
  for (cudaEvent_t& e : ev) cudaEventDestroy(e);
  cudaFreeHost(hx);
  if (rc) return rc;
  // the list of the bins now in place
  enqueue_build(s);
  for (int k = 0; k < 6; ++k) ms[k] = acc[k] / reps;
  rc = check_flags(s);
  s->fresh = rc == MD_OK;
  return rc;
}

int md_early_rebins(md_system* s, int64_t* count) {
  if (!s || !count) return fail(s, MD_EINVAL, "bad arguments");
  unsigned long long v = 0;
  CU(cudaStreamSynchronize(s->st));
  CU(cudaMemcpy(&v, s->early, sizeof v, cudaMemcpyDeviceToHost));
  *count = (int64_t)v;
  return MD_OK;
}

int md_get_thermostat(md_system* s, double* xi) {
  if (!s || !xi) return fail(s, MD_EINVAL, "bad arguments");
  CU(cudaStreamSynchronize(s->st));
  std::vector<double> h((size_t)kNhDoubles * s->n_reps);
  CU(cudaMemcpy(h.data(), s->lam, h.size() * sizeof(double), cudaMemcpyDeviceToHost));
  for (int r = 0; r < s->n_reps; ++r) xi[r] = s->thermo == MD_NOSE_HOOVER ? h[(size_t)kNhDoubles * r] : 0.0;
  return MD_OK;
}

void* md_stream(md_system* s) { return s ? (void*)s->st : nullptr; }

int md_info(md_system* s, int64_t* n_atoms, int64_t* n_cells, int32_t* cap, int32_t* M) {
  if (!s) return fail(s, MD_EINVAL, "null system");
  if (n_atoms) *n_atoms = s->N;
  if (n_cells) *n_cells = s->C;
  if (cap) *cap = s->cap;
  if (M) *M = s->reps_h[0].M;
  return MD_OK;
}

int md_get_bins(md_system* s, int32_t* cell_of, int32_t* cell_start, int32_t* perm) {
  if (!s) return fail(s, MD_EINVAL, "null system");
  CU(cudaStreamSynchronize(s->st));
  if (cell_of) CU(cudaMemcpy(cell_of, s->cell_of, s->N * sizeof(int), cudaMemcpyDeviceToHost));
  if (cell_start) CU(cudaMemcpy(cell_start, s->cell_start, (s->C + 1) * sizeof(int), cudaMemcpyDeviceToHost));
  if (perm) CU(cudaMemcpy(perm, s->perm, s->N * sizeof(int), cudaMemcpyDeviceToHost));
  return MD_OK;
}

int md_get_neighbors(md_system* s, int32_t* count, int32_t* entries) {
  if (!s) return fail(s, MD_EINVAL, "null system");
  CU(cudaStreamSynchronize(s->st));
  const size_t N = (size_t)s->N;
  std::vector<int> pm(N), cs(s->C + 1), cls(s->C + 1);
  CU(cudaMemcpy(pm.data(), s->perm, N * sizeof(int), cudaMemcpyDeviceToHost));
  CU(cudaMemcpy(cs.data(), s->cell_start, (s->C + 1) * sizeof(int), cudaMemcpyDeviceToHost));
  CU(cudaMemcpy(cls.data(), s->cl_start, (s->C + 1) * sizeof(int), cudaMemcpyDeviceToHost));
  const size_t ncl_used = (size_t)cls[s->C];
  std::vector<int> nc(ncl_used);
  std::vector<unsigned> lst(ncl_used * s->cap);
  if (ncl_used) {
    CU(cudaMemcpy(nc.data(), s->ncl, ncl_used * sizeof(int), cudaMemcpyDeviceToHost));
    CU(cudaMemcpy(lst.data(), s->list, lst.size() * sizeof(unsigned), cudaMemcpyDeviceToHost));
  }
  // every listed pair, both ways, by original atom index: the region tiles
  // rebuilt here exactly as the kernels stage them
  std::vector<int> region_cells((size_t)kRegionCells * s->n_regions);
  CU(cudaMemcpy(region_cells.data(), s->region_cells, region_cells.size() * sizeof(int), cudaMemcpyDeviceToHost));
  std::vector<std::vector<int>> nb(N);
  const int G = s->lj_region;
  int rep = 0;
  for (int r = 0; r < s->n_regions; ++r) {
    while (rep + 1 < s->n_reps && s->reps_h[rep + 1].region_off <= r) ++rep;
    const RepDev& q = s->reps_h[rep];
    const int nx = (q.M + G - 1) / G, x = (r - q.region_off) % nx * G, y = (r - q.region_off) / nx % nx * G;
    const RegionShape& S = s->shapes_h[std::min(G, q.M - x) - 1 + G * (std::min(G, q.M - y) - 1)];
    const int* cell = region_cells.data() + (size_t)kRegionCells * r;
    int start[kMaxTileCells], off[kMaxTileCells + 1];
    off[0] = 0;
    for (int k = 0; k < S.n_tile; ++k) {
      start[k] = cs[cell[k]];
      off[k + 1] = off[k] + cs[cell[k] + 1] - cs[cell[k]];
    }
    for (int h = 0; h < S.n_home; ++h) {
      const int th = S.nb[h][0], n_h = off[th + 1] - off[th];
      for (int kq = 0; kq < (n_h + 3) / 4; ++kq) {
        const int cl = cls[cell[th]] + kq;
        for (int e = 0; e < nc[cl]; ++e) {
          const unsigned E = lst[(size_t)cl * s->cap + e];
          const int t = (int)(E & 0xffffu);
          const int kc = (int)(std::upper_bound(off + 1, off + S.n_tile, t) - (off + 1));   // its tile cell
          const int j = pm[start[kc] + (t - off[kc])];
          for (int u = 0; u < 4; ++u)
            if ((E >> (16 + u)) & 1u) {
              const int i = pm[start[th] + 4 * kq + u];
              nb[i].push_back(j);
              nb[j].push_back(i);
            }
        }
      }
    }
  }
  for (size_t i = 0; i < N; ++i) {
    if ((int)nb[i].size() > s->cap) return fail(s, MD_EOVERFLOW, "an atom has more listed neighbours than the capacity");
    if (count) count[i] = (int)nb[i].size();
    if (entries)
      for (size_t m = 0; m < nb[i].size(); ++m) entries[i * s->cap + m] = nb[i][m];
  }
  return MD_OK;
}

int md_get_cell_units(md_system* s, float* u) {
  if (!s || !u) return fail(s, MD_EINVAL, "bad arguments");
  CU(cudaStreamSynchronize(s->st));
  const size_t N = (size_t)s->N;
  std::vector<float4> p(N);
  std::vector<int> ip(N);
  CU(cudaMemcpy(p.data(), s->pos, N * sizeof(float4), cudaMemcpyDeviceToHost));
  CU(cudaMemcpy(ip.data(), s->inv_perm, N * sizeof(int), cudaMemcpyDeviceToHost));
  for (size_t i = 0; i < N; ++i) {
    const float4 q = p[ip[i]];
    u[3 * i] = q.x; u[3 * i + 1] = q.y; u[3 * i + 2] = q.z;
  }
  return MD_OK;
}

int md_profile_enable(md_system* s, int32_t on) {
  if (!s) return fail(s, MD_EINVAL, "null system");
  CU(cudaStreamSynchronize(s->st));
  const int need = 3 + 3 * s->R + 1;
  while ((int)s->ev.size() < need) {
    cudaEvent_t e;
    CU(cudaEventCreate(&e));
    s->ev.push_back(e);
  }
  s->profile = on != 0;
  return capture_cycle(s);   // the graph carries the event records when on
}

int md_profile_read(md_system* s, double* ms, int64_t* n) {
  if (!s) return fail(s, MD_EINVAL, "null system");
  for (int k = 0; k < kNumProf; ++k) {
    if (ms) ms[k] = s->prof_ms[k];
    if (n) n[k] = s->prof_n[k];
  }
  return MD_OK;
}

int md_profile_reset(md_system* s) {
  if (!s) return fail(s, MD_EINVAL, "null system");
  for (int k = 0; k < kNumProf; ++k) { s->prof_ms[k] = 0; s->prof_n[k] = 0; }
  return MD_OK;
}

int64_t md_launches_per_call(md_system* s, int64_t n) {
  if (!s || n < 0) return 0;
  const int64_t full = n / s->R, rem = n % s->R;
  return full * block_launches(s, s->R) + (rem ? block_launches(s, (int)rem) : 0);
}

// ------------------------------------------------------------------ autotuner
static std::string tune_key(const md_desc* d) {
  int dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceProp prop;
  std::string name = "gpu";
  int sms = 0;
  if (cudaGetDeviceProperties(&prop, dev) == cudaSuccess) { name = prop.name; sms = prop.multiProcessorCount; }
  for (char& ch : name) if (ch == ' ') ch = '_';
  long long N = 0;
  double lmin = 1e300, lmax = 0.0;
  for (int r = 0; r < d->n_replicas; ++r) {
    N += (long long)d->n_chains[r] * d->sites_per_chain;
    lmin = std::min(lmin, d->box[r]);
    lmax = std::max(lmax, d->box[r]);
  }
  char buf[256];
  snprintf(buf, sizeof buf, "%s:%d:p%d:t%d:r%d:n%d:L%.1f-%.1f", name.c_str(), sms, d->precision, d->thermostat,
           d->n_replicas, (int)std::floor(2.0 * std::log2((double)std::max(N, 1LL))), std::round(2.0 * lmin) / 2.0,
           std::round(2.0 * lmax) / 2.0);
  return buf;
}

// time one candidate: create, one warm-up cycle, trial_cycles timed cycles
static int tune_trial(md_desc cand, int cycles, double* us) {
  cand.workspace = nullptr;
  cand.workspace_bytes = 0;
  cand.cuda_stream = nullptr;
  md_system* s = nullptr;
  int rc = md_create(&cand, &s);
  if (rc) return rc;
  rc = md_step(s, cand.rebin_every);
  if (!rc) {
    cudaEvent_t a, b;
    cudaEventCreate(&a);
    cudaEventCreate(&b);
    cudaEventRecord(a, s->st);
    rc = md_step_async(s, (int64_t)cand.rebin_every * cycles);
    cudaEventRecord(b, s->st);
    if (!rc) rc = md_sync(s);
    float ms = 0.f;
    cudaEventSynchronize(b);
    cudaEventElapsedTime(&ms, a, b);
    *us = 1000.0 * ms / ((double)cand.rebin_every * cycles);
    cudaEventDestroy(a);
    cudaEventDestroy(b);
  }
  md_destroy(s);
  return rc;
}

extern "C" int md_autotune(md_desc* d, int32_t trial_cycles, const char* cache_path, md_tuning* out) {
  if (!d || trial_cycles < 1) return fail(nullptr, MD_EINVAL, "autotune needs a descriptor and trial_cycles >= 1");
  const std::string key = tune_key(d);
  const int region0 = d->lj_region ? d->lj_region : 3;
  md_tuning best{d->skin, d->rebin_every, d->lj_block ? d->lj_block : (region0 == 3 ? 384 : 256), d->schedule,
                 d->lj_lanes ? d->lj_lanes : 8, region0, 0, 1e300};
  auto apply_to = [](md_desc& c, const md_tuning& t) {
    c.skin = t.skin; c.rebin_every = t.rebin_every; c.lj_block = t.lj_block; c.schedule = t.schedule;
    c.lj_lanes = t.lj_lanes; c.lj_region = t.lj_region;
  };
  auto apply = [&](const md_tuning& t) { apply_to(*d, t); };
  if (cache_path) {
    if (FILE* f = fopen(cache_path, "r")) {
      char line[512], k[256];
      double skin, us;
      int R, blk, sch, lanes, reg;
      bool found = false;
      // one setting per line; lines of another layout are skipped
      while (fgets(line, sizeof line, f))
        if (sscanf(line, "%255s %lf %d %d %d %d %d %lf", k, &skin, &R, &blk, &sch, &lanes, &reg, &us) == 8 && key == k) {
          best = md_tuning{skin, R, blk, sch, lanes, reg, 1, us};
          found = true;
        }
      fclose(f);
      if (found) {
        apply(best);
        if (out) *out = best;
        return MD_OK;
      }
    }
  }
  bool any = false;
  // the block that a descriptor's default stands for: 768 threads, which only
  // the default gives, where one tile fills an SM (plan_regions)
  auto default_block = [](md_desc c) {
    md_system t;
    c.lj_block = 0;
    return configure(&t, &c) == MD_OK ? t.lj_block : 0;
  };
  // region side x block shape x schedule at the descriptor's cell size
  const int shapes[5][2] = {{2, 128}, {2, 256}, {3, 256}, {3, 384}, {3, 0}};
  for (const auto& rb : shapes)
    for (int sch : {(int)MD_SCHED_GRID, (int)MD_SCHED_PERSISTENT}) {
      md_desc c = *d;
      c.lj_region = rb[0];
      c.lj_block = rb[1];
      c.schedule = sch;
      if (!rb[1] && default_block(c) != 768) continue;   // one of the others
      c.lj_lanes = best.lj_lanes;
      double us = 0.0;
      if (tune_trial(c, trial_cycles, &us) == MD_OK && us < best.us_per_step) {
        best = md_tuning{c.skin, c.rebin_every, rb[1], sch, best.lj_lanes, rb[0], 0, us};
        any = true;
      }
    }
  // lanes per cluster with that region, block shape and schedule
  for (int lanes : {8, 16, 32}) {
    if (lanes == best.lj_lanes) continue;
    md_desc c = *d;
    c.lj_region = best.lj_region;
    c.lj_block = best.lj_block;
    c.schedule = best.schedule;
    c.lj_lanes = lanes;
    double us = 0.0;
    if (tune_trial(c, trial_cycles, &us) == MD_OK && us < best.us_per_step) {
      best = md_tuning{c.skin, c.rebin_every, best.lj_block, best.schedule, lanes, best.lj_region, 0, us};
      any = true;
    }
  }
  // cell size through (skin, rebin interval)
  // (a block that is the default's at one size stays the default's at the others)
  auto at_best = [&](int block) {
    md_desc c = *d;
    apply_to(c, best);
    c.lj_block = block;
    return c;
  };
  const bool dflt = best.lj_block == 0 || best.lj_block == default_block(at_best(0));
  const double skins[4] = {0.08, 0.10, 0.12, 0.15};
  const int reb[4] = {6, 10, 12, 16};
  for (int k = 0; k < 4; ++k) {
    if (skins[k] == best.skin && reb[k] == best.rebin_every) continue;
    md_desc c = at_best(best.lj_block);
    c.skin = skins[k];
    c.rebin_every = reb[k];
    if (dflt) c.lj_block = default_block(c) == 768 ? 0 : default_block(c);
    double us = 0.0;
    if (tune_trial(c, trial_cycles, &us) == MD_OK && us < best.us_per_step) {
      best = md_tuning{skins[k], reb[k], c.lj_block, best.schedule, best.lj_lanes, best.lj_region, 0, us};
      any = true;
    }
  }
  if (!any) return fail(nullptr, MD_EUNSTABLE, "autotune: no candidate ran cleanly");
  apply(best);
  if (cache_path)
    if (FILE* f = fopen(cache_path, "a")) {
      fprintf(f, "%s %.4f %d %d %d %d %d %.3f\n", key.c_str(), best.skin, best.rebin_every, best.lj_block, best.schedule,
              best.lj_lanes, best.lj_region, best.us_per_step);
      fclose(f);
    }
  if (out) *out = best;
  return MD_OK;
}

void md_destroy(md_system* s) {
  if (!s) return;
  if (s->st) cudaStreamSynchronize(s->st);
  if (s->cycle) cudaGraphExecDestroy(s->cycle);
  if (s->cycle_fresh) cudaGraphExecDestroy(s->cycle_fresh);
  drop_rem_graphs(s);
  if (s->side) cudaStreamDestroy(s->side);
  for (cudaEvent_t e : s->ev) cudaEventDestroy(e);
  if (s->own_mem && s->base) cudaFree(s->base);
  if (s->acf_ring) cudaFree(s->acf_ring);
  if (s->acf_acc) cudaFree(s->acf_acc);
  if (s->own_stream && s->st) cudaStreamDestroy(s->st);
  delete s;
}

const char* md_last_error(const md_system* s) { return s ? s->err.c_str() : g_create_error.c_str(); }

}  // extern "C"
