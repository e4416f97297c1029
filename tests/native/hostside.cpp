// hostside.cpp -- test helper: the library's entry points on a CUDA runtime in
// host memory (fakecuda.h), with kernels that only leave traces: a solve adds 1
// to every y and to every cell's step count per step, and is noted in `solves`.
//
// usage: hostside <scenario>; exits 0 when the scenario holds, and prints why not.
#include "fakecuda.h"

#include <algorithm>

#include "internal.h"

using namespace chemgpu;

struct Solve {
  int64_t n;
  int warps, bps, steps;
  int regs;
  bool lanes;           // the queue order was made by lanes (launch_order: solved)
};
static std::vector<Solve> solves;
static bool order_lanes = false;

#define CHECK(x)                                             \
  do {                                                       \
    if (!(x)) {                                              \
      std::printf("line %d: %s\n", __LINE__, #x);            \
      return 1;                                              \
    }                                                        \
  } while (0)

namespace chemgpu {
static const cudaError_t UNUSED = cudaErrorNotSupported;
cudaError_t set_constants() { return cudaSuccess; }
size_t smem_per_cell(const MechDev &, int) { return 16384; }
size_t staged_bytes(const MechDev &, int) { return 0; }
int max_warps_per_block(const MechDev &, int, int) { return 12; }
int best_warps_per_block(const MechDev &, int, int driver, int) { return driver == CHEM_DRIVER_PERSISTENT ? 12 : 1; }
int occupancy(const MechDev &, int, int, int, int w) { return w <= 12 ? 12 / w : 0; }
// the cells of a batch spread over 10 SMs
int solve_registers(const MechDev &m, int prec, int driver, int couple, int64_t n) { return register_rule(m.S, prec, driver, couple, n, 10); }
void auto_shape(const MechDev &, int, int driver, int, int, bool, int64_t n, int *w, int *bps) {
  const int64_t per = (n + 9) / 10;
  if (driver != CHEM_DRIVER_PERSISTENT) { *w = 1; return; }
  *w = per < 12 ? (int)(per < 1 ? 1 : per) : 12;
  if (per < 12) *bps = 1;
}
cudaError_t launch_order(const MechDev &, const CellsDev &c, double, double, bool solved, int *bucket, int *hist, int *order,
                         cudaStream_t s) {
  const int64_t n = c.n_cells;
  const chem_cell_stats *stats = c.stats;
  fake::enqueue(s, (char *)order, n * sizeof(int), [=] {
    order_lanes = solved;
    if (!s) return;
    fake::touch(stats, n * sizeof(chem_cell_stats));
    fake::touch(bucket, n * sizeof(int));
    fake::touch(hist, ORDER_HIST_INTS * sizeof(int));
    fake::touch(order, n * sizeof(int));
  });
  return cudaSuccess;
}
cudaError_t launch_order_groups(const CellsDev &c, int, int *bucket, int *hist, int *order, cudaStream_t s) {
  return launch_order(MechDev{}, c, 0, 0, false, bucket, hist, order, s);
}
static cudaError_t solve_error = cudaSuccess;
cudaError_t launch_solve(const MechDev &m, const CellsDev &c, const LaunchCfg &cfg, cudaStream_t s) {
  if (solve_error != cudaSuccess) return solve_error;
  const CellsDev cd = c;
  const int S = m.S, k = cfg.n_steps > 1 ? cfg.n_steps : 1;
  const LaunchCfg f = cfg;
  fake::enqueue(s, (char *)cd.y, cd.n_cells * S * sizeof(double), [=] {
    if (s) {
      fake::touch(cd.T, cd.n_cells * sizeof(double));
      fake::touch(cd.P, cd.n_cells * sizeof(double));
      fake::touch(cd.y, cd.n_cells * S * sizeof(double));
      fake::touch(cd.stats, cd.n_cells * sizeof(chem_cell_stats));
      fake::touch(cd.stage - 1, 3 * sizeof(unsigned long long));
      fake::touch(m.blob[0], 16);
      if (cd.tape_n) {
        fake::touch(cd.tape_n, cd.n_cells * sizeof(int));
        fake::touch(cd.tape_rows, cd.n_cells * sizeof(int));
        fake::touch(cd.tape_bad, cd.n_cells * sizeof(int));
      }
    }
    for (int64_t i = 0; i < cd.n_cells * S; ++i) cd.y[i] += k;
    for (int64_t i = 0; i < cd.n_cells; ++i) cd.stats[i].steps = k;
    solves.push_back({cd.n_cells, f.warps_per_block, f.blocks_per_sm, k, f.regs, order_lanes});
  });
  return cudaSuccess;
}
cudaError_t launch_order_tape(const CellsDev &, int *, int *, int *, cudaStream_t) { return UNUSED; }
cudaError_t launch_probe(const MechDev &, const CellsDev &, int, int, double, const double *, const double *, double *, cudaStream_t) { return UNUSED; }
cudaError_t launch_adjoint(const MechDev &, const CellsDev &, const AdjDev &, cudaStream_t) { return UNUSED; }
cudaError_t launch_tangent(const MechDev &, const CellsDev &, const TanDev &, cudaStream_t) { return UNUSED; }
cudaError_t launch_recip_probe(const double *, double *, int64_t, cudaStream_t) { return UNUSED; }
cudaError_t launch_wsum_probe(const double *, double *, int64_t, cudaStream_t) { return UNUSED; }
cudaError_t launch_count_flags(const int *, int64_t, unsigned long long *, cudaStream_t) { return UNUSED; }
cudaError_t launch_rates(const MechDev &, const CellsDev &, double *, cudaStream_t) { return UNUSED; }
cudaError_t launch_deriv_design(const MechDev &, const CellsDev &, int, const double *, const double *, double *, cudaStream_t) { return UNUSED; }
cudaError_t launch_deriv_gather(const MechDev &, const CellsDev &, const double *, const double *, double *, cudaStream_t) { return UNUSED; }
int noalloc_stage_counts(int64_t *, int64_t *, cudaStream_t) { return CHEM_EINVAL; }
}  // namespace chemgpu

// A + B -> C, C -> A + B (photolysis)
static chem_mech *mechanism() {
  chem_reaction rx[2];
  std::memset(rx, 0, sizeof(rx));
  rx[0].kind = CHEM_THERMAL;
  rx[0].n_reac = 2;
  rx[0].reac[0] = 0;
  rx[0].reac[1] = 1;
  rx[0].n_prod = 1;
  rx[0].prod[0] = 2;
  rx[0].yield[0] = 1.0;
  rx[0].A = 1e-12;
  rx[1].kind = CHEM_PHOTOLYSIS;
  rx[1].n_reac = 1;
  rx[1].reac[0] = 2;
  rx[1].n_prod = 2;
  rx[1].prod[0] = 0;
  rx[1].prod[1] = 1;
  rx[1].yield[0] = rx[1].yield[1] = 1.0;
  rx[1].J = 1e-3;
  chem_mech *m = nullptr;
  if (chem_mechanism_create(3, 2, rx, &m) != 0) {
    std::printf("mechanism: %s\n", chem_last_error());
    std::exit(8);
  }
  return m;
}

static chem_opts persistent() {
  chem_opts o;
  chem_opts_default(&o);
  o.driver = CHEM_DRIVER_PERSISTENT;
  return o;
}

// What a creating call clears or copies is done when it returns: the caller's
// streams do not wait for the default stream.
static int create_is_complete() {
  chem_mech *m = mechanism();
  CHECK(fake::legacy.empty());
  for (int rec = 0; rec < 2; ++rec) {
    chem_opts o = persistent();
    o.record_adjoint = rec;
    o.tape_steps = 10;
    chem_cells *c = nullptr;
    CHECK(chem_cells_create(m, 50, &o, &c) == 0);
    CHECK(fake::legacy.empty());
    cudaStream_t s;
    cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
    std::vector<double> T(50, 300.0), P(50, 1e5), y(150, 0.0);
    chem_cell_stats st[50];
    CHECK(chem_cells_set_state(c, T.data(), P.data(), y.data(), CHEM_MEM_HOST, s) == 0);
    CHECK(chem_solve_step(c, 600.0, s) == 0);
    CHECK(fake::races == 0);
    fake::drain_legacy();
    CHECK(chem_get_stats(c, st, CHEM_MEM_HOST, s) == 0);
    for (int i = 0; i < 50; ++i) CHECK(st[i].steps == 1);
    chem_cells_destroy(c);
    cudaStreamDestroy(s);
  }
  chem_mechanism_destroy(m);
  return 0;
}

static int host_chunk(int64_t, int64_t, int32_t, void *) { return 0; }

struct Host {
  std::vector<double> T, P, y;
  std::vector<chem_cell_stats> st;
  explicit Host(int n) : T(n, 300.0), P(n, 1e5), y(3 * n, 0.0), st(n) {}
  int run(chem_pipeline *p, int steps, chem_chunk_fn fn) {
    return chem_pipeline_run(p, T.data(), P.data(), nullptr, y.data(), 600.0, steps, fn, nullptr, st.data());
  }
};

// A run uses nothing that is still to be cleared on the default stream, with and without host work.
static int pipeline_is_ordered() {
  chem_mech *m = mechanism();
  const chem_opts o = persistent();
  chem_pipeline *p = nullptr;
  CHECK(chem_pipeline_create(m, 50, 4, &o, &p) == 0);
  Host h(50);
  for (int with = 0; with < 2; ++with) {
    CHECK(h.run(p, 2, with ? host_chunk : nullptr) == 0);
    CHECK(fake::races == 0);
    fake::drain_legacy();
    for (double v : h.y) CHECK(v == 2.0 * (with + 1));
    for (auto &s : h.st) CHECK(s.steps == (with ? 1 : 2));       // the last launch's count
  }
  chem_pipeline_destroy(p);
  chem_mechanism_destroy(m);
  return 0;
}

// A run allocates nothing and a pipeline holds one copy of its cells, whatever the
// host does between the steps; a run that fails for another reason says so, and
// the next one is as before.
static int pipeline_memory() {
  chem_mech *m = mechanism();
  const chem_opts o = persistent();
  const size_t base = fake::live;
  const int n = 1000, K = 8;
  chem_cells *c = nullptr;
  CHECK(chem_cells_create(m, n, &o, &c) == 0);
  const size_t one = fake::live - base;
  chem_cells_destroy(c);
  CHECK(fake::live == base);
  chem_pipeline *p = nullptr;
  CHECK(chem_pipeline_create(m, n, K, &o, &p) == 0);
  const size_t held = fake::live, calls = fake::n_malloc;
  CHECK(held - base <= one + K * (ORDER_HIST_INTS * sizeof(int) + 128));
  Host h(n);
  fake::device = 1;                                // another device is current
  CHECK(h.run(p, 1, nullptr) == CHEM_EINVAL);
  fake::device = 0;
  for (int with = 0; with < 2; ++with) {
    solves.clear();
    CHECK(h.run(p, 1, with ? host_chunk : nullptr) == 0);
    CHECK(fake::live == held && fake::n_malloc == calls);
    CHECK(solves.size() == (with ? (size_t)K : 1u));
    for (double v : h.y) CHECK(v == 1.0 + with);
  }
  chem_pipeline_destroy(p);
  CHECK(fake::live == base);
  for (int fit = 0; fit < (int)(calls); ++fit) {   // no memory for the allocation after `fit`
    fake::fail_malloc = fit;
    const int rc = chem_pipeline_create(m, n, K, &o, &p);
    fake::fail_malloc = -1;
    if (rc == 0) {
      chem_pipeline_destroy(p);
      break;
    }
    CHECK(rc == CHEM_ENOMEM && fake::live == base);
  }
  chem_mechanism_destroy(m);
  return 0;
}

// The chunks of a pipeline run side by side: each has the launch shape of all cells
// together (or the one the caller gave), not that of a batch alone on the device.
static int pipeline_shape() {
  chem_mech *m = mechanism();
  for (int given = 0; given < 2; ++given)
    for (int n : {40, 100, 1000}) {
      chem_opts o = persistent();
      if (given) o.cells_per_block = 7, o.lu_precision = 32;
      chem_pipeline *p = nullptr;
      CHECK(chem_pipeline_create(m, n, 4, &o, &p) == 0);
      Host h(n);
      solves.clear();
      CHECK(h.run(p, 1, nullptr) == 0 && h.run(p, 1, host_chunk) == 0);
      CHECK(solves.size() == 5 && solves[0].n == n);
      for (const Solve &x : solves) CHECK(x.warps == solves[0].warps && x.bps == solves[0].bps && x.regs == (given && n == 1000 ? 80 : 168));
      CHECK(solves[0].warps == (given ? 7 : n < 120 ? n / 10 : 12));
      chem_pipeline_destroy(p);
    }
  chem_mechanism_destroy(m);
  return 0;
}

// The queue order is keyed by the whole-warp kernel for a first solve and by lanes
// once the cells have costs, also when the steps are a graph; a solve that was not
// launched leaves no costs.
static int graph_order() {
  chem_mech *m = mechanism();
  const chem_opts o = persistent();
  chem_cells *c = nullptr;
  CHECK(chem_cells_create(m, 50, &o, &c) == 0);
  cudaStream_t s;
  cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
  std::vector<double> T(50, 300.0), P(50, 1e5), y(150, 0.0);
  CHECK(chem_cells_set_state(c, T.data(), P.data(), y.data(), CHEM_MEM_HOST, s) == 0);
  solve_error = cudaErrorLaunchOutOfResources;
  CHECK(chem_solve_step(c, 600.0, s) == CHEM_ECUDA);
  CHECK(chem_solve_steps(c, 600.0, 3, s) == CHEM_ECUDA);
  solve_error = cudaSuccess;
  for (int call = 0; call < 4; ++call) {
    solves.clear();
    CHECK(chem_solve_steps(c, 600.0, 3, s) == 0);
    CHECK(solves.size() == 1 && solves[0].steps == 3 && solves[0].lanes == (call > 0));
  }
  CHECK(chem_solve_step(c, 600.0, s) == 0 && solves.back().lanes);
  CHECK(chem_solve_steps(c, 600.0, 2, s) == 0 && solves.back().steps == 2 && solves.back().lanes);
  CHECK(chem_get_state(c, y.data(), CHEM_MEM_HOST, s) == 0);
  for (double v : y) CHECK(v == 15.0);
  chem_cells_destroy(c);
  chem_mechanism_destroy(m);
  return 0;
}

// Launch shapes for every block size that a mechanism's cells may fit in: a batch
// is narrowed to two warps per FP64 unit and never below, whole groups stay whole,
// and a batch that cannot fill its blocks spreads over the SMs.
static int shape_rule() {
  const int n_sm = 152;
  for (int full = 1; full <= MAX_WARPS_PER_BLOCK; ++full)
    for (int64_t n = 1; n < 60 * n_sm; n += 37) {
      const int64_t per = (n + n_sm - 1) / n_sm;
      const int w = shape_warps(full, 1, n, n_sm, true), wide = shape_warps(full, 1, n, n_sm, false);
      CHECK(wide == (per < full ? per : full));
      if (per < full || per > 36) CHECK(w == wide);
      else CHECK(w == std::min(full, per <= 24 ? 8 : 10));
    }
  for (int couple : {2, 3, 5})
    for (int64_t n = couple; n < 5000; n += couple) {
      const int full = MAX_WARPS_PER_BLOCK / couple * couple, w = shape_warps(full, couple, n, n_sm, false);
      CHECK(w >= couple && w <= full && w % couple == 0 && (w == full || (int64_t)w * n_sm >= n));
    }
  return 0;
}

// Registers of the solve kernels: 168 but for up to 32 species, where large plain
// batches take 128 and large batches of the FP32 factorisation 80.
static int register_choice() {
  const int P = CHEM_DRIVER_PLAIN, Q = CHEM_DRIVER_PERSISTENT;
  for (int S : {1, 20, 32, 33, 72, 128})
    for (int prec : {64, 32})
      for (int drv : {P, Q})
        for (int64_t n : {1, 1824, 1825, 12160, 12161, 1000000}) {
          const int r = register_rule(S, prec, drv, 1, n, 152);
          if (S > 32) CHECK(r == 168);
          else if (prec == 32 && n > 12160) CHECK(r == 80);
          else CHECK(r == (drv == P && n > 1824 ? 128 : 168));
          CHECK(register_rule(S, prec, drv, 2, n, 152) == 168);
        }
  return 0;
}

int main(int argc, char **argv) {
  const std::string what = argc > 1 ? argv[1] : "";
  if (what == "create_is_complete") return create_is_complete();
  if (what == "pipeline_is_ordered") return pipeline_is_ordered();
  if (what == "pipeline_memory") return pipeline_memory();
  if (what == "pipeline_shape") return pipeline_shape();
  if (what == "graph_order") return graph_order();
  if (what == "shape_rule") return shape_rule();
  if (what == "register_choice") return register_choice();
  std::printf("unknown scenario\n");
  return 2;
}
