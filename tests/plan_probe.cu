// The launch that a call takes (family, lanes a sample, samples a lane, ...)
// as the library's own planning functions give it, for tests that must not
// slide to another variant (plan_probe.py); and the alignment of what the
// kernels access as vectors.  Links against libbrmppi.so.
#include <vector>

#include "internal.h"

namespace brmppi_host {
brmppi::KConst make_kconst(const brmppi_params& q);
brmppi::Inst make_inst(const double* x0, const float* U_nom, const float* obs, int n_obs, const float* path,
                       int n_pts, float ds, int S, int H, uint64_t seed, uint64_t counter, float* U_out,
                       float* traj_out, float* J_out, float* U_next, int32_t* status, float* part,
                       unsigned int* sync, int spb, int n_discs);
}  // namespace brmppi_host
using namespace brmppi_host;

struct ProbedPlan {
  int32_t tps, bpt, threads, family, rows, ns, local, tiles;
  int64_t smem;
};

// A context without device buffers (planning only, no GPU needed).
extern "C" brmppi_ctx* probe_ctx(const brmppi_params* p, int num_sms, int64_t smem_limit) {
  brmppi_ctx* c = new brmppi_ctx();
  c->prm = *p;
  c->num_sms = num_sms;
  c->smem_limit = static_cast<size_t>(smem_limit);
  return c;
}
extern "C" void probe_free(brmppi_ctx* c) { delete c; }

extern "C" int probe_single(const brmppi_ctx* c, int S, int H, int n_obs, int n_pts, ProbedPlan* out) {
  Shape sh;
  if (!plain_shape(c, n_obs, n_pts, &sh)) return -1;
  const brmppi::KConst k = make_kconst(c->prm);
  brmppi::LaunchDesc L{};
  L.single = make_inst(nullptr, nullptr, nullptr, n_obs, nullptr, n_pts, 0.1f, S, H, 0, 0, nullptr, nullptr, nullptr,
                       nullptr, nullptr, nullptr, nullptr, sh.threads / sh.tps, c->prm.n_discs);
  brmppi::LaunchMode mode;
  const size_t smem = plan_single(c, sh, k, L.single.tiles, &L, &mode);
  *out = {sh.tps, sh.bpt, sh.threads, brmppi::family_of(k), L.rows, mode.ns, mode.local, L.single.tiles,
          static_cast<int64_t>(smem)};
  return 0;
}

// (of a live context: the occupancy of the variant is the device's)
extern "C" int probe_batch(brmppi_ctx* c, const brmppi_instance* inst, int n, ProbedPlan* out) {
  std::vector<brmppi::Inst> table(c->batch.max_batch);
  std::vector<int2> work(c->batch.max_work);
  BatchPlan plan;
  const brmppi_status st = plan_batch(c, c->batch, inst, n, nullptr, table.data(), work.data(), &plan);
  if (st != BRMPPI_OK) return st;
  *out = {plan.shape.tps, plan.shape.bpt, plan.shape.threads, brmppi::family_of(make_kconst(c->prm)), 0, plan.mode.ns,
          plan.mode.local, plan.n_work, static_cast<int64_t>(plan.smem)};
  return 0;
}

// What the autotuners time: (lanes, threads) pairs, at most `room` of them.
static int shapes_out(const std::vector<Shape>& v, int32_t* out, int room) {
  for (int i = 0; i < static_cast<int>(v.size()) && i < room; ++i) {
    out[2 * i] = v[i].tps;
    out[2 * i + 1] = v[i].threads;
  }
  return static_cast<int>(v.size());
}
extern "C" int probe_plain_candidates(const brmppi_ctx* c, int n_obs, int n_pts, int32_t* out, int room) {
  return shapes_out(plain_candidates(c, n_obs, n_pts), out, room);
}
extern "C" int probe_batch_candidates(const brmppi_ctx* c, int32_t* out, int room) {
  return shapes_out(batch_candidates(c, philox_blocks(rows_of(c->prm, c->prm.max_obstacles))), out, room);
}

extern "C" void probe_alignments(int64_t* tables, int64_t* local_rows) {
  *tables = alignof(brmppi::NoiseTables);
  *local_rows = alignof(brmppi::LocalRows<3>);
}
