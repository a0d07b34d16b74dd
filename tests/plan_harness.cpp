// The planner of the tensor-core kernel for tests/test_plan.py: host code, no GPU.
#include <cstring>

#include "snn_tc_plan.h"

using namespace snn;

namespace {

Geom geom(const int* v) {   // N, H, W, C, K, stride, pad, ksize
  Geom g;
  g.N = v[0]; g.H = v[1]; g.W = v[2]; g.C = v[3]; g.K = v[4]; g.stride = v[5]; g.pad = v[6]; g.ksize = v[7];
  g.Cw = (g.C + 31) / 32;
  g.Ho = (g.H + 2 * g.pad - g.ksize) / g.stride + 1;
  g.Wo = (g.W + 2 * g.pad - g.ksize) / g.stride + 1;
  g.tau = 5; g.T = 32;
  return g;
}

// Everything the kernel's index arithmetic relies on.
const char* wrong(const GPlan* plan, int count, int mode, const GParams& p, size_t smem) {
  if (smem > (size_t)kMaxDynSmem) return "shared memory";
  if (p.NA < 2 || p.NA > 4 || p.NS < 3 || p.NS > G_NS_MAX) return "ring depths";
  if (mode == M_FP4 && p.NA % G_XTEAMS) return "activation slots are no multiple of the teams";
  const uint32_t tmem = mode == M_FP4 ? G_TMEM_FP4 : G_TMEM_F16;
  if (p.n_acc < 2 || p.n_acc > 4 || p.n_acc * p.acc_cols > tmem) return "accumulators";
  for (int i = 0; i < count; ++i) {
    const GLayer& o = plan[i].L;
    if (o.Np < 16 || o.Np % 16 || (uint32_t)o.Np > p.acc_cols) return "tile width";
    // slices of 32 columns are read whole
    if ((p.n_acc - 1) * p.acc_cols + ((o.Np + 31) / 32) * 32 > 512 || (o.Np + 31) / 32 > G_MAX_CHUNKS) return "slices";
    if (o.steps < 1 || o.steps >= kGTapsMax || o.st_steps < 1) return "steps";
    if (o.st_steps * o.step_bytes > p.b_slot_bytes) return "weight stage";
    if (plan[i].w_bytes != (size_t)o.n_ct * o.n_cb * o.steps * o.step_bytes) return "weight operand";
    if (plan[i].unit_bytes > p.a_slot_bytes) return "activation unit";
    const int units = o.tma ? o.n_pu : 1;
    for (int t = 0; t < o.steps; ++t) {
      const uint32_t at = o.tap[t] & 0xffffu, dist = o.tap[t] >> 16;
      size_t end;   // in 16-byte units of the slot
      if (o.tma)    // rows of 128 bytes; the first row of a tile is any of a row of positions
        end = (size_t)8 * (o.Wg - 1) + at + (size_t)8 * o.Np;
      else
        end = (size_t)at + dist + (size_t)(o.kpt - 1) * 2 * o.n_planes * o.Rr + o.Np;
      if (end * 16 > plan[i].unit_bytes) return "operand past the unit";
    }
    if (o.pu_end[units - 1] != o.steps) return "units";
    // a tile's instructions add into one accumulator, and only those of one shape do so in the order in which they are issued
    if (o.pair != 0 && o.pair != 1) return "instructions of two shapes on one accumulator";
  }
  return nullptr;
}

}  // namespace

extern "C" {

int plan_takes(const int* g, int f16) { return g_path_takes(geom(g), f16 ? M_F16 : M_FP4); }

// q / d as the kernel divides
uint32_t plan_divide(uint32_t q, uint32_t d) {
  const FastDiv f = make_fastdiv(d);
  return (uint32_t)((uint64_t)(2u * q) * f.m >> 32) >> f.s;
}

// The packed bit of a sum as the epilogue takes it
int plan_sign(float sum, float threshold, int negative_scale) {
  const float x = sum + g_minus_threshold(threshold);
  uint32_t bits;
  memcpy(&bits, &x, 4);
  return (int)(bits >> 31) ^ (negative_scale ? 0 : 1);
}

// Does a chain with at most so many words between two members run on words with tags?
int plan_tagged(uint64_t words) { return g_tagged((size_t)words); }

// The count of a chain's launches of `ctas` CTAs after those in `ended` (ranks, in this order) have ended.
uint64_t plan_launches(uint32_t ctas, const uint32_t* ended, int n) {
  unsigned long long count = 0;
  const GLaunches l = g_launches(&count, ctas);
  for (int i = 0; i < n; ++i) *l.count += g_launch_share(l, ended[i], ctas);   // as the kernel's tear-down does
  return count;
}

// The tiles of problems of so many dealt to `grid` CTAs: ranks per problem and CTA as GParams has them.
void plan_assign(const int* tiles, int count, int grid, uint32_t* ranks) {
  std::vector<GPlan> plan(count);
  for (int i = 0; i < count; ++i) plan[i].L.total_tiles = tiles[i];
  std::vector<uint32_t> r((size_t)count * grid);
  g_assign(plan, grid, &r);
  std::copy(r.begin(), r.end(), ranks);
}

// A plan of a given tile: the epilogue warps that write of a position tile, rows a copy or pixel of it has (0: cannot be planned).
int plan_tile(const int* v, int f16, int kind, int lg, int Np, int* rows) {
  GPlan plan;
  if (!g_plan_layer(geom(v), f16 ? M_F16 : M_FP4, kind, lg, Np, f16 != 0, &plan)) return 0;
  *rows = 1 << plan.L.kp_log;
  return g_writing_warps(plan.L);
}

// out per problem: lg, Np, tma, tiles, channel blocks.  Returns what is wrong with the plan, or null.
const char* plan_make(const int* gs, int count, int f16, int kind, int sms, int* out) {
  const int mode = f16 ? M_F16 : M_FP4;
  std::vector<Geom> g(count);
  std::vector<GPlan> plan(count);
  for (int i = 0; i < count; ++i) g[i] = geom(gs + 8 * i);
  if (kind == TCG_CHAIN) {
    for (int i = 0; i < count; ++i)
      if (!g_plan_by_end(g[i], mode, kind, sms, &plan[i])) return "no plan";
  } else if (!g_plan_independent(g.data(), count, mode, kind, f16 != 0, sms, plan.data())) {
    return "no plan";
  }
  for (int i = 0; i < count; ++i) g_finish_plan(g[i], &plan[i]);
  GParams ring{};
  size_t smem = 0;
  if (!g_ring(plan.data(), count, mode, &ring, &smem)) return "no ring";
  for (int i = 0; i < count; ++i) {
    const GLayer& o = plan[i].L;
    const int v[5] = {o.lg, o.Np, o.tma, o.total_tiles, o.n_cb};
    memcpy(out + 5 * i, v, sizeof(v));
  }
  return wrong(plan.data(), count, mode, ring, smem);
}

// The products that make output position 0 of a pair layer, from what the kernel is told: rows[i] = {channel, kernel row, kernel column, position
// that is read, halves} of every row and step whose sum the epilogue adds to it, steps in ascending order.  Returns how many, 0: no pairs.
int plan_pair_products(const int* v, int* rows) {
  const Geom g = geom(v);
  GPlan P;
  if (!g_plan_independent(&g, 1, M_F16, TCG_WORDS, true, 148, &P) || !P.L.pair) return 0;
  g_finish_plan(g, &P);
  int n = 0;
  for (int t = 0; t < P.L.steps; ++t)
    for (int r = 0; r < G_ROWS; ++r) {
      const GPairRow at = g_pair_row(r, P.taps.col[t][0]);
      // (the sums of the upper lanes, 16 to 31 of each 32, are taken from the accumulator column after)
      const int out[5] = {at.channel, P.taps.row[t][0], at.column, (int)((P.L.tap[t] & 0xffffu) / 8) + (r >> 4 & 1), at.halves};
      memcpy(rows + 5 * n++, out, sizeof(out));
    }
  return n;
}

// positions of the layer, positions whose sums a tile gives, positions it multiplies, tiles of positions
void plan_pair_tiles(const int* v, int* out) {
  const Geom g = geom(v);
  GPlan P;
  g_plan_independent(&g, 1, M_F16, TCG_WORDS, true, 148, &P);
  out[0] = (int)P.L.Qtot; out[1] = P.L.Np - P.L.pair; out[2] = P.L.Np; out[3] = P.L.total_tiles / P.L.n_ct; out[4] = P.L.Wg;
}

// the order in which a group's problems are walked through (by: a GOrder, -1: the one of the rule), and the cycles a tile of each problem given takes for
// its MMAs and its stores.  Returns the GOrder, -1: cannot be planned.
int plan_order(const int* gs, int count, int f16, int kind, int sms, int by, int* order, double* mma, double* drain) {
  std::vector<Geom> g(count);
  std::vector<GPlan> plan(count);
  for (int i = 0; i < count; ++i) g[i] = geom(gs + 8 * i);
  if (!g_plan_independent(g.data(), count, f16 ? M_F16 : M_FP4, kind, f16 != 0, sms, plan.data())) return -1;
  if (by < 0) by = g_order_kind(plan.data(), count, kind);
  g_order(plan.data(), count, (GOrder)by, order);
  for (int i = 0; i < count; ++i) { mma[i] = plan[i].mma; drain[i] = plan[i].drain; }
  return by;
}

// do a group's word outputs leave the L2 first?
int plan_streams(const int* gs, int count, int f16, int kind, int sms) {
  std::vector<Geom> g(count);
  std::vector<GPlan> plan(count);
  for (int i = 0; i < count; ++i) g[i] = geom(gs + 8 * i);
  return g_plan_independent(g.data(), count, f16 ? M_F16 : M_FP4, kind, f16 != 0, sms, plan.data()) ? g_streams(plan.data(), count, kind) : -1;
}

}  // extern "C"
