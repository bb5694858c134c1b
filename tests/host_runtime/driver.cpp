// Host code of the library on the runtime of fake_cudart.cpp: one scenario
// per name; prints what is wrong and exits 1, or exits 0.
#include <algorithm>
#include <array>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include "fake_cudart.h"
#include "zef_internal.h"

using namespace zef;

namespace {

int g_bad = 0;
#define CHECK(cond, ...)          \
  do {                            \
    if (!(cond)) {                \
      ++g_bad;                    \
      std::printf(__VA_ARGS__);   \
      std::printf("\n");          \
    }                             \
  } while (0)

// an octahedron of radius r, every face cut into m^2 triangles by its planes
struct Surface {
  std::vector<float> v;
  std::vector<int32_t> t;
};
Surface octahedron(float r, int m) {
  Surface s;
  std::map<std::array<int, 3>, int32_t> index;
  auto vertex = [&](int x, int y, int z) {
    const std::array<int, 3> k = {x, y, z};
    const auto [it, fresh] = index.emplace(k, (int32_t)index.size());
    if (fresh)
      for (int c : k) s.v.push_back(r * (float)c / (float)m);
    return it->second;
  };
  for (int o = 0; o < 8; ++o) {
    const int sx = o & 1 ? -1 : 1, sy = o & 2 ? -1 : 1, sz = o & 4 ? -1 : 1;
    const bool flip = sx * sy * sz < 0;
    auto at = [&](int i, int j) { return vertex(sx * i, sy * j, sz * (m - i - j)); };
    auto add = [&](int32_t a, int32_t b, int32_t c) {
      s.t.insert(s.t.end(), {a, flip ? c : b, flip ? b : c});
    };
    for (int i = 0; i < m; ++i)
      for (int j = 0; i + j < m; ++j) {
        add(at(i + 1, j), at(i, j + 1), at(i, j));
        if (i + j + 1 < m) add(at(i + 1, j), at(i + 1, j + 1), at(i, j + 1));
      }
  }
  return s;
}

zef_status add(zef_ctx *ctx, int id, const Surface &s) {
  return zef_add_compartment(ctx, id, s.v.data(), (int64_t)s.v.size() / 3, s.t.data(), (int64_t)s.t.size() / 3, 0);
}

// no capacity is claimed for a buffer that is not there
void check_buffers(const LabelBuffers &b, long k, const char *when) {
  CHECK(!b.cap_points || (b.spts && b.perm && b.keys && b.in_mask && b.unc_mask),
        "allocation %ld failed, %s: %lld points without their buffers", k, when, (long long)b.cap_points);
  CHECK(!b.cap_items || (b.tile_box && b.flags && b.items && b.block_sums),
        "allocation %ld failed, %s: %lld items without their buffers", k, when, (long long)b.cap_items);
  CHECK(!b.cap_stage || (b.labels_tmp && b.pts_tmp), "allocation %ld failed, %s: no staging", k, when);
  CHECK(!b.cap_pending || b.pending, "allocation %ld failed, %s: no list", k, when);
}

// Every device allocation of a registration, and of a call behind it, fails
// once in turn: whatever the call returns, the context stays usable.
int out_of_memory() {
  const Surface small = octahedron(1.f, 2), large = octahedron(2.f, 24);
  const std::vector<float> pts(3 * 5000, 0.25f);
  std::vector<int32_t> lab(5000);
  zef_label_opts general;
  std::memset(&general, 0, sizeof(general));
  general.block_threads = 256;
  general.points_per_thread = 2;
  long last = 1;
  for (long k = 0; k < last; ++k) {
    zef_ctx *ctx = nullptr;
    CHECK(zef_create(&ctx, 0, nullptr) == ZEF_OK, "create");
    CHECK(add(ctx, 1, small) == ZEF_OK, "first surface: %s", zef_last_error(ctx));
    fake_fail_alloc(k);
    const zef_status reg = add(ctx, 2, large);
    check_buffers(ctx->lb, k, "after the registration");
    zef_status call = ZEF_OK;
    for (int n : {100, 5000})
      if (!call) call = zef_label_points(ctx, pts.data(), n, lab.data(), nullptr, &general, nullptr);
    if (fake_allocs() > last) last = fake_allocs();
    fake_fail_alloc(-1);
    CHECK(reg == ZEF_OK || reg == ZEF_ERR_OOM, "allocation %ld: registration returned %d", k, reg);
    CHECK(call == ZEF_OK || call == ZEF_ERR_OOM, "allocation %ld: the call returned %d", k, call);
    CHECK(!reg || !call, "allocation %ld: one failure, reported by the registration and by the call", k);
    check_buffers(ctx->lb, k, "after the failure");
    for (int n : {100, 5000}) {
      const zef_status st = zef_label_points(ctx, pts.data(), n, lab.data(), nullptr, &general, nullptr);
      CHECK(st == ZEF_OK, "allocation %ld failed: the next call of %d points returned %d: %s", k, n, st,
            zef_last_error(ctx));
      check_buffers(ctx->lb, k, "after the next call");
      CHECK(ctx->lb.cap_points >= n, "allocation %ld failed: buffers of %lld points for %d", k,
            (long long)ctx->lb.cap_points, n);
    }
    CHECK(add(ctx, 3, small) == ZEF_OK, "allocation %ld failed: the next surface: %s", k, zef_last_error(ctx));
    check_buffers(ctx->lb, k, "after the next surface");
    zef_destroy(ctx);
  }
  return 0;
}

// Copies and sets that the library's kernels read or overwrite are in order
// with them, also on a non-blocking stream.
int uploads() {
  const Surface a = octahedron(1.f, 3), b = octahedron(2.f, 5);
  const std::vector<float> pts(300, 0.25f);
  std::vector<int32_t> lab(100);
  const int32_t order[2] = {2, 1};
  zef_ctx *ctx = nullptr;
  std::string first;
  CHECK(zef_create(&ctx, 0, nullptr) == ZEF_OK, "create");
  CHECK(add(ctx, 1, a) == ZEF_OK && add(ctx, 2, b) == ZEF_OK, "surfaces: %s", zef_last_error(ctx));
  CHECK(zef_compartment_priority(ctx, order, 2) == ZEF_OK, "priority: %s", zef_last_error(ctx));
  CHECK(zef_label_points(ctx, pts.data(), 100, lab.data(), nullptr, nullptr, nullptr) == ZEF_OK, "labels: %s",
        zef_last_error(ctx));
  CHECK(fake_unordered(&first) == 0, "%ld launches beside a copy on the legacy stream, the first %s",
        fake_unordered(nullptr), first.c_str());
  zef_destroy(ctx);
  return 0;
}

// An error that a kernel recorded is reported once.
int status_once() {
  const std::vector<float> pts(300, 0.25f);
  std::vector<int32_t> lab(100);
  zef_ctx *ctx = nullptr;
  CHECK(zef_create(&ctx, 0, nullptr) == ZEF_OK, "create");
  CHECK(add(ctx, 1, octahedron(1.f, 3)) == ZEF_OK, "surface: %s", zef_last_error(ctx));
  for (const uint32_t bit : {ST_TIMEOUT, ST_INVALID}) {
    fake_on_launch("k_grid_label", [ctx, bit] { ctx->d_status[0] |= bit; });
    CHECK(zef_label_points(ctx, pts.data(), 100, lab.data(), nullptr, nullptr, nullptr) ==
              (bit == ST_TIMEOUT ? ZEF_ERR_TIMEOUT : ZEF_ERR_INVALID_ARG), "bit %u: not reported", bit);
    fake_on_launch("", [] {});
    CHECK(zef_synchronize(ctx) == ZEF_OK, "bit %u: reported twice: %s", bit, zef_last_error(ctx));
    CHECK(zef_label_points(ctx, pts.data(), 100, lab.data(), nullptr, nullptr, nullptr) == ZEF_OK,
          "bit %u: reported by the next call: %s", bit, zef_last_error(ctx));
  }
  zef_destroy(ctx);
  return 0;
}

// Host meshes without tets: every entry point that works in place leaves the
// nodes as they are.
int no_tets() {
  const std::vector<float> x = {0.1f, 0.2f, 0.3f, 1.f, 2.f, 3.f};
  zef_smooth_opts o = {0.4f, 0.4f, 0.f, 3};
  zef_ctx *ctx = nullptr;
  CHECK(zef_create(&ctx, 0, nullptr) == ZEF_OK, "create");
  CHECK(add(ctx, 1, octahedron(1.f, 3)) == ZEF_OK, "surface: %s", zef_last_error(ctx));
  int32_t it = 0;
  int64_t count = 0;
  std::vector<float> y = x;
  CHECK(zef_taubin_smooth_surface(ctx, y.data(), 2, nullptr, 0, nullptr, &o, &it, &count) == ZEF_OK, "boundaries: %s",
        zef_last_error(ctx));
  CHECK(y == x, "boundary smoothing without tets changed the nodes: %g %g %g", y[0], y[1], y[2]);
  y = x;
  CHECK(zef_inflate(ctx, y.data(), 2, nullptr, 0, 1, 0.05f, &count) == ZEF_OK, "inflation: %s", zef_last_error(ctx));
  CHECK(y == x, "inflation without tets changed the nodes: %g %g %g", y[0], y[1], y[2]);
  zef_destroy(ctx);
  return 0;
}

// Anchors whose solid angles were cut short by an expired wait make no grid:
// the registration reports it, the next call builds the grid anew, and an
// error of an earlier call stays to be reported.
int anchors_cut_short() {
  const std::vector<float> pts(300, 0.25f);
  std::vector<int32_t> lab(100);
  zef_ctx *ctx = nullptr;
  CHECK(zef_create(&ctx, 0, nullptr) == ZEF_OK, "create");
  fake_settle();
  ctx->d_status[0] = ST_INVALID;
  fake_on_launch("k_label32", [ctx] { ctx->d_status[0] |= ST_TIMEOUT; });
  CHECK(add(ctx, 1, octahedron(1.f, 3)) == ZEF_ERR_TIMEOUT, "registration did not report the expired wait");
  CHECK(ctx->grids.empty(), "a grid from anchors that were cut short");
  fake_on_launch("", [] {});
  CHECK(zef_synchronize(ctx) == ZEF_ERR_INVALID_ARG, "the earlier call's error is lost");
  CHECK(zef_label_points(ctx, pts.data(), 100, lab.data(), nullptr, nullptr, nullptr) == ZEF_OK, "next call: %s",
        zef_last_error(ctx));
  CHECK(ctx->grids.size() == 1 && ctx->grids[0].usable, "the next call did not build the grid");
  zef_destroy(ctx);
  return 0;
}

// What registration needed for itself is given back where it is large.
int scratch_given_back() {
  zef_ctx *ctx = nullptr;
  CHECK(zef_create(&ctx, 0, nullptr) == ZEF_OK, "create");
  size_t largest = 0;
  for (int m : {4, 60, 120, 8}) {
    CHECK(add(ctx, m, octahedron(1.f, m)) == ZEF_OK, "surface: %s", zef_last_error(ctx));
    const CompGrid &g = ctx->grids.back();
    largest = std::max(largest, (size_t)g.n[0] * g.n[1] * g.n[2] * 24);
    const size_t held = ctx->gr_cap[0] + ctx->gr_cap[1];
    CHECK(held <= (size_t)32 << 20, "%zu bytes of scratch held after a surface of %d triangles", held, 8 * m * m);
    for (int k = 0; k < 2; ++k)
      CHECK((ctx->gr_buf[k] != nullptr) == (ctx->gr_cap[k] > 0), "buffer %d and its size differ", k);
  }
  CHECK(largest > (size_t)32 << 20, "no surface needed more than is kept");
  zef_destroy(ctx);
  return 0;
}

// A new priority order uploads the rows, not the surfaces; the same one nothing.
int priority_uploads() {
  zef_ctx *ctx = nullptr;
  CHECK(zef_create(&ctx, 0, nullptr) == ZEF_OK, "create");
  CHECK(add(ctx, 1, octahedron(1.f, 20)) == ZEF_OK && add(ctx, 2, octahedron(2.f, 20)) == ZEF_OK, "surfaces: %s",
        zef_last_error(ctx));
  const int32_t same[2] = {1, 2}, other[2] = {2, 1};
  size_t before = fake_uploaded();
  const uint64_t gen = ctx->gen;
  CHECK(zef_compartment_priority(ctx, same, 2) == ZEF_OK, "priority: %s", zef_last_error(ctx));
  CHECK(fake_uploaded() == before && ctx->gen == gen, "the same order uploaded %zu bytes", fake_uploaded() - before);
  CHECK(zef_compartment_priority(ctx, other, 2) == ZEF_OK, "priority: %s", zef_last_error(ctx));
  CHECK(fake_uploaded() > before && fake_uploaded() - before <= 4096, "another order uploaded %zu bytes",
        fake_uploaded() - before);
  CHECK(ctx->gen != gen && ctx->h_grid[0].comp == 1 && ctx->h_grid[1].comp == 0, "the rows are the old order's");
  fake_settle();
  const int32_t *ids = ctx->d_row_ids;
  CHECK(ids[0] == 2 && ids[1] == 1 && ctx->d_comps[0].row == 1 && ctx->d_comps[1].row == 0, "the old order's records");
  before = fake_uploaded();
  CHECK(add(ctx, 3, octahedron(3.f, 20)) == ZEF_OK, "surface: %s", zef_last_error(ctx));
  CHECK(fake_uploaded() - before > 100000, "a surface uploaded %zu bytes", fake_uploaded() - before);
  zef_destroy(ctx);
  return 0;
}

// Cells that list more triangles than 32 bits count (the scans' totals wrap to
// small ones) make no grid.
int sums_beyond_32_bits() {
  for (const bool refs : {true, false}) {
    zef_ctx *ctx = nullptr;
    CHECK(zef_create(&ctx, 0, nullptr) == ZEF_OK, "create");
    const long before = fake_launches("k_gr_finish");
    fake_on_launch_args("k_gr_sizes", [refs](void **args) {
      int64_t *sums = *reinterpret_cast<int64_t **>(args[3]) + 1;  // triangles of all lists, words of all blocks
      return [=] {
        sums[0] = refs ? ((int64_t)1 << 32) + 100 : 100;
        sums[1] = refs ? 25 : ((int64_t)1 << 32) + 25;
      };
    });
    CHECK(add(ctx, 1, octahedron(1.f, 8)) == ZEF_OK, "surface: %s", zef_last_error(ctx));
    fake_on_launch("", [] {});
    CHECK(ctx->grids.size() == 1 && !ctx->grids[0].usable, "a grid with %s beyond 32 bits", refs ? "lists" : "blocks");
    CHECK(fake_launches("k_gr_finish") == before, "blocks were written");
    zef_destroy(ctx);
  }
  return 0;
}

// A call whose launches failed half-way leaves counts in the lists: the next
// call clears them first, and enqueueing into a graph (which may never run)
// does not count as having done so.
int lists_cleared_after_a_failure() {
  zef_ctx *ctx = nullptr;
  CHECK(zef_create(&ctx, 0, nullptr) == ZEF_OK, "create");
  CHECK(add(ctx, 1, octahedron(1.f, 4)) == ZEF_OK, "surface: %s", zef_last_error(ctx));
  const int64_t n = 1 << 18;
  const std::vector<float> pts(3 * n, 0.25f);
  std::vector<int32_t> lab(n);
  auto call = [&] { return zef_label_points(ctx, pts.data(), n, lab.data(), nullptr, nullptr, nullptr); };
  CHECK(call() == ZEF_OK, "call: %s", zef_last_error(ctx));
  const long resets = fake_launches("k_grid_reset");
  CHECK(call() == ZEF_OK && fake_launches("k_grid_reset") == resets, "a plain call clears lists that are empty");
  fake_fail_launch("k_grid_pending");
  CHECK(call() == ZEF_ERR_CUDA, "the failed launch was not reported");
  fake_fail_launch("");
  CHECK(zef_label_points(ctx, pts.data(), 100, lab.data(), nullptr, nullptr, nullptr) == ZEF_OK, "a call without lists: %s",
        zef_last_error(ctx));
  LabelPlan p;
  std::memset(&p.opts, 0, sizeof(p.opts));
  fill_default_opts(&p.opts);
  p.pts = ctx->lb.pts_tmp;
  p.labels = ctx->lb.labels_tmp;
  p.omega = nullptr;
  p.omega_ld = p.n_cap = n;
  p.d_n = p.d_off = ctx->lb.counters;
  p.timed = false;
  p.counted = false;
  CHECK(grid_enqueue(ctx, p) == ZEF_OK, "enqueue: %s", zef_last_error(ctx));
  CHECK(fake_launches("k_grid_reset") == resets + 1, "enqueueing did not clear the lists");
  CHECK(call() == ZEF_OK && fake_launches("k_grid_reset") == resets + 2, "the call behind a failure did not clear the lists");
  CHECK(call() == ZEF_OK && fake_launches("k_grid_reset") == resets + 2, "the lists are cleared for good");
  zef_destroy(ctx);
  return 0;
}

// The cells of all triangles' boxes, which registration goes through, stay in
// proportion to the triangles also where these are long and thin.
int needles() {
  Surface s;
  const int count = 2000;
  for (int i = 0; i < count; ++i) {  // tetrahedra from corner to corner, side by side
    const float x = 0.4f * (float)(i % 50), y = 0.4f * (float)(i / 50);
    const float v[4][3] = {{x, y, 0.f}, {x + 0.01f, y, 0.f}, {x, y + 0.01f, 0.f}, {x + 100.f, y + 100.f, 100.f}};
    for (auto &p : v) s.v.insert(s.v.end(), p, p + 3);
    const int32_t b = 4 * i;
    s.t.insert(s.t.end(), {b, b + 2, b + 1, b, b + 1, b + 3, b + 1, b + 2, b + 3, b + 2, b, b + 3});
  }
  zef_ctx *ctx = nullptr;
  CHECK(zef_create(&ctx, 0, nullptr) == ZEF_OK, "create");
  for (const Surface &q : {s, octahedron(50.f, 40)}) {
    CHECK(add(ctx, (int)ctx->comps.size() + 1, q) == ZEF_OK, "surface: %s", zef_last_error(ctx));
    const CompHost &h = ctx->comps.back();
    const CompGrid &g = ctx->grids.back();
    double cells = 0.0;
    for (size_t t = 0; t < q.t.size(); t += 3) {
      double box = 1.0;
      for (int k = 0; k < 3; ++k) {
        float lo = 1e30f, hi = -1e30f;
        for (int c = 0; c < 3; ++c) {
          lo = std::min(lo, q.v[3 * q.t[t + c] + k]);
          hi = std::max(hi, q.v[3 * q.t[t + c] + k]);
        }
        box *= std::floor((hi - h.lo[k]) * g.inv[k]) - std::floor((lo - h.lo[k]) * g.inv[k]) + 1.0;
      }
      cells += box;
    }
    const double nt = (double)q.t.size() / 3.0;
    CHECK(cells <= 67108864.0 + 1024.0 * nt, "%.3g cells in the boxes of %.0f triangles (grid of %d x %d x %d)", cells, nt,
          g.n[0], g.n[1], g.n[2]);
    CHECK(g.usable && g.n[0] >= 8, "no grid, or one of %d cells a side", g.n[0]);
  }
  CHECK(ctx->grids[1].n[0] > 50, "the octahedron's cells grew: %d a side", ctx->grids[1].n[0]);
  zef_destroy(ctx);
  return 0;
}

// A small host call without page-locked memory to be had takes the way of the
// large ones.
int no_pinned_memory() {
  const std::vector<float> pts(300, 0.25f);
  std::vector<int32_t> lab(100, -7);
  zef_ctx *ctx = nullptr;
  CHECK(zef_create(&ctx, 0, nullptr) == ZEF_OK, "create");
  CHECK(add(ctx, 1, octahedron(1.f, 3)) == ZEF_OK, "surface: %s", zef_last_error(ctx));
  fake_fail_pinned(true);
  for (int k = 0; k < 2; ++k)
    CHECK(zef_label_points(ctx, pts.data(), 100, lab.data(), nullptr, nullptr, nullptr) == ZEF_OK, "call %d: %s", k,
          zef_last_error(ctx));
  fake_fail_pinned(false);
  CHECK(!ctx->h_stage, "page-locked memory from nowhere");
  CHECK(zef_label_points(ctx, pts.data(), 100, lab.data(), nullptr, nullptr, nullptr) == ZEF_OK && ctx->h_stage,
        "the next call: %s", zef_last_error(ctx));
  zef_destroy(ctx);
  return 0;
}

}  // namespace

int main(int argc, char **argv) {
  const std::string name = argc > 1 ? argv[1] : "";
  if (name == "out_of_memory") out_of_memory();
  else if (name == "uploads") uploads();
  else if (name == "status_once") status_once();
  else if (name == "no_tets") no_tets();
  else if (name == "anchors_cut_short") anchors_cut_short();
  else if (name == "scratch_given_back") scratch_given_back();
  else if (name == "priority_uploads") priority_uploads();
  else if (name == "sums_beyond_32_bits") sums_beyond_32_bits();
  else if (name == "lists_cleared_after_a_failure") lists_cleared_after_a_failure();
  else if (name == "needles") needles();
  else if (name == "no_pinned_memory") no_pinned_memory();
  else return 2;
  return g_bad ? 1 : 0;
}
