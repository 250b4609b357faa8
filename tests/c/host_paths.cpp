// Drives the library's host code on the CPU (fake_cuda.h in place of the CUDA
// runtime). One path per argument; exits 0 if it holds.
#include "fake_cuda.h"

#include <algorithm>

#include "vplbm.h"
#include "vplbm_params.h"

using vplbm::ReduceArgs;

#define CHECK(cond)                                                  \
  do {                                                               \
    if (!(cond)) {                                                   \
      fprintf(stderr, "%s:%d: %s\n", __FILE__, __LINE__, #cond);     \
      return 1;                                                      \
    }                                                                \
  } while (0)

static vplbm_solver* create(int nx, int ny, int storage = VPLBM_F32) {
  vplbm_config c;
  vplbm_config_init(&c);
  c.nx = nx;
  c.ny = ny;
  c.storage = storage;
  c.collision = VPLBM_MRT;
  c.tau = 0.6;
  c.force_ring_len = 256;
  vplbm_solver* s = nullptr;
  if (vplbm_create(&c, &s) != VPLBM_OK) return nullptr;
  g_launches.clear();
  return s;
}

// (t0, steps) of each sum of records launched so far.
static std::vector<std::pair<long long, long long>> sums() {
  std::vector<std::pair<long long, long long>> r;
  for (const auto& l : g_launches)
    if (l.arg.size() == sizeof(ReduceArgs) && l.kernel.find("reduce_kernel") != std::string::npos) {
      ReduceArgs a;
      memcpy(&a, l.arg.data(), sizeof(a));
      r.push_back({a.t0, a.steps});
    }
  return r;
}
using Sums = std::vector<std::pair<long long, long long>>;

// A call that runs out of memory after some of its steps has still summed
// their records.
static int records_of_a_failed_call(int nx, int ny) {
  vplbm_solver* s = create(nx, ny);
  CHECK(s);
  CHECK(vplbm_enable_timing(s, 1) == VPLBM_OK);
  g_fail_at["cudaEventCreate"] = 5;  // two events a launch: the third launch's first
  CHECK(vplbm_step(s, 6) == VPLBM_ERR_NOMEM);
  const long long made = vplbm_step_count(s);
  CHECK(made == (nx * ny > 4000000 ? 4 : 2));  // large FP32 grids: two steps a launch
  CHECK((sums() == Sums{{0, made}}));
  double fx[8];
  int64_t n = 0;
  CHECK(vplbm_forces(s, fx, nullptr, nullptr, 8, &n) == VPLBM_OK && n == made);
  CHECK(vplbm_step(s, 3) == VPLBM_OK && vplbm_step_count(s) == made + 3);
  CHECK((sums() == Sums{{0, made}, {made, 3}}));
  vplbm_destroy(s);
  return 0;
}

// The same where the sum's own launch fails: the next call makes it.
static int records_of_a_failed_sum() {
  vplbm_solver* s = create(300, 100);
  CHECK(s);
  g_fail_at["launch"] = 4;  // the third step
  CHECK(vplbm_step(s, 1) == VPLBM_OK);
  CHECK(vplbm_step(s, 5) == VPLBM_ERR_NOMEM && vplbm_step_count(s) == 2);
  CHECK((sums() == Sums{{0, 1}, {1, 1}}));
  g_fail_at["launch"] = 2;
  CHECK(vplbm_step(s, 1) == VPLBM_ERR_NOMEM && vplbm_step_count(s) == 3);  // its sum failed, then was made
  CHECK((sums() == Sums{{0, 1}, {1, 1}, {2, 1}}));
  vplbm_destroy(s);
  return 0;
}

// A captured call of n steps swaps the two population buffers as often as n
// single steps do (odd or even), and still makes n steps.
static int captured_pairs() {
  vplbm_solver* s = create(2049, 2049);
  CHECK(s);
  g_capturing = true;
  long long t = 0;
  for (int n = 1; n <= 9; ++n) {
    g_launches.clear();
    CHECK(vplbm_step(s, n) == VPLBM_OK);
    CHECK(vplbm_step_count(s) == (t += n));
    const int twos = launches_of("pair_step_kernel"), ones = launches_of("fused_step_kernel");
    CHECK(2 * twos + ones == n && (twos + ones) % 2 == n % 2);
    CHECK(twos >= n / 2 - 1);
  }
  vplbm_destroy(s);
  return 0;
}

// Setting bodies takes no memory, captured or not; the second mask of moving
// bodies is taken by the first call that pairs its steps outside capture.
static int second_mask(bool refuse) {
  vplbm_solver* s = create(2049, 2049);
  CHECK(s);
  vplbm_body b{};
  b.cx = b.cy = 1000.0;
  b.radius = 50.0;
  b.amp_y = 4.0;
  b.period = 100.0;
  const size_t allocs = g_allocs.size();
  for (bool captured : {true, false}) {
    g_capturing = captured;
    CHECK(vplbm_set_bodies(s, &b, 1) == VPLBM_OK && vplbm_step(s, 1) == VPLBM_OK && g_allocs.size() == allocs);
  }
  g_capturing = true;
  g_launches.clear();
  CHECK(vplbm_step(s, 4) == VPLBM_OK && g_allocs.size() == allocs);
  CHECK(launches_of("pair_step_kernel") == 0 && launches_of("fused_step_kernel") == 4);
  g_capturing = false;
  if (refuse) g_fail_at["cudaMallocAsync"] = 1;
  for (int call = 0; call < 2; ++call) {
    g_launches.clear();
    CHECK(vplbm_step(s, 4) == VPLBM_OK && g_allocs.size() == allocs + (refuse ? 0 : 1));
    CHECK(launches_of("pair_step_kernel") == (refuse ? 0 : 2) && launches_of("fused_step_kernel") == (refuse ? 4 : 0));
  }
  if (!refuse) CHECK(g_allocs.back() == size_t(2049) * 2080);  // a byte a node of padded rows
  vplbm_destroy(s);
  return 0;
}

// A buffer that a call does without leaves no error behind.
static int refused_buffers_are_no_error(int nx, int ny, bool moving) {
  vplbm_solver* s = create(nx, ny);
  CHECK(s);
  vplbm_body b{};
  b.radius = 5.0;
  b.amp_y = 4.0;
  b.period = moving ? 100.0 : 0.0;
  CHECK(vplbm_set_bodies(s, &b, 1) == VPLBM_OK);
  for (const char* before : {"", "n must be >= 0"}) {
    if (*before) CHECK(vplbm_step(s, -1) == VPLBM_ERR_INVALID);
    g_fail_at["cudaMallocAsync"] = 1;
    CHECK(vplbm_step(s, 40) == VPLBM_OK);
    CHECK(*before || g_fail_at["cudaMallocAsync"] == 0);  // asked for, once
    CHECK(strcmp(vplbm_last_error(s), before) == 0);
  }
  vplbm_destroy(s);
  return 0;
}

// Stepping takes at most 8 MiB beyond what creation took, whatever the grid,
// and no window of records is longer than what was taken (a tile's scratch at
// creation holds 64 partials, eight steps of eight units).
static int bounded_window(int nx, int ny, int storage) {
  vplbm_solver* s = create(nx, ny, storage);
  CHECK(s);
  const size_t allocs = g_allocs.size();
  for (int n : {1, 8, 200, 9}) CHECK(vplbm_step(s, n) == VPLBM_OK);
  size_t late = 0;
  for (size_t i = allocs; i < g_allocs.size(); ++i) late += g_allocs[i];
  CHECK(late <= size_t(8) << 20);
  long long t = 0;
  for (const auto& l : g_launches) {
    if (l.arg.empty()) continue;
    ReduceArgs a;
    memcpy(&a, l.arg.data(), sizeof(a));
    CHECK(a.t0 == t);
    t += a.steps;
    const size_t bytes = size_t(a.steps) * a.n_tiles * (a.units ? a.units : 1) * 24;
    CHECK(bytes <= std::max(late, size_t(a.n_tiles) * 64 * 24));
  }
  CHECK(t == 218);
  vplbm_destroy(s);
  return 0;
}

// A grouped call takes one buffer and makes one copy for its tables, whatever
// the storages and schemes of its solvers.
static int grouped_tables() {
  vplbm_config c;
  vplbm_config_init(&c);
  c.tau = 0.6;
  c.stream = reinterpret_cast<void*>(8);
  vplbm_solver* s[3];
  int64_t steps[3] = {3, 1, 2};
  for (int i = 0; i < 3; ++i) {
    c.nx = 300 + i;
    c.ny = 70;
    c.storage = i == 0 ? VPLBM_F16_OFFSET : VPLBM_F32;
    c.streaming = i == 2 ? VPLBM_STREAM_AA : VPLBM_STREAM_AB;
    CHECK(vplbm_create(&c, &s[i]) == VPLBM_OK);
  }
  g_calls.clear();
  CHECK(vplbm_group_step(s, 3, steps) == VPLBM_OK);
  CHECK(g_calls["cudaMallocAsync"] == 1 && g_calls["cudaMemcpyAsync"] == 1);
  for (int i = 0; i < 3; ++i) CHECK(vplbm_step_count(s[i]) == steps[i]);
  for (vplbm_solver* v : s) vplbm_destroy(v);
  return 0;
}

// The name of the step kernel is that of the launches a call makes.
static int named_kernel() {
  for (int storage : {VPLBM_F64, VPLBM_F32, VPLBM_F16_OFFSET})
    for (int nx : {300, 1200, 2049})
      for (int rows : {0, 8, 32})
        for (bool exchange : {false, true}) {
          vplbm_config c;
          vplbm_config_init(&c);
          c.nx = nx;
          c.ny = nx;
          c.tau = 0.6;
          c.storage = storage;
          c.tile_rows = rows;
          vplbm_solver* s = nullptr;
          CHECK(vplbm_create(&c, &s) == VPLBM_OK);
          CHECK(vplbm_enable_momentum_exchange(s, exchange) == VPLBM_OK);
          g_launches.clear();
          CHECK(vplbm_step(s, 2) == VPLBM_OK);
          CHECK(launches_of(vplbm_step_kernel(s)) == (strcmp(vplbm_step_kernel(s), "pair_step_kernel") ? 2 : 1));
          CHECK(launches_of("_step_kernel") == launches_of(vplbm_step_kernel(s)));
          vplbm_destroy(s);
        }
  return 0;
}

int main(int argc, char** argv) {
  g_keep["reduce_kernel"] = sizeof(ReduceArgs);
  const std::string path = argc > 1 ? argv[1] : "";
  if (path == "failed_call") return records_of_a_failed_call(300, 100);
  if (path == "failed_call_vector") return records_of_a_failed_call(2048, 512);
  if (path == "failed_call_pairs") return records_of_a_failed_call(2049, 2049);
  if (path == "failed_sum") return records_of_a_failed_sum();
  if (path == "captured_pairs") return captured_pairs();
  if (path == "second_mask") return second_mask(false);
  if (path == "second_mask_refused") return second_mask(true);
  if (path == "refused_window") return refused_buffers_are_no_error(300, 100, false);
  if (path == "refused_mask") return refused_buffers_are_no_error(2049, 2049, true);
  if (path == "window_f64") return bounded_window(2048, 1024, VPLBM_F64);
  if (path == "window_f64_mid") return bounded_window(1024, 512, VPLBM_F64);
  if (path == "window_f32") return bounded_window(700, 700, VPLBM_F32);
  if (path == "window_f16") return bounded_window(128, 64, VPLBM_F16_OFFSET);
  if (path == "grouped_tables") return grouped_tables();
  if (path == "named_kernel") return named_kernel();
  fprintf(stderr, "no such path: %s\n", path.c_str());
  return 2;
}
