// Scenarios of test_host_calls.py: the library's host side on the runtime of
// fake_cudart.h. Exit code 0: the scenario holds; else the reasons are printed.
#include "fake_cudart.h"

#include "gsr.h"
#include "gsr_pmm.h"
#include "gsr_pnp.h"

static int failed = 0;
#define CHECK(x)                                                \
  do {                                                          \
    if (!(x)) {                                                 \
      std::printf("line %d: %s (%s)\n", __LINE__, #x, gs_last_error()); \
      ++failed;                                                 \
    }                                                           \
  } while (0)

static gs_camera camera(int w, int h) {
  gs_camera c{};
  c.fx = c.fy = (float)w;
  c.cx = 0.5f * w;
  c.cy = 0.5f * h;
  c.width = w;
  c.height = h;
  return c;
}
static gs_pose pose(double z) {
  gs_pose p{};
  for (int i = 0; i < 4; ++i) p.T_cw[5 * i] = 1.0;
  p.T_cw[11] = z;
  return p;
}
static gs_scene* scene(int64_t n, int feat_dim = 0) {
  static std::vector<float> v(4096, 0.5f);
  gs_scene_desc d{};
  d.n = n;
  d.feat_dim = feat_dim;
  d.feats_bf16 = feat_dim ? (const uint16_t*)v.data() : nullptr;
  d.means = d.scales = d.quats = d.opacities = d.sh = v.data();
  d.device_resident = 1;
  gs_scene* s = nullptr;
  CHECK(gs_create_scene(&d, &s) == GS_OK);
  return s;
}

// Asynchronous replays of one size after another: the table of a replay that
// has not run yet is neither freed nor overwritten when the next size is captured.
static void batches_of_changing_size() {
  gs_scene* s = scene(100);
  for (int k = 0; k < 6; ++k) {
    const gs_camera c[2] = {camera(64 + 32 * (k % 3), 64), camera(32, 32)};
    const gs_pose p[2] = {pose(k), pose(1)};
    const gs_outputs o[2] = {};
    CHECK(gs_render_batch(s, 2, c, p, o, GS_BATCH_GRAPH, nullptr) == GS_OK);
  }
  cudaDeviceSynchronize();
  gs_destroy_scene(s);
}

// A second device of the process: kernels with large shared memory are allowed it
// there too, and the persistent grids are that device's.
static void two_devices() {
  static float maps[2][32 * 64 * 64] __attribute__((aligned(16))), image[32 * 256 * 256];
  for (int d = 0; d < 2; ++d) {
    cudaSetDevice(d);
    gs_scene* s = scene(100, 32);
    gs_outputs o{};
    o.feats = image;
    const gs_camera c = camera(1920, 1080);
    const gs_pose p = pose(0);
    CHECK(gs_render(s, &c, &p, &o, nullptr) == GS_OK);
    CHECK(fake::count["grid k_composite"] == 152 * fake::occupancy[d]);
    std::vector<uint8_t> mask(100);
    CHECK(gs_visibility(s, &c, &p, mask.data(), nullptr, nullptr, nullptr, nullptr, nullptr, nullptr) == GS_OK);
    CHECK(fake::count["grid k_vis_backward"] == 152 * fake::occupancy[d]);
    gs_destroy_scene(s);
    gs_pmm* m = nullptr;
    CHECK(gs_pmm_create(32, 64, 64, &m) == GS_OK);
    gs_pmm_result r{};
    CHECK(gs_pmm_match(m, maps[0], maps[1], 0.1f, &r, nullptr) == GS_OK);
    gs_pmm_destroy(m);
  }
}

// A kernel that may start early stands directly behind another kernel of its
// stream: also without Gaussians, without matches, and at a refinement's start.
static void early_starts() {
  static float image[4 * 64 * 64];
  static int32_t matches[3 * 64];
  static uint32_t words[3 * 8];
  const gs_camera c = camera(64, 64);
  for (int n : {0, 100}) {
    gs_scene* s = scene(n);
    const gs_outputs o{};
    double loss, grad[6];
    for (int timed = 0; timed < 2; ++timed) {
      CHECK(gs_scene_set_timing(s, timed) == GS_OK);
      for (int k = 0; k < 40; ++k) {
        const gs_pose p = pose(k);
        CHECK(gs_render(s, &c, &p, &o, nullptr) == GS_OK);
        CHECK(gs_render_pose_grad(s, &c, &p, image, image, nullptr, 1.0f, nullptr, &loss, grad, nullptr) == GS_OK);
        CHECK(gs_render_batch(s, 1, &c, &p, &o, GS_BATCH_GRAPH, nullptr) == GS_OK);
      }
      gs_refine_opts ro = gs_refine_defaults();
      ro.iterations = 3;
      gs_pose p = pose(0);
      CHECK(gs_refine_pose(s, &c, &p, image, image, nullptr, &ro, nullptr, nullptr) == GS_OK);
    }
    gs_destroy_scene(s);
  }
  gs_pnp* q = nullptr;
  CHECK(gs_pnp_create(64, 8, &q) == GS_OK);
  const gs_pnp_opts po = gs_pnp_defaults();
  const gs_pose p = pose(0);
  gs_pnp_result r{};
  for (int n : {0, 64})
    for (int h : {0, 8}) CHECK(gs_pnp_solve(q, &c, &p, image, image, matches, n, words, h, &po, &r, nullptr) == GS_OK);
  gs_pnp_destroy(q);
}

static void render(gs_scene* s, const gs_camera& c) {
  const gs_outputs o{};
  const gs_pose p = pose(0);
  CHECK(gs_render(s, &c, &p, &o, nullptr) == GS_OK);
}

// Synchronous calls are captured once their size has come up often enough (a
// gradient, whose replay saves more, sooner), and only once: not again for a size
// that comes back, and never for sizes that are many.
static void sizes_in_pairs() {
  gs_scene* s = scene(100);
  fake::count.clear();
  for (int k = 0; k < 100; ++k)
    for (int w : {64, 64, 96, 96}) render(s, camera(w, 64));
  CHECK(fake::count["captures"] == 2);
  CHECK(fake::count["replays"] >= 380);
  const int mallocs = fake::count["cudaMallocHost"];
  for (int k = 0; k < 400; ++k) render(s, camera(32 + 16 * (k / 2 % 20), 32));  // 20 sizes
  CHECK(fake::count["captures"] == 2);
  CHECK(fake::count["cudaMallocHost"] == mallocs);
  for (int w = 0; w < 3; ++w)  // a size rendered twice by each of many scenes
    for (int k = 0; k < 10; ++k) {
      gs_scene* t = scene(10);
      render(t, camera(64, 64));
      render(t, camera(64, 64));
      gs_destroy_scene(t);
    }
  CHECK(fake::count["captures"] == 2);
  static float image[4 * 64 * 64];
  const gs_camera c = camera(64, 64);
  const gs_pose p = pose(0);
  double loss, grad[6];
  for (int k = 0; k < 5; ++k) {
    const int before = fake::count["replays"];
    CHECK(gs_render_pose_grad(s, &c, &p, image, image, nullptr, 1.0f, nullptr, &loss, grad, nullptr) == GS_OK);
    CHECK(fake::count["replays"] == before + (k >= 2));
  }
  CHECK(fake::count["captures"] == 3);
  gs_destroy_scene(s);
}

// A scene's graphs outlive whatever other scenes allocate or are told to launch.
static void other_scenes() {
  gs_scene* s = scene(100);
  const gs_camera c = camera(64, 64);
  const gs_pose p[2] = {pose(0), pose(1)};
  const gs_outputs o[2] = {};
  const gs_camera cs[2] = {c, c};
  CHECK(gs_render_batch(s, 2, cs, p, o, GS_BATCH_GRAPH, nullptr) == GS_OK);
  for (int k = 0; k < 40; ++k) render(s, c);
  fake::count.clear();
  for (int k = 0; k < 40; ++k) {
    gs_scene* t = scene(10);
    render(t, camera(64 + 16 * k, 64));
    gs_launch cfg{};
    cfg.grid_mult = 4;
    CHECK(gs_scene_set_launch(t, GS_MODE_FORWARD, 1, &c, &cfg) == GS_OK);
    gs_destroy_scene(t);
    render(s, c);
    CHECK(gs_render_batch(s, 2, cs, p, o, GS_BATCH_GRAPH, nullptr) == GS_OK);
  }
  CHECK(fake::count["captures"] == 0);
  CHECK(fake::count["replays"] == 80);
  gs_launch cfg{};
  cfg.grid_mult = 4;
  CHECK(gs_scene_set_launch(s, GS_MODE_FORWARD, 1, &c, &cfg) == GS_OK);  // its own: captured again
  for (int k = 0; k < 40; ++k) render(s, c);
  CHECK(fake::count["captures"] == 1);
  gs_destroy_scene(s);
}

// A warmed scene's synchronous calls allocate nothing that they cannot do
// without: with no memory for a graph or its page-locked table they go on plain.
static void no_memory_for_graphs() {
  static float image[4 * 64 * 64];
  const gs_camera c = camera(64, 64);
  const gs_pose p = pose(0);
  double loss, grad[6];
  for (bool* gone : {&fake::no_pinned, &fake::no_graphs}) {
    gs_scene* s = scene(100);
    render(s, c);
    CHECK(gs_render_pose_grad(s, &c, &p, image, image, nullptr, 1.0f, nullptr, &loss, grad, nullptr) == GS_OK);
    fake::count.clear();
    *gone = true;
    for (int k = 0; k < 40; ++k) {
      render(s, c);
      CHECK(gs_render_pose_grad(s, &c, &p, image, image, nullptr, 1.0f, nullptr, &loss, grad, nullptr) == GS_OK);
    }
    CHECK(fake::count["replays"] == 0 && fake::count["kernel k_project"] >= 80);
    *gone = false;
    for (int k = 0; k < 20; ++k) render(s, c);
    CHECK(fake::count["replays"] > 0);
    CHECK(cudaGetLastError() == cudaSuccess);
    gs_destroy_scene(s);
  }
}

// A call recorded by the caller's own capture has not run: the tile counters of
// a new workspace are still cleared by the next call.
static void callers_capture() {
  gs_scene* s = scene(100);
  const gs_camera c = camera(64, 64);
  const gs_pose p = pose(0);
  const gs_outputs o{};
  cudaStream_t st;
  cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
  cudaGraph_t g;
  cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal);
  CHECK(gs_render_async(s, &c, &p, &o, st) == GS_OK);
  cudaStreamEndCapture(st, &g);
  const int sets = fake::count["cudaMemsetAsync"];
  render(s, c);
  CHECK(fake::count["cudaMemsetAsync"] == sets + 1);
  render(s, c);
  CHECK(fake::count["cudaMemsetAsync"] == sets + 1);
  cudaGraphDestroy(g);
  cudaStreamDestroy(st);
  gs_destroy_scene(s);
}

int main(int argc, char** argv) {
  const std::map<std::string, void (*)()> all = {{"batches_of_changing_size", batches_of_changing_size},
                                                    {"two_devices", two_devices},
                                                    {"early_starts", early_starts},
                                                    {"sizes_in_pairs", sizes_in_pairs},
                                                    {"other_scenes", other_scenes},
                                                    {"no_memory_for_graphs", no_memory_for_graphs},
                                                    {"callers_capture", callers_capture}};
  const auto it = all.find(argc > 1 ? argv[1] : "");
  if (it == all.end()) return 2;
  it->second();
  for (const std::string& v : fake::violations) std::printf("%s\n", v.c_str());
  return failed || !fake::violations.empty() ? 1 : 0;
}
