// Scenarios of test_host_calls.py: the library's host side on the runtime of
// fake_cudart.h. Exit code 0: the scenario holds; else the reasons are printed.
#include "fake_cudart.h"

#include "gsr.h"

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
static gs_scene* scene(int64_t n) {
  static std::vector<float> v(4096, 0.5f);
  gs_scene_desc d{};
  d.n = n;
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

int main(int argc, char** argv) {
  const std::map<std::string, void (*)()> all = {{"batches_of_changing_size", batches_of_changing_size}};
  const auto it = all.find(argc > 1 ? argv[1] : "");
  if (it == all.end()) return 2;
  it->second();
  for (const std::string& v : fake::violations) std::printf("%s\n", v.c_str());
  return failed || !fake::violations.empty() ? 1 : 0;
}
