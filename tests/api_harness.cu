// The host side of the library (lbm_api.cu) on a machine without a GPU: the
// kernel launchers and the CUDA runtime are replaced by fakes that work on
// host memory, note what was launched and return the error codes a check asks
// for.  `api_harness NAME` runs one check and prints "ok".  Built and run by
// test_api_host.py.
#include <cstdio>
#include <cstring>

#include <sys/mman.h>

#include "api_fakes.h"
#include "lbm.h"
#include "lbm_internal.cuh"

static int failures = 0;
#define CHECK(c)                                              \
  do {                                                        \
    if (!(c)) {                                               \
      std::printf("FAIL line %d: %s\n", __LINE__, #c);        \
      ++failures;                                             \
    }                                                         \
  } while (0)

// ---- launchers ----

static hmcsc::FieldsOut last_fields;
static unsigned *last_fault_host;  // of the workspace density was last launched on

namespace hmcsc {
size_t workspace_bytes(long long nx, long long ny, long long nz, int, bool pc, Workspace *w, char *b) {
  const Tiling t = tiling(nx, ny, nz);
  const size_t nt = (size_t)t.ntiles * kTile, f = (size_t)t.ntiles * kTileFloats * 4;
  if (w) {
    w->f = b;
    w->rho = (float2 *)(b + f);
    w->rho_enc = w->rho + nt;
    w->ns = (float *)(w->rho_enc + nt);
    w->ads = w->ns + nt;
    w->ns2 = pc ? w->ads + nt : nullptr;
    w->ads2 = pc ? w->ads + 2 * nt : nullptr;
    w->stage = w->ads + 3 * nt;
    w->red = (double *)(w->stage + 6 * t.nlin);
    w->fault = (unsigned *)(w->red + kRedBlocks * kRedK);
    w->wave = w->fault + 64;
    w->fault_host = nullptr;
  }
  return f + nt * (16 + 16) + 24 * (size_t)t.nlin + 8 * kRedBlocks * kRedK + 1024;
}
cudaError_t launch_init_equilibrium(const StepParams &, const Workspace &, const float *, const float *,
                                    cudaStream_t) { return launch("init"); }
cudaError_t launch_geometry(const StepParams &, const Workspace &, const float *, const float *, const float *,
                            cudaStream_t) { return launch("geometry"); }
cudaError_t launch_density(const StepParams &, const Workspace &w, int, int, cudaStream_t) {
  last_fault_host = w.fault_host;
  return launch("density");
}
cudaError_t launch_collide_stream(const StepParams &, const Workspace &, int, int, cudaStream_t) {
  return launch("collide");
}
// field k of node n is 1000 k + n
static void write_fields(const StepParams &p, const FieldsOut &out) {
  last_fields = out;
  const long long N = (long long)p.nx * p.ny * p.nz;
  for (int k = 0; k < 6; ++k)
    for (long long n = 0; out.p[k] && n < N; ++n) {
      const float v = 1000.0f * k + n;
      memcpy((char *)out.p[k] + 4 * n, &v, 4);
    }
}
cudaError_t launch_fields(const StepParams &p, const Workspace &, int, const FieldsOut &out, cudaStream_t) {
  write_fields(p, out);
  return launch("fields");
}
cudaError_t launch_density_fields(const StepParams &p, const Workspace &, const FieldsOut &out, cudaStream_t) {
  write_fields(p, out);
  return launch("density_fields");
}
cudaError_t launch_single_pass(const StepParams &, const Workspace &, int, int, cudaStream_t) {
  return launch("single_pass");
}
cudaError_t launch_wave(const StepParams &, const Workspace &, int, int, int, unsigned, long long, cudaStream_t) {
  return launch("wave");
}
cudaError_t launch_wave_batch(const WaveJob &, int, cudaStream_t) { return launch("wave_batch"); }
cudaError_t launch_resident(const StepParams &, const Workspace &, int, int, unsigned, bool, cudaStream_t) {
  return launch("resident");
}
cudaError_t launch_batch_density(const BatchArgs &, int, cudaStream_t) { return launch("batch_density"); }
cudaError_t launch_batch_collide(const BatchArgs &, int, cudaStream_t) { return launch("batch_collide"); }
cudaError_t launch_batch_collide_pipe(const BatchArgs &, int, int, int, cudaStream_t) {
  return launch("batch_collide_pipe");
}
cudaError_t launch_populations(const StepParams &p, const Workspace &, int, float *out, int k0, int nk,
                               cudaStream_t) {
  const long long N = (long long)p.nx * p.ny * p.nz;
  for (int k = 0; k < nk; ++k)
    for (long long n = 0; n < N; ++n) out[k * N + n] = 1000.0f * (k0 + k) + n;
  return launch("populations");
}
cudaError_t launch_reduce(const StepParams &, const Workspace &, ReduceResult *out, cudaStream_t) {
  memset(out, 0, sizeof *out);
  return launch("reduce");
}
}  // namespace hmcsc

// ---- checks ----

struct Lattice {
  lbm_ctx *ctx = nullptr;
  std::vector<char> ws;
  long long N;
  Lattice(int nx, int ny, int nz, int storage = LBM_STORAGE_F32) : N((long long)nx * ny * nz) {
    lbm_params p = {};
    p.nx = nx, p.ny = ny, p.nz = nz, p.storage = storage;
    p.tau[0] = p.tau[1] = 1.0;
    p.G = 1.75;
    const size_t n = lbm_workspace_bytes(&p);
    ws.resize(n + 256);
    char *at = (char *)(((uintptr_t)ws.data() + 255) / 256 * 256);
    CHECK(lbm_create(&p, at, n, nullptr, &ctx) == LBM_OK);
    const std::vector<float> one(N, 1.0f), zero(N, 0.0f);
    CHECK(lbm_set_geometry(ctx, zero.data(), nullptr) == LBM_OK);
    CHECK(lbm_init_equilibrium(ctx, one.data(), one.data()) == LBM_OK);
    launched.clear();
  }
  ~Lattice() { lbm_destroy(ctx); }
};

// A pinned destination that does not start on a float gets its fields through
// the staging planes: a kernel cannot store floats there.
static void misaligned_destination() {
  for (const int nx : {8, 64}) {            // through the buffer, and too large for it
    Lattice l(nx, 32, 16);
    std::vector<char> mem(5 * 4 * l.N + 64);
    ranges = {{mem.data(), mem.size(), cudaMemoryTypeHost, 0}};
    for (const int off : {0, 1, 2, 3}) {
      char *at = (char *)(((uintptr_t)mem.data() + 15) / 16 * 16) + off;
      for (const bool u : {false, true}) {
        memset(mem.data(), 0, mem.size());
        CHECK(lbm_read_fields(l.ctx, (float *)at, nullptr, u ? (float *)(at + 4 * l.N) : nullptr,
                              (float *)(at + 16 * l.N)) == LBM_OK);
        for (const float *p : last_fields.p) CHECK((uintptr_t)p % sizeof(float) == 0);
        if (nx == 64 && off == 0) CHECK(last_fields.p[0] == (float *)at);  // written in place
        for (const int k : {0, 2, 3, 4, 5}) {
          if (!u && k > 1 && k < 5) continue;
          float v;
          memcpy(&v, at + 4 * ((k == 0 ? 0 : k == 5 ? 4 : k - 1) * l.N + l.N - 1), 4);
          CHECK(v == 1000.0f * k + (l.N - 1));
        }
      }
    }
    ranges.clear();
  }
}

// An address the host cannot write is refused by the copy to it, whatever the
// lattice's size; the host never writes there itself.
static void device_destination() {
  for (const int nx : {8, 64}) {
    Lattice l(nx, 32, 16);
    const size_t bytes = 4 * 38 * l.N;
    float *at = (float *)mmap(nullptr, bytes, PROT_NONE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
    CHECK(at != MAP_FAILED);
    ranges = {{(const char *)at, bytes, cudaMemoryTypeDevice, 0}};
    std::vector<float> host(38 * l.N);
    CHECK(lbm_read_fields(l.ctx, at, nullptr, nullptr, nullptr) == LBM_ECUDA);
    CHECK(lbm_read_fields(l.ctx, nullptr, at, nullptr, nullptr) == LBM_ECUDA);
    CHECK(lbm_read_fields(l.ctx, host.data(), nullptr, at, nullptr) == LBM_ECUDA);
    CHECK(lbm_read_fields(l.ctx, nullptr, nullptr, nullptr, at) == LBM_ECUDA);
    CHECK(lbm_get_populations(l.ctx, at) == LBM_ECUDA);
    CHECK(lbm_read_fields(l.ctx, host.data(), nullptr, nullptr, host.data() + l.N) == LBM_OK);
    CHECK(host[l.N - 1] == l.N - 1 && host[l.N] == 5000.0f);
    CHECK(lbm_get_populations(l.ctx, host.data()) == LBM_OK);
    CHECK(host[37 * l.N] == 37000.0f);
    ranges.clear();
    munmap(at, bytes);
  }
}

// Where the launch lbm_step chose by itself is refused, the steps run as two
// passes, from then on without asking again; a step the caller asked for
// reports the error.
static void refused_choice() {
  const struct { int nx, ny, nz; const char *name; } own[] = {{32, 32, 32, "resident"}, {128, 128, 128, "wave"}};
  for (const auto &o : own)
    for (const cudaError_t e : {cudaErrorCooperativeLaunchTooLarge, cudaErrorLaunchOutOfResources}) {
      Lattice l(o.nx, o.ny, o.nz);
      CHECK(lbm_step(l.ctx, 1) == LBM_OK);
      CHECK(launched[o.name] == 1 && launched["density"] == 0);
      refused = {{o.name, e}};
      CHECK(lbm_step(l.ctx, 3) == LBM_OK);
      CHECK(cudaGetLastError() == cudaSuccess);
      CHECK(launched["density"] == 3 && launched["collide"] == 3);
      CHECK(lbm_time(l.ctx) == 4);
      refused.clear();
      CHECK(lbm_step(l.ctx, 2) == LBM_OK);
      CHECK(launched["density"] == 5 && launched[o.name] == 1);
    }
  Lattice l(32, 32, 32);
  CHECK(lbm_set_wavefront(l.ctx, 2, 4) == LBM_OK);
  refused = {{"wave", cudaErrorCooperativeLaunchTooLarge}};
  CHECK(lbm_step(l.ctx, 1) == LBM_ECUDA);
  refused = {{"density", cudaErrorIllegalAddress}, {"resident", cudaErrorIllegalAddress}};
  Lattice m(32, 32, 32);
  CHECK(lbm_step(m.ctx, 1) == LBM_ECUDA);  // an error of the context stays one
  refused.clear();
}

// After a wait that ran out no call advances the state, until a new one is set.
static void undefined_state() {
  Lattice l(32, 32, 32), other(32, 32, 32);
  lbm_ctx *both[2] = {other.ctx, l.ctx};
  lbm_graph *g = nullptr;
  CHECK(lbm_batch_graph_create(both, 2, 2, (void *)1, &g) == LBM_OK);
  CHECK(lbm_batch_graph_launch(g, (void *)1) == LBM_OK);
  CHECK(lbm_density(l.ctx) == LBM_OK);
  *last_fault_host = LBM_FAULT_WAIT;
  launched.clear();
  CHECK(lbm_step(l.ctx, 1) == LBM_EINTERNAL);
  CHECK(lbm_collide_stream(l.ctx) == LBM_EINTERNAL);
  CHECK(lbm_density(l.ctx) == LBM_EINTERNAL);
  CHECK(lbm_batch_step(both, 2, 2, (void *)1) == LBM_EINTERNAL);
  CHECK(lbm_batch_graph_launch(g, (void *)1) == LBM_EINTERNAL);
  CHECK(launched.empty());
  CHECK(lbm_time(l.ctx) == 2 && lbm_time(other.ctx) == 2);
  CHECK(strlen(lbm_last_error(l.ctx)) > 0);
  const std::vector<float> one(l.N, 1.0f);
  for (lbm_ctx *c : both) CHECK(lbm_init_equilibrium(c, one.data(), one.data()) == LBM_OK);
  CHECK(lbm_batch_graph_launch(g, (void *)1) == LBM_OK);
  CHECK(lbm_density(l.ctx) == LBM_OK && lbm_collide_stream(l.ctx) == LBM_OK);
  CHECK(lbm_time(l.ctx) == 3);
  lbm_batch_graph_destroy(g);
}

// Asking for no wavefront, no single pass, or for launch shapes asks for the
// two passes; lbm_set_automatic_step gives the choice back to the library.
static void step_choice() {
  const struct { int nx, ny, nz; const char *name; } own[] = {{32, 32, 32, "resident"}, {128, 128, 128, "wave"}};
  for (const auto &o : own) {
    Lattice l(o.nx, o.ny, o.nz);
    int first[3], cfg[3], shape, lag;
    CHECK(lbm_get_launch_config(l.ctx, &first[0], &first[1], &first[2]) == LBM_OK);
    const auto takes = [&](const char *name) {
      launched.clear();
      CHECK(lbm_step(l.ctx, 1) == LBM_OK);
      return launched.size() == 1 + !strcmp(name, "density") && launched[name] == 1;
    };
    CHECK(takes(o.name));
    CHECK(lbm_set_wavefront(l.ctx, 0, 0) == LBM_OK);
    CHECK(takes("density"));
    CHECK(lbm_set_automatic_step(l.ctx) == LBM_OK);
    CHECK(takes(o.name));
    CHECK(lbm_set_single_pass(l.ctx, 3) == LBM_OK);
    CHECK(takes("single_pass"));
    CHECK(lbm_set_single_pass(l.ctx, 0) == LBM_OK);
    CHECK(takes("density"));
    CHECK(lbm_set_wavefront(l.ctx, 1, 5) == LBM_OK);
    CHECK(takes("wave"));
    CHECK(lbm_set_automatic_step(l.ctx) == LBM_OK);
    CHECK(takes(o.name));
    CHECK(lbm_get_wavefront(l.ctx, &shape, &lag) == LBM_OK);
    CHECK(shape == 0 && lag == hmcsc::kWaveLagDefault);
    CHECK(lbm_set_launch_config(l.ctx, 2, 3, 4) == LBM_OK);
    CHECK(takes("density"));
    CHECK(lbm_set_automatic_step(l.ctx) == LBM_OK);
    CHECK(takes(o.name));
    CHECK(lbm_get_launch_config(l.ctx, &cfg[0], &cfg[1], &cfg[2]) == LBM_OK);
    CHECK(memcmp(first, cfg, sizeof cfg) == 0);
    CHECK(lbm_set_launch_config(l.ctx, -1, 0, 0) == LBM_EINVAL);
    CHECK(takes(o.name));
  }
  CHECK(lbm_set_automatic_step(nullptr) == LBM_EINVAL);
}

int main(int argc, char **argv) {
  const std::string name = argc > 1 ? argv[1] : "";
  if (name == "misaligned_destination") misaligned_destination();
  else if (name == "device_destination") device_destination();
  else if (name == "refused_choice") refused_choice();
  else if (name == "undefined_state") undefined_state();
  else if (name == "step_choice") step_choice();
  else return std::printf("no check '%s'\n", name.c_str()), 2;
  if (failures == 0) std::printf("ok\n");
  return failures != 0;
}
