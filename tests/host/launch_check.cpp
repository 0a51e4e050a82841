// The host side of the library against launches that the runtime refuses (fake_cudart.h).
// usage: launch_check <check>; exit status 0 if it holds.
#include "fake_cudart.h"

#include <cstdio>
#include <string>
#include <vector>

#include "../../paper_1508_04596_gb300/csrc/nc_internal.cuh"

static int report(const char* what, bool ok) {
  std::printf("%s: %s\n", what, ok ? "ok" : "FAILED");
  return ok ? 0 : 1;
}

// The one-block smoother on a large and a small level in turn, as two contexts' solves
// (or two levels of one) call it: neither takes the other's shared memory away.
static int smoother_levels() {
  int bad = 0;
  for (int n : {4, 8, 4, 8}) {
    nc::LevelDev d = {};
    d.nx = d.ny = d.nz = n;
    d.E = (long long)n * n * n;
    d.Nn = (long long)(n + 1) * (n + 1) * (n + 1);
    for (bool tr : {false, true}) {
      const long before = fake::launches;
      const bool took = nc::smooth_block(d, nc::ElemConst<float>{}, nc::LevelBuf<float>{}, tr, 6, true, nullptr, nullptr);
      bad += report(("smooth_block " + std::to_string(n)).c_str(),
                    took && fake::launches == before + 1 && cudaGetLastError() == cudaSuccess);
    }
  }
  return bad;
}

// A context on a small grid of the stand-in's memory.
static nc_ctx* context(int n) {
  nc_params p = {};
  p.nx = p.ny = p.nz = n;
  p.h = 1.0 / n;
  p.Gr = 1e3;
  p.Pr = 0.71;
  p.alpha_max = 1e4;
  p.q_alpha = p.q_f = 1.0;
  p.Ck = 0.1;
  p.g_dir[2] = -1.0;
  nc_bcs b = {};
  b.p_pin = -1;
  nc_ctx* ctx = nullptr;
  if (nc_setup(&p, &b, &ctx) != NC_OK) std::exit(3);
  return ctx;
}

// The calls whose host loop waits for the device: launches that the runtime refuses end
// them with an error.
static int device_loops() {
  int bad = 0;
  for (int n : {2, 5}) {
    nc_ctx* ctx = context(n);
    const long long E = (long long)n * n * n;
    std::vector<double> v[8];
    for (auto& q : v) q.assign(E, 0.5);
    fake::refuse = true;
    bad += report("nc_filter", nc_filter(ctx, v[0].data(), v[1].data(), 2.5 / n, nullptr) == NC_ERR_CUDA);
    bad += report("nc_mma_update",
                  nc_mma_update(ctx, E, 0, v[0].data(), v[1].data(), v[2].data(), v[3].data(), v[4].data(),
                                v[5].data(), 0.1, v[6].data(), nullptr, nullptr, nullptr, nullptr,
                                nullptr) == NC_ERR_CUDA);
    double g;
    bad += report("nc_volume", nc_volume(ctx, E, v[0].data(), nullptr, 0.05, &g, v[1].data(), nullptr) == NC_ERR_CUDA);
    bad += report("no error is left", cudaGetLastError() == cudaSuccess);
    fake::refuse = false;
    nc_destroy(ctx);
  }
  return bad;
}

// A count that overlapping reductions (calls on two streams) left in a context's ticket is gone
// with the next call, on whichever stream.
static int tickets() {
  int bad = 0;
  nc_ctx* ctx = context(4);
  const cudaStream_t first = (cudaStream_t)16, second = (cudaStream_t)32;
  unsigned* const ticket = nc::red_ticket(ctx->partial);
  const long long n = 5LL * 125, E = 64;
  std::vector<double> x(n, 0.0), g(E, 0.5), r(n, 0.0), l(n, 0.0);
  double h[3];
  nc_solve_info info;
  nc_arnoldi_orth(ctx, n, 1, r.data(), n, l.data(), h, NC_FP64, first);
  auto call = [&](const char* what, auto f) {
    for (cudaStream_t s : {second, second, first}) {
      *ticket = 7;
      f(s);
      bad += report(what, *ticket == 0);
    }
  };
  call("nc_arnoldi_orth", [&](cudaStream_t s) { nc_arnoldi_orth(ctx, n, 1, r.data(), n, l.data(), h, NC_FP64, s); });
  call("nc_objective", [&](cudaStream_t s) { nc_objective(ctx, x.data(), h, r.data(), s); });
  call("nc_newton_solve", [&](cudaStream_t s) { nc_newton_solve(ctx, g.data(), x.data(), nullptr, &info, s); });
  call("nc_adjoint_solve", [&](cudaStream_t s) { nc_adjoint_solve(ctx, x.data(), g.data(), r.data(), l.data(), nullptr, &info, s); });
  nc_destroy(ctx);
  return bad;
}

// Calls that read a sum from the device: with every launch refused they end with an error, and
// not with what the memory happened to hold.
static int refused_sums() {
  int bad = 0;
  nc_ctx* ctx = context(4);
  const long long n = 5LL * 125, E = 64;
  std::vector<double> x(n, 0.0), g(E, 0.5), r(n, 0.0), l(n, 0.0);
  double h[3];
  nc_solve_info info;
  fake::refuse = true;
  bad += report("nc_arnoldi_orth", nc_arnoldi_orth(ctx, n, 1, r.data(), n, l.data(), h, NC_FP64, nullptr) == NC_ERR_CUDA);
  bad += report("nc_objective", nc_objective(ctx, x.data(), h, r.data(), nullptr) == NC_ERR_CUDA);
  bad += report("nc_newton_solve",
                nc_newton_solve(ctx, g.data(), x.data(), nullptr, &info, nullptr) == NC_ERR_CUDA &&
                    info.status == NC_ERR_CUDA);
  bad += report("nc_adjoint_solve",
                nc_adjoint_solve(ctx, x.data(), g.data(), r.data(), l.data(), nullptr, &info, nullptr) == NC_ERR_CUDA);
  fake::refuse = false;
  nc_destroy(ctx);
  return bad;
}

// The marching plan of a grid: the cheapest of all run lengths by its rule (a plain search), sums
// that fit the element scratch, and every face row covered.
static int plans() {
  int bad = 0;
  auto up = [](long long a, long long b) { return (a + b - 1) / b; };
  auto check = [&](int nx, int ny, int nz, bool fp64) {
    nc::LevelDev d = {};
    d.nx = nx;
    d.ny = ny;
    d.nz = nz;
    d.E = (long long)nx * ny * nz;
    d.Nn = (nx + 1LL) * (ny + 1) * (nz + 1);
    const nc::MarchPlan p = nc::march_plan(d, fp64);
    const long long stride = 32 % (nx + 1) == 0 ? 32 : 31, faces = (nx + 1LL) * nz, slots = fp64 ? 608 : 8 * 152;
    const double extra = fp64 ? 0.05 : 0.6;
    auto steps = [&](int rc, long long warps) {
      const long long turns = up(warps, slots);
      return (rc + extra) * (fp64 && turns == 1 ? 1.12 : (double)turns);
    };
    int rc = 1;
    double cost = steps(1, up(faces * ny, stride));
    for (int r = 2; r <= 24 && r <= ny; ++r) {
      const long long warps = up(faces, stride) * up(ny, r);
      if (steps(r, warps) < cost && warps * (r + 1) * 320 <= nc::scratch_len(d.E)) {
        rc = r;
        cost = steps(r, warps);
      }
    }
    const bool ok = p.rc == rc && p.stride == stride && p.flat == (rc == 1) && p.runs == up(ny, rc) &&
                    p.nchunk == up(p.flat ? faces * ny : faces, stride) && p.scratch() <= nc::scratch_len(d.E);
    if (!ok) bad += report((std::to_string(nx) + "x" + std::to_string(ny) + "x" + std::to_string(nz)).c_str(), false);
  };
  for (bool fp64 : {false, true}) {
    for (int nx = 1; nx <= 34; ++nx)
      for (int ny = 1; ny <= 30; ++ny)
        for (int nz = 1; nz <= 12; ++nz) check(nx, ny, nz, fp64);
    unsigned s = 12345;
    auto next = [&](int hi) { return 1 + (int)((s = s * 1664525u + 1013904223u) >> 8) % hi; };
    for (int t = 0; t < 20000; ++t) {
      check(next(400), next(400), next(400), fp64);
      check(next(6), next(40), next(200000), fp64);
      check(next(300000), next(6), next(6), fp64);
    }
  }
  return bad;
}

int main(int argc, char** argv) {
  const std::string check = argc > 1 ? argv[1] : "";
  if (check == "smoother_levels") return smoother_levels();
  if (check == "device_loops") return device_loops();
  if (check == "tickets") return tickets();
  if (check == "refused_sums") return refused_sums();
  if (check == "plans") return plans();
  std::printf("unknown check\n");
  return 2;
}
