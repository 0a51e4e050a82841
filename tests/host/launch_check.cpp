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
    bad += report("no error is left", cudaGetLastError() == cudaSuccess);
    fake::refuse = false;
    nc_destroy(ctx);
  }
  return bad;
}

// A count that overlapping reductions left in a context's ticket is gone with the next call.
static int tickets() {
  int bad = 0;
  nc_ctx* ctx = context(4);
  unsigned* const ticket = nc::red_ticket(ctx->partial);
  const long long n = 5LL * 125, E = 64;
  std::vector<double> x(n, 0.0), g(E, 0.5), r(n, 0.0), l(n, 0.0);
  double h[3];
  nc_solve_info info;
  auto call = [&](const char* what, auto f) {
    *ticket = 7;
    f();
    bad += report(what, *ticket == 0);
  };
  call("nc_arnoldi_orth", [&] { nc_arnoldi_orth(ctx, n, 1, r.data(), n, l.data(), h, NC_FP64, nullptr); });
  call("nc_objective", [&] { nc_objective(ctx, x.data(), h, r.data(), nullptr); });
  call("nc_newton_solve", [&] { nc_newton_solve(ctx, g.data(), x.data(), nullptr, &info, nullptr); });
  call("nc_adjoint_solve", [&] { nc_adjoint_solve(ctx, x.data(), g.data(), r.data(), l.data(), nullptr, &info, nullptr); });
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

int main(int argc, char** argv) {
  const std::string check = argc > 1 ? argv[1] : "";
  if (check == "smoother_levels") return smoother_levels();
  if (check == "device_loops") return device_loops();
  if (check == "tickets") return tickets();
  if (check == "refused_sums") return refused_sums();
  std::printf("unknown check\n");
  return 2;
}
