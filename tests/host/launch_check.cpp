// The host side of the library against launches that the runtime refuses (fake_cudart.h).
// usage: launch_check <check>; exit status 0 if it holds.
#include "fake_cudart.h"

#include <cstdio>
#include <string>

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

int main(int argc, char** argv) {
  const std::string check = argc > 1 ? argv[1] : "";
  if (check == "smoother_levels") return smoother_levels();
  std::printf("unknown check\n");
  return 2;
}
