// Host logic of the launches on two devices of one process, without a GPU, on the stand-ins for
// the CUDA runtime of fake_cudart.cpp.  Prints one line per finding; exits 0 without one.
// Argument "no-map": the driver has no tensor maps.
#include <stdio.h>
#include <string.h>

#include <string>
#include <thread>
#include <vector>

#include "dd.h"
#include "dd_kernels.hpp"
#include "fake_cudart.hpp"

// Every launch of the library that takes more than 48 KB of shared memory, and a grid sized by
// the device, on device `dev`.
static void run(int dev) {
  set_device(dev);
  grids().clear();
  auto ok = [&](const char* what, dd_status s) {
    if (s != DD_OK) finding(std::string(what) + " returned " + std::to_string(s));
  };
  const int shapes[2][4] = {{4, 4, 4, 4}, {8, 4, 4, 4}}, dims[4] = {16, 8, 8, 8};
  for (auto& b : shapes) {
    dd_ctx* c = nullptr;
    ok("dd_create", dd_create(&c, dims, b, 1, nullptr));
    const size_t sites = 16 * 8 * 8 * 8;
    std::vector<double> U(sites * 72), f(sites * 24), x(sites * 24);
    ok("dd_load_gauge", dd_load_gauge(c, U.data(), DD_HOST));
    ok("dd_build_clover", dd_build_clover(c, 0.125, 1.0));
    ok("dd_apply_D", dd_apply_D(c, f.data(), x.data(), DD_PREC_FP64, DD_LAYOUT_CANONICAL));
    for (int prec : {DD_PREC_FP32, DD_PREC_FP16, DD_PREC_FP16_H2})
      for (int tps = 1; tps <= 2; ++tps) {
        if (prec == DD_PREC_FP16_H2 && tps == 1) continue;
        const dd_sap_params p = {1, 1, prec, tps, 0};
        ok("dd_sap_precondition",
           dd_sap_precondition(c, (const float*)f.data(), (float*)x.data(), &p, DD_LAYOUT_INTERNAL));
      }
    const dd_sap_params p = {1, 1, DD_PREC_FP16, 0, 0};
    const float* in = (const float*)f.data();
    float* out = (float*)x.data();
    ok("dd_sap_precondition_lattices", dd_sap_precondition_lattices(&c, &in, &out, 1, 1, &p));
    ok("dd_destroy", dd_destroy(c));
  }
  // the restart's dense step with its workspace in shared memory
  std::vector<double> h(2 * 64 * 64), y(2 * 64 * 64);
  double ms;
  ok("dd_deflate_device", dd_deflate_device(40, 8, h.data(), h.data(), h.data(), y.data(), y.data(), y.data(), y.data(), &ms));
  // the fused Gram-Schmidt pass in each of its forms, and the two passes that replace it
  const long long n4 = 6 * 24 * 24 * 24 * 48;
  const int most = 4 * multiprocessors(dev);
  dd::GsTail tail;
  for (int nv : {1, 8, 16, 32, 63}) {
    grids().clear();
    const int rows = dd::launch_gs_project_dot(nullptr, nullptr, nullptr, nv, n4, nullptr, nullptr, nullptr, nullptr,
                                               dd::GsWait{nullptr}, nullptr, tail);
    const int groups = nv <= 15 ? 4 : nv <= 31 ? 3 : nv <= 51 ? 2 : 1;
    const std::vector<unsigned> two = {(unsigned)most, (unsigned)(most * ((nv + 7) / 8))}, one = {(unsigned)multiprocessors(dev)};
    if (rows != (tensor_maps() ? multiprocessors(dev) * groups : most) || grids() != (tensor_maps() ? one : two) || cudaGetLastError())
      finding("projection of " + std::to_string(nv) + " vectors: " + std::to_string(rows) + " rows, " +
              std::to_string(grids().size()) + " launches");
  }
  if (dd::blas_partials_blocks() != most) finding("grid of the vector kernels: " + std::to_string(dd::blas_partials_blocks()));
}

int main(int argc, char** argv) {
  tensor_maps() = !(argc > 1 && !strcmp(argv[1], "no-map"));
  run(0);
  run(1);
  std::thread a(run, 0), b(run, 1);
  a.join();
  b.join();
  return findings() ? 1 : 0;
}
