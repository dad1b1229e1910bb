// Compiles the kernels of one plan with the cubin cache in the directory given.
#include <cuda_runtime.h>

#include <cstdio>

#include "jit.h"
#include "kernels.h"
#include "plan.h"

namespace svk {
int device_sm_count() { return 152; }
}  // namespace svk

int main(int, char **argv) {
  svp::Options po;
  po.m = 12;
  po.pack = true;
  po.rk = po.r = 4;
  po.layout = 1;
  svp::Plan P;
  const char *err = nullptr;
  if (!svp::build_plan(12, {svp::Gate{svp::K_SX, 5, 0}}, po, false, &P, &err)) return 2;
  std::vector<std::string> cubins;
  std::string log;
  if (!svj::compile_plan(P, 4, "sm_103a", &cubins, &log, argv[1])) {
    std::printf("%s\n", log.c_str());
    return 1;
  }
  return 0;
}
