// Plans of random gate lists in each form of plan, with every stage's register set searched one
// candidate at a time as well (plan.cpp, SV_PLAN_CHECK).
#include <cstdio>
#include <random>
#include <string>

#include "plan.h"

namespace svp {
extern int plan_checks, plan_check_differences;
}

int main(int argc, char **argv) {
  const std::string form = argc > 1 ? argv[1] : "";
  std::mt19937 rng(7);
  auto pick = [&](int below) { return (int)(rng() % (unsigned)below); };
  for (int list = 0; list < 120; ++list) {
    const int n = 12 + pick(list % 4 == 0 ? 23 : 9);
    std::vector<svp::Gate> g;
    const int count = 1 + pick(list % 3 == 0 ? 40 : 500);
    // all kinds, or mostly the phases that wait for the next gate on their qubit
    const std::vector<svp::Kind> kinds =
        list % 2 ? std::vector<svp::Kind>{svp::K_T, svp::K_TDG, svp::K_SX, svp::K_SY, svp::K_CZ}
                 : std::vector<svp::Kind>{svp::K_H, svp::K_T, svp::K_SX, svp::K_SY, svp::K_CZ, svp::K_CZ, svp::K_P0,
                                          svp::K_Z, svp::K_TDG, svp::K_SXDG, svp::K_SYDG, svp::K_PEQ};
    for (int i = 0; i < count; ++i) {
      const svp::Kind k = kinds[(size_t)pick((int)kinds.size())];
      const int a = pick(n), b = (a + 1 + pick(n - 1)) % n;
      g.push_back(svp::Gate{k, (uint8_t)a, (uint8_t)(svp::kind_two_qubit(k) ? b : 0)});
    }
    svp::Options po;
    if (form == "pipelined" || form == "matrix_stages") {  // TMA tiles, phases that wait / post gates
      po.m = form == "pipelined" ? 10 + pick(4) : 12;
      po.pack = true;
      po.layout = 1;
      po.fused = form == "matrix_stages";
      po.rk = po.r = form == "pipelined" ? 4 + pick(2) : 4;
    } else {  // the tensor-core tile kernel's blocks of five or four qubits
      po.fused = true;
      po.rk = po.r = form == "blocks_of_4" ? 4 : 5;
      po.m = form == "blocks_of_4" ? 12 : 12 + pick(2);
    }
    svp::Plan P;
    const char *err = nullptr;
    if (!svp::build_plan(n, g, po, list % 2 == 1, &P, &err)) {
      std::printf("%s\n", err ? err : "no plan");
      return 2;
    }
  }
  std::printf("%d choices, %d differ\n", svp::plan_checks, svp::plan_check_differences);
  return svp::plan_checks < 500 || svp::plan_check_differences != 0;
}
