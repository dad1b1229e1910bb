// A batch's pass programs past 4 GiB: where the last of them says it lies.
#include <cstdio>
#include <cstring>

#include "batch.h"
#include "interp.h"
#include "plan.h"

int main() {
  svp::Options po;
  po.m = 10;
  po.pack = true;
  po.rk = po.r = 4;
  svp::Plan P;
  const char *err = nullptr;
  std::vector<svp::Gate> g;
  for (uint8_t q = 0; q < 12; ++q) g.push_back(svp::Gate{svp::K_SX, q, 0});
  if (!svp::build_plan(12, g, po, true, &P, &err)) return 2;
  svp::InterpProgram prog;
  const size_t before = 1ull << 32;  // the programs of the circuits before
  prog.blocks.reserve(before + (1u << 20));
  prog.blocks.resize(before);
  if (!svp::lower_interp(P, &prog) || prog.offset.size() != P.passes.size()) return 3;
  size_t at = before;
  for (size_t p = 0; p < prog.offset.size(); ++p) {
    svk::BatchCP cp{};
    cp.block = prog.offset[p];
    svp::IHead h;
    std::memcpy(&h, &prog.blocks[cp.block], sizeof(h));
    if (cp.block != at || h.bytes != prog.bytes[p]) {
      std::printf("pass %zu: block at %llu, not %zu\n", p, (unsigned long long)cp.block, at);
      return 1;
    }
    at += h.bytes;
  }
  return 0;
}
