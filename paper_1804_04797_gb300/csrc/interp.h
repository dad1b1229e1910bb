// Lowering of a packed plan (layout 0) to the interpreting kernels' programs.
#pragma once

#include <cstdint>
#include <vector>

#include "interp_dev.h"
#include "plan.h"

namespace svp {

struct InterpProgram {
  std::vector<unsigned char> blocks;  // one block per pass (IHead, stages, steps, gates), 16-byte aligned
  std::vector<uint64_t> offset;       // of each pass's block (a batch's blocks can pass 4 GiB)
  std::vector<uint32_t> bytes;        // its size
};

// Appends the plan's passes to *out (offsets relative to out->blocks).  Returns false for a
// plan that is not in the interpreter's form, or a pass whose block takes 4 GiB or more.
bool lower_interp(const Plan &plan, InterpProgram *out);

}  // namespace svp
