// Rules of the dispatch that are functions of sizes and options alone (host only, no CUDA): each says how
// a level or a launch runs. Every choice gives the same bits.
#pragma once

#include <tuple>

namespace hz {
namespace rules {

// Key under which the tile autotuner keeps its choice for a fused pass. The FP64 passes run other code
// for each operator kind (real or complex diagonals: 29 or 49 FP64 instructions a node), so a choice
// timed for one kind is not the other's; the FP32 code does not depend on it. bA, bB: the shifts of the
// relaxation and of the residual (the pass on the way up has no residual).
using TuneKey = std::tuple<int, int, bool, bool, bool, bool, bool>;
inline TuneKey tune_key(int n, int batch, bool up, bool finest, bool fp32, double bA, double bB) {
  const bool relax_l = !fp32 && bA == 0.0, resid_l = !fp32 && !up && bB == 0.0;
  return TuneKey(n, batch, up, finest, fp32, relax_l, resid_l);
}

}  // namespace rules
}  // namespace hz
