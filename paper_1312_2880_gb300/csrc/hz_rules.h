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

// Geometry of the whole passes of an FP32 Kaczmarz level (hz_kpass.cu): tiles of 13 nodes for four sweeps a
// launch, of 37 or of 62 for two. The one with the least expected time of a level's four launches or launch
// pairs in an iteration: a block fills an SM, so a launch takes a wave of blocks' time per `sms` blocks.
// Measured per iteration (us, geometries 0, 1, 2): n_l = 128 93, 101, 143; n_l = 192 119, 103, 155;
// n_l = 256 178, 105, 156; n_l = 512 565, 171, 156; n_l = 1024 2114, 416, 292, i.e. about 58 + 35, 32 + 72
// and 20 + 136 per wave; 16 right-hand sides on n_l = 144 and 288 (whole iteration) 1243, 566, 583 and
// 4165, 1503, 1320. From four waves of the largest tiles on, the halo decides and not the waves, many of
// whose blocks lie mostly outside the square: 64 and 152 right-hand sides on n_l = 128 (six iterations)
// 9.08 and 19.65 ms with 37-node tiles, which the expected times prefer, 7.89 and 16.72 ms with 62.
constexpr int PASS_EDGE[3] = {13, 37, 62};
inline long long pass_blocks(int cfg, int n, int batch) {
  const long long t = (n + PASS_EDGE[cfg]) / PASS_EDGE[cfg];
  return t * t * batch;
}
inline int pass_config(int n, int nu, int batch, int sms) {
  const double fixed[3] = {58, 32, 20}, wave[3] = {35, 72, 136};
  if (pass_blocks(2, n, batch) > 3ll * sms) return 2;
  int best = 1;
  double cost = 0;
  for (int q = nu % 4 == 0 ? 0 : 1; q < 3; ++q) {
    const double c = fixed[q] + wave[q] * (double)((pass_blocks(q, n, batch) + sms - 1) / sms);
    if (cost == 0 || c < cost) {
      best = q;
      cost = c;
    }
  }
  return best;
}

}  // namespace rules
}  // namespace hz
