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

// How the tiles of an FP32 Kaczmarz level run: 0 .. 2, whole passes with their transfers (hz_kpass.cu) in
// tiles of 13 nodes for four sweeps a launch, of 37 or of 62 for two; 3 and 4, two-sweep launches over tiles
// of 32 or 64 nodes between separate transfers (hz_kaczmarz.cu). Of the first three, the one with the least expected time of a level's four launches or launch
// pairs in an iteration: a block fills an SM, so a launch takes a wave of blocks' time per `sms` blocks.
// Measured per iteration (us, geometries 0, 1, 2): n_l = 128 93, 101, 143; n_l = 192 119, 103, 155;
// n_l = 256 178, 105, 156; n_l = 512 565, 171, 156; n_l = 1024 2114, 416, 292, i.e. about 58 + 35, 32 + 72
// and 20 + 136 per wave; 16 right-hand sides on n_l = 144 and 288 (whole iteration) 1243, 566, 583 and
// 4165, 1503, 1320. From four waves of the largest tiles on, the halo decides and not the waves, many of
// whose blocks lie mostly outside the square: 64 and 152 right-hand sides on n_l = 128 (six iterations)
// 9.08 and 19.65 ms with 37-node tiles, which the expected times prefer, 7.89 and 16.72 ms with 62.
//
// The two-sweep launches act only on what can still reach a tile, a fifth fewer row actions than whole passes
// of the same size, and pay two launches and the transfers' traffic for it. V-cycles whose only Kaczmarz
// level is n_l, in us, whole passes (37 or 62), 32 and 64: n_l = 416 131, 149, 152; 448 153, 149, 154; 512
// 165, 159, 166; 576 178, 194, 181; 704 210, 238, 208; 768 256, 248, 251; 896 291, 307, 280; 1024 324, 362,
// 309; 1536 604, 692, 578; 2048 993, 1139, 929. So 64 from where the 62-node tiles take a second wave, and
// 32 where the 37-node tiles take one and at most two of the 32-node tiles come on an SM (n_l = 544, more
// than two, 177 and 186). Batches keep whole passes below that size: 16 right-hand sides on n_l = 256 and 512 (six iterations)
// 6.55, 7.53, 6.98 and 21.0, 24.1, 21.6 ms.
constexpr int PASS_EDGE[3] = {13, 37, 62};
inline int tile_edge(int cfg) { return cfg == 3 ? 32 : cfg == 4 ? 64 : 0; }
inline long long pass_blocks(int cfg, int n, int batch) {
  const long long t = (n + PASS_EDGE[cfg]) / PASS_EDGE[cfg];
  return t * t * batch;
}
inline int pass_config(int n, int nu, int batch, int sms) {
  const double fixed[3] = {58, 32, 20}, wave[3] = {35, 72, 136};
  if (nu % 4 == 0) {  // the two-sweep launches end in the array they start from
    if (pass_blocks(2, n, 1) > sms) return 4;
    const long long t = (n + 32) / 32;
    if (batch == 1 && pass_blocks(1, n, 1) > sms && t * t <= 2ll * sms) return 3;
  }
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

// FP32 Kaczmarz levels of batches that take clusters before tiles: from two waves of the 62-node tiles on, levels
// whose third tile each way lies mostly outside the square. Tiles and clusters, six iterations with 24, 64
// and 152 right-hand sides: n_l = 120 3.51, 7.16, 14.9 and 3.61, 7.41, 15.5 ms; 128 4.21, 7.93, 16.8 and 3.84, 7.97,
// 16.9; 136 4.70, 9.66, 20.6 and 4.30, 8.84, 18.7; 144 5.03, 10.2, 21.5 and 4.81, 9.72, 20.5; 160 5.47, 11.1, 23.8 and
// 5.15, 11.1, 23.1; 168 5.69, 12.4, 27.2 and 5.35, 12.3, 26.9; 184 6.10, 13.5, 30.2 and 6.37, 14.2, 31.5. With 16
// tiles are the faster way (128 3.04 and 3.16).
inline bool batch_takes_cluster(int n, int batch, int sms) {
  return batch > 1 && n >= 2 * PASS_EDGE[2] && n <= 2 * PASS_EDGE[2] + PASS_EDGE[1] && pass_blocks(2, n, batch) > sms;
}

// Coarse tail (hz_tail.cu): the levels that one block runs. In FP64 its pipe makes every level above 16 intervals
// slower than launches over several SMs (iteration at n = 64 193 us with levels 32 .. 8 in the tail, 158 without
// one; n = 512 1104 and 1015; n = 240 848 and 812) while a few instances leave the SMs idle. A batch gives
// every SM a tail of its own and the launches no idle SMs: six iterations with the limit at 16 and at 32 (48),
// n = 64 with a Kaczmarz level of 32, 24, 48, 64 and 152 right-hand sides 3.2, 4.5, 5.4, 10.1 and 4.0, 4.4, 4.7,
// 6.8 ms; n = 96 with one of 24, 24, 48 and 152 3.6, 5.3, 12.9 and 3.7, 4.9, 9.9 ms; and with the limit at 32 and
// 48, n = 72 with one of 36, 56, 64 and 100 4.86, 5.72, 7.72 and 5.04, 5.28, 6.22 ms, n = 88 with one of 44, 64, 80
// and 100 6.63, 7.50, 8.91 and 6.67, 7.18, 7.81 ms.
inline int tail_max_n64(int batch, int sms) { return 4 * batch <= sms ? 16 : 5 * batch <= 2 * sms ? 32 : 48; }
// The most unknowns on the coarsest level: beyond, coarse_solve_kernel over several blocks is the faster way (FP32
// iteration at n = 864, 784 unknowns: 488 us with the tail, 363 without; at 256 212 both ways), but not beside a
// tail on every SM: FP64, without and with the tail, n = 88, 120 and 240 (coarsest 11 and 15), 58 right-hand sides
// 4.90, 6.90, 19.5 and 4.34, 7.06, 19.8 ms, 64 5.41, 7.58, 22.0 and 4.59, 7.39, 21.9, 152 10.8, 16.1, 49.0 and 7.8,
// 12.9, 46.0; FP32 n = 136 and 368 (17 and 23), 64 2.66, 11.1 and 2.68, 11.0 ms, 152 5.35, 24.1 and 5.07, 23.4.
inline int tail_max_coarse(bool fp32, int batch, int sms) { return 5 * batch > 2 * sms ? 1 << 30 : fp32 ? 256 : 100; }

// Operator kernels of the FP64 form (hz_krylov.cu): part of the neighbour sums goes to the integer pipe where
// the launch, all right-hand sides together, fills the GPU: from the nodes of one n = 512 grid on. Smaller
// launches are bound by latency. Measured without and with it (v = A y, t = A z in us): n = 128, 16, 64
// and 152 right-hand sides 23.6, 61.0, 128 -> 21.9, 54.3, 116 and 25.1, 63.2, 138 -> 23.5, 56.3, 126;
// n = 400 17.4 -> 17.5 and 16.9 -> 17.0; n = 2000 alone 91 -> 64.
inline bool operator_fills_gpu(long long nodes, int batch) { return nodes * batch >= 513ll * 513ll; }

}  // namespace rules
}  // namespace hz
