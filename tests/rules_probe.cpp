// C entries around the dispatch rules of hz_rules.h, for test_dispatch_rules.py.
#include "hz_rules.h"

using namespace hz::rules;

extern "C" int same_tuning(int n, int batch, int up, int finest, int fp32, double bA, double bB, double bA2, double bB2) {
  return tune_key(n, batch, up, finest, fp32, bA, bB) == tune_key(n, batch, up, finest, fp32, bA2, bB2);
}
extern "C" int same_shape(int n, int n2, int batch, int batch2) {
  return tune_key(n, batch, false, false, true, 0, 0) == tune_key(n2, batch2, false, false, true, 0, 0);
}
extern "C" int pass_cfg(int n, int nu, int batch, int sms) { return pass_config(n, nu, batch, sms); }
extern "C" int fills_gpu(long long nodes, int batch) { return operator_fills_gpu(nodes, batch); }
extern "C" int ragged_batch(int n, int batch, int sms) { return batch_takes_cluster(n, batch, sms); }
