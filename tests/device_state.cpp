// hz_host.h against a fake runtime: two devices with different SM counts, an attribute call that fails once.
#include "hz_host.h"

#include <cstdio>
#include <thread>
#include <vector>

static thread_local int current = 0;
static std::atomic<int> asked{0};

extern "C" cudaError_t cudaGetDevice(int* dev) {
  *dev = current;
  return cudaSuccess;
}
extern "C" cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int dev) {
  ++asked;
  *v = dev == 0 ? 152 : 132 + dev;
  return cudaSuccess;
}

#define CHECK(c) \
  if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); return 1; }

int main() {
  CHECK(hz::device_sms() == 152);
  current = 1;
  CHECK(hz::device_sms() == 133);
  current = 70;  // beyond the table: asked at every call
  CHECK(hz::device_sms() == 202 && hz::device_sms() == 202);
  current = 0;
  const int before = asked;
  CHECK(hz::device_sms() == 152 && asked == before);

  static hz::OncePerDevice once;
  int runs[80] = {};
  bool fail = true;
  auto step = [&] {
    ++runs[current];
    return fail ? cudaErrorInvalidValue : cudaSuccess;
  };
  CHECK(once(step) == cudaErrorInvalidValue);  // a failed step is not taken as done
  fail = false;
  CHECK(once(step) == cudaSuccess && once(step) == cudaSuccess && runs[0] == 2);
  current = 63;
  CHECK(once(step) == cudaSuccess && once(step) == cudaSuccess && runs[63] == 1);
  current = 64;
  CHECK(once(step) == cudaSuccess && once(step) == cudaSuccess && runs[64] == 2);

  // concurrent first calls on two devices: after any of them returns, the step has run on its device
  static hz::OncePerDevice many;
  std::atomic<int> set[2] = {{0}, {0}};
  std::atomic<int> wrong{0};
  std::vector<std::thread> ts;
  for (int t = 0; t < 8; ++t)
    ts.emplace_back([&, t] {
      current = t & 1;
      for (int q = 0; q < 1000; ++q)
        if (many([&] { set[current] = 1; return cudaSuccess; }) != cudaSuccess || !set[current]) ++wrong;
    });
  for (auto& t : ts) t.join();
  CHECK(wrong == 0);
  return 0;
}
