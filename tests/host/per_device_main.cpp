// PerDevice against a fake of the runtime's current device: every device gets its own call of the
// setter, a failed call is repeated, an error of the query is returned.
#include <cstdio>
#include <thread>
#include <vector>

#include "sp_device.h"

static thread_local int g_dev = 0;
static bool g_fail = false;
extern "C" cudaError_t cudaGetDevice(int* d) {
  *d = g_dev;
  return g_fail ? cudaErrorInitializationError : cudaSuccess;
}

#define CHECK(x) do { if (!(x)) { std::printf("failed: %s\n", #x); return 1; } } while (0)

int main() {
  sp::PerDevice p;
  int calls = 0;
  auto set = [&] { ++calls; return cudaSuccess; };
  CHECK(p.run(set) == cudaSuccess && calls == 1);
  CHECK(p.run(set) == cudaSuccess && calls == 1);
  g_dev = 3;
  CHECK(p.run([] { return cudaErrorInvalidValue; }) == cudaErrorInvalidValue);
  CHECK(p.run(set) == cudaSuccess && calls == 2);
  CHECK(p.run(set) == cudaSuccess && calls == 2);
  g_dev = 0;
  CHECK(p.run(set) == cudaSuccess && calls == 2);
  g_dev = 100;  // beyond the flags: set every time
  CHECK(p.run(set) == cudaSuccess && p.run(set) == cudaSuccess && calls == 4);
  g_fail = true;
  CHECK(p.run(set) == cudaErrorInitializationError && calls == 4);
  g_fail = false;
  sp::PerDevice q;
  std::atomic<int> n{0};
  std::vector<std::thread> th;
  for (int d = 0; d < 8; ++d)
    th.emplace_back([&, d] {
      g_dev = d;
      for (int i = 0; i < 1000; ++i) q.run([&] { ++n; return cudaSuccess; });
    });
  for (auto& t : th) t.join();
  CHECK(n == 8);
  std::printf("ok\n");
  return 0;
}
