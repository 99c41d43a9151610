// Shared-memory limits on several devices: a fake runtime counts what it is asked to set on
// the current device.  Prints the calls per device of two "kernels", in three rounds over the
// devices (the second finds device 2 failing once), then the calls of eight threads.
#include <cstdio>
#include <thread>
#include <vector>

#include "qf_internal.h"

static thread_local int current = 0;
static std::atomic<int> calls[2][80];
static std::atomic<bool> failing{false};
static void kernel_a(int) {}
static void kernel_b(int) {}

extern "C" {
cudaError_t cudaGetDevice(int* d) {
  *d = current;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int bytes) {
  if (a != cudaFuncAttributeMaxDynamicSharedMemorySize || bytes != (f == (const void*)kernel_a ? 70000 : 80000))
    return cudaErrorInvalidValue;
  ++calls[f == (const void*)kernel_b][current];
  return failing ? cudaErrorInvalidDevice : cudaSuccess;
}
}

static int use(int dev) {
  current = dev;
  return (qf::smem_limit<kernel_a>(70000) != cudaSuccess) + 2 * (qf::smem_limit<kernel_b>(80000) != cudaSuccess);
}

int main() {
  int bad = use(0) | use(1) | use(0) | use(1);
  failing = true;
  std::printf("%d ", use(2));  // 3: reported, and tried again
  failing = false;
  bad |= use(2) | use(2) | use(63) | use(63) | use(70) | use(70);
  std::printf("%d", bad);
  for (int d : {0, 1, 2, 63, 70}) std::printf(" %d,%d", calls[0][d].load(), calls[1][d].load());
  std::vector<std::thread> t;
  std::atomic<int> failed{0};
  for (int i = 0; i < 8; ++i)
    t.emplace_back([&, i] {
      for (int d = 3; d < 60; ++d) failed += use((d + i) % 57 + 3);
    });
  for (auto& th : t) th.join();
  int missing = 0;
  for (int d = 3; d < 60; ++d) missing += !calls[0][d] + !calls[1][d];
  std::printf(" %d %d\n", failed.load(), missing);
  return 0;
}
