// Host check of SmemOptIn against a fake of the two runtime calls it makes:
// the limit is raised once on every device, and again after a failure.
#include <cuda_runtime.h>

#include <cstdio>
#include <vector>

namespace fake {
int device = 0, error = 0;
std::vector<int> raised;  // the device of each successful call
cudaError_t get_device(int* d) {
  *d = device;
  return cudaSuccess;
}
template <typename K>
cudaError_t set_attribute(K, cudaFuncAttribute, int bytes) {
  if (error) return cudaErrorInvalidValue;
  raised.push_back(bytes == 64 * 1024 ? device : -1);
  return cudaSuccess;
}
}  // namespace fake
#define cudaGetDevice fake::get_device
#define cudaFuncSetAttribute fake::set_attribute
#include "fmm_internal.h"

int main() {
  static fmmgb::SmemOptIn opt;
  void (*kernel)() = nullptr;
  bool ok = true;
  for (int d : {0, 0, 1, 0, 1, 5, 63}) {
    fake::device = d;
    ok &= opt(kernel, 64 * 1024) == cudaSuccess;
  }
  ok &= fake::raised == std::vector<int>({0, 1, 5, 63});
  fake::raised.clear();
  fake::device = 2, fake::error = 1;  // a failure is reported and not recorded
  ok &= opt(kernel, 64 * 1024) == cudaErrorInvalidValue;
  fake::error = 0;
  ok &= opt(kernel, 64 * 1024) == cudaSuccess && fake::raised == std::vector<int>({2});
  fake::device = 64;  // beyond the record: raised on every call
  for (int i = 0; i < 2; ++i) ok &= opt(kernel, 64 * 1024) == cudaSuccess;
  ok &= fake::raised == std::vector<int>({2, 64, 64});
  std::printf("%s\n", ok ? "ok" : "FAILED");
  return ok ? 0 : 1;
}
