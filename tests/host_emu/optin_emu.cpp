// Host run of csrc/optin.cuh (tests/test_smem_optin_host.py) against a fake runtime of three
// devices that keeps each kernel's dynamic shared-memory limit per device.
#include <cstdio>
#include <map>
#include <utility>

#include "optin.cuh"

static int device = 0, calls = 0;
static cudaError_t next_error = cudaSuccess;
static std::map<std::pair<const void*, int>, int> limit;
cudaError_t cudaGetDevice(int* d) {
  *d = device;
  return cudaSuccess;
}
cudaError_t fake_set_attribute(const void* f, int attr, int value) {
  ++calls;
  if (attr != cudaFuncAttributeMaxDynamicSharedMemorySize) return 1;
  if (next_error != cudaSuccess) return next_error;
  limit[{f, device}] = value;
  return cudaSuccess;
}

static void kernel_a(int) {}
template <int N>
static void kernel_b(double*) {}

#define CHECK(c)                              \
  do {                                        \
    if (!(c)) {                               \
      std::printf("line %d: %s\n", __LINE__, #c); \
      return 1;                               \
    }                                         \
  } while (0)

int main() {
  using mlmc::allow_dynamic_smem;
  for (device = 0; device < 3; ++device) {  // each device's own limit, for each kernel
    CHECK(allow_dynamic_smem<kernel_a>(100000) == cudaSuccess);
    CHECK(allow_dynamic_smem<kernel_b<3>>(200000) == cudaSuccess);
    CHECK((limit[{(const void*)kernel_a, device}] == 100000));
    CHECK((limit[{(const void*)kernel_b<3>, device}] == 200000));
  }
  const int before = calls;
  for (device = 0; device < 3; ++device) CHECK(allow_dynamic_smem<kernel_a>(100000) == cudaSuccess);
  CHECK(calls == before);  // known: no further runtime call
  // a failure is reported on every call, and the limit is raised once the runtime takes it
  device = 1;
  next_error = 2;
  for (int i = 0; i < 3; ++i) CHECK(allow_dynamic_smem<kernel_b<5>>(70000) == 2);
  next_error = cudaSuccess;
  CHECK(allow_dynamic_smem<kernel_b<5>>(70000) == cudaSuccess);
  CHECK((limit[{(const void*)kernel_b<5>, 1}] == 70000));
  device = 200;  // beyond the table: raised on every call
  CHECK(allow_dynamic_smem<kernel_a>(100000) == cudaSuccess);
  CHECK((limit[{(const void*)kernel_a, 200}] == 100000));
  return 0;
}
