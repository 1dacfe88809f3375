// Host check of which memory sea_set_orbitals' kernels read where it lies.
// Prints "ok" and exits 0, or prints the first mismatch and exits 1.
#include <cstdio>

#include "../../paper_2208_06097_gb300/csrc/sea_internal.cuh"

int main() {
  const struct {
    cudaMemoryType type;
    int device;
    bool in_place;
  } cases[] = {
      {cudaMemoryTypeDevice, 1, true},       // the context's device
      {cudaMemoryTypeDevice, 0, false},      // another one, perhaps without peer access
      {cudaMemoryTypeHost, 1, false},        // page-locked
      {cudaMemoryTypeUnregistered, 1, false},
      {cudaMemoryTypeManaged, 1, false},
  };
  for (const auto& t : cases) {
    cudaPointerAttributes a{};
    a.type = t.type;
    a.device = t.device;
    if (sea_reads_in_place(a, 1) != t.in_place) {
      printf("type %d device %d\n", (int)t.type, t.device);
      return 1;
    }
  }
  printf("ok\n");
  return 0;
}
