// Host-only driver (no GPU needed): reads "type memory_device context_device
// current_device" lines on stdin (type: 0 unregistered, 1 host, 2 device, 3
// managed) and prints 1 where a field's rows go by kernel, 0 by copy.
#include <cstdio>

#include "../../paper_2404_04441_gb300/csrc/common.cuh"

int main() {
  int type, mem, ctx, cur;
  while (std::scanf("%d %d %d %d", &type, &mem, &ctx, &cur) == 4) {
    cudaPointerAttributes at{};
    at.type = static_cast<cudaMemoryType>(type);
    at.device = mem;
    std::printf("%d\n", (int)rows_by_kernel(at, ctx, cur));
  }
  return 0;
}
