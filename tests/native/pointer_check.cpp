// Host-side check of kernel_can_address (paper_2312_13094_gb300/csrc/fd_runtime.h),
// built with g++ by tests/test_pointer_rule_host.py.  Prints one line per case:
// memory type, owner, device, answer.
#include <cstdio>

#include "fd_runtime.h"

int main() {
  for (int type : {int(cudaMemoryTypeUnregistered), int(cudaMemoryTypeHost),
                   int(cudaMemoryTypeDevice), int(cudaMemoryTypeManaged)})
    for (int owner : {-2, 0, 1})
      for (int device : {0, 1})
        printf("%d %d %d %d\n", type, owner, device,
               fd::kernel_can_address(cudaMemoryType(type), owner, device) ? 1 : 0);
  return 0;
}
