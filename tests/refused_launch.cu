// Linked into a copy of the library: cooperative launches are refused while a switch is on, nothing is enqueued.
#include <cuda_runtime.h>

extern "C" {
int refuse_cooperative = 0;
cudaError_t __real_cudaLaunchKernelExC(const cudaLaunchConfig_t* config, const void* fn, void** args);
cudaError_t __wrap_cudaLaunchKernelExC(const cudaLaunchConfig_t* config, const void* fn, void** args) {
  for (unsigned i = 0; refuse_cooperative && i < config->numAttrs; ++i)
    if (config->attrs[i].id == cudaLaunchAttributeCooperative && config->attrs[i].val.cooperative)
      return cudaErrorCooperativeLaunchTooLarge;
  return __real_cudaLaunchKernelExC(config, fn, args);
}
}
