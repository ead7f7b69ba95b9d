// A stream of a part of the current device's SMs (a green context); both live as
// long as the process.
#include <cuda.h>

// Creates it; the number of SMs it has, or 0 if it cannot be had.
extern "C" int green_stream(int sms, void** out) {
  CUdevice dev;
  CUdevResource all, part, rest;
  CUdevResourceDesc desc;
  CUgreenCtx ctx;
  CUstream stream;
  unsigned n = 1;
  if (cuCtxGetDevice(&dev) != CUDA_SUCCESS || cuDeviceGetDevResource(dev, &all, CU_DEV_RESOURCE_TYPE_SM) != CUDA_SUCCESS ||
      cuDevSmResourceSplitByCount(&part, &n, &all, &rest, 0, (unsigned)sms) != CUDA_SUCCESS || n != 1 ||
      cuDevResourceGenerateDesc(&desc, &part, 1) != CUDA_SUCCESS ||
      cuGreenCtxCreate(&ctx, desc, dev, CU_GREEN_CTX_DEFAULT_STREAM) != CUDA_SUCCESS)
    return 0;
  if (cuGreenCtxStreamCreate(&stream, ctx, CU_STREAM_NON_BLOCKING, 0) != CUDA_SUCCESS) {
    cuGreenCtxDestroy(ctx);
    return 0;
  }
  *out = stream;
  return (int)part.sm.smCount;
}
