// sf_host_device.h - functions that the kernels and the host tests both compile.
#pragma once

#ifdef __CUDACC__
#define SF_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define SF_HOST_DEVICE inline
#endif
