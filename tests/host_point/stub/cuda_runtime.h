// The names of the CUDA runtime that nr_internal.h mentions, for host builds of the per-point code.
#pragma once
typedef int cudaError_t;
typedef struct CUstream_st* cudaStream_t;
typedef struct CUgraphExec_st* cudaGraphExec_t;
enum : int { cudaSuccess = 0 };
