// The queue that the replaced runtime (fake_cuda.cpp) keeps for all streams.
#pragma once

#include <cuda_runtime_api.h>

#include <functional>

using Op = std::function<void()>;
void fake_push(cudaStream_t s, Op op);
