// What the replaced runtime (fake_cuda.cpp) keeps: one queue for all streams, and the size of
// each device block (0 for other pointers).
#pragma once

#include <cuda_runtime_api.h>

#include <functional>

using Op = std::function<void()>;
void fake_push(cudaStream_t s, Op op);
size_t fake_size(const void* p);
