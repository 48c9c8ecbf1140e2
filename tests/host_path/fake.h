// Shared by the two halves of the stand-in.
#pragma once
#include <cuda_runtime_api.h>
#include <cstddef>

extern "C" {
struct FakeCounts {
  long captures, instantiated, live_graphs, graph_launches, direct, captured, side_launches, copies, guard_launches, violations;
};
struct FakeCopy { void* dst; const void* src; size_t bytes; };
extern FakeCounts counts;
}
void enqueue(cudaStream_t st);          // work on a stream: part of a capture, or a direct launch
