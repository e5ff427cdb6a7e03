// What api_harness.cu and api_fakes.cpp share.
#pragma once
#include <cuda_runtime_api.h>

#include <map>
#include <string>
#include <vector>

// A range of host memory that stands for pinned or device memory.
struct Range {
  const char *p;
  size_t n;
  cudaMemoryType type;
  unsigned flags;
};
extern std::vector<Range> ranges;
extern std::map<std::string, int> launched;         // launches by launcher
extern std::map<std::string, cudaError_t> refused;  // the error a launcher returns
cudaError_t launch(const char *name);
