// What a test driver linked with the library's objects needs beside them.
#pragma once

#include "../paper_2605_13987_gb300/csrc/wt_internal.cuh"

#include <cstdio>

namespace wt {
void fail(wt_status c, const std::string& m) { throw Error{c, m}; }
void cuda_check(cudaError_t e, const char* w) {
    if (e != cudaSuccess) fail(WT_ERR_CUDA, std::string(w) + ": " + cudaGetErrorString(e));
}
}  // namespace wt
