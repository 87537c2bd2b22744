// Test-only C entry point over the library's mixed pair-once block choice for
// systems below 65,536 bodies (paper_2112_15079_gb300/csrc/pair_once_plan.h).
// tests/test_msym_plan.py builds it with g++; no CUDA involved.
#include <cstdint>
#include <vector>

#include "pair_once_plan.h"

extern "C" int ms_block(const int64_t *sizes, int64_t n_sys, int64_t nsm) {
  return nb::msym_small_block(std::vector<int64_t>(sizes, sizes + n_sys), nsm);
}
