// Order of a matrix's rows on the device (internal, host code).
#pragma once

#include "mmd_internal.h"

namespace mmd {

// Entries lie far from the diagonal in the order given by iperm.
bool scattered(const HCSR& A, const std::vector<int32_t>& iperm, int threads);
// A's rows, compact pieces of its graph one after the other.
std::vector<int32_t> bisection_order(const HCSR& A, int threads);

}  // namespace mmd
