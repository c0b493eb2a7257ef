// The table-lookup draft model of the tree construction kernel (the same integer functions as the oracle's).
#pragma once

#include "common.cuh"

namespace dyspec {

// The row of a child is this modulo the number of rows.
__device__ __forceinline__ uint32_t draft_child_hash(uint32_t parent_row, uint32_t token) {
  return parent_row * 2654435761u + (token + 1u) * 40503u;
}
__device__ __forceinline__ uint32_t draft_uniform_index(uint32_t row, uint32_t attempt, uint32_t n_uniforms) {
  return (row * 7919u + attempt * 104729u + 17u) % n_uniforms;
}

}  // namespace dyspec
