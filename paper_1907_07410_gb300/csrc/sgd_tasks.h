// How many tasks the blocked SGD's epoch order can have. Plain C++, so that
// it can be checked without a GPU.
#pragma once
#include <cstdint>

namespace bsvd {

// An owner has at most one task in each block of its block row or column (a
// batch has one block a matrix). A rating with an id out of range is reported,
// but sorted all the same, as cell (0, 0) of block 0. Where explicit bounds
// leave that block empty on the owner's side no owner has that cell, and such
// ratings are a task more.
inline int64_t sgd_max_tasks(int64_t nnz, bool diag, bool own_items, int64_t p,
                             int64_t q, int64_t m, int64_t n) {
  const int64_t owners = own_items ? n : m;
  const int64_t most = 1 + (diag ? owners : (own_items ? p : q) * owners);
  return nnz < most ? nnz : most;
}

}  // namespace bsvd
