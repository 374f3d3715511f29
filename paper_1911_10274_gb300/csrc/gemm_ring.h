// gemm_ring.h -- bookkeeping of the staged operand rings of the tensor-core
// products (mlp.cu): which arrivals may still be under way when the loops are
// over.  A CTA may leave only when none is: a copy or a commit that lands later
// would write into shared memory that is no longer its own.
//
// Item j (a k-block, or a tile's accumulator) of a ring of `stages` barriers
// completes phase j / stages of barrier j mod stages.
#pragma once

#include <stdint.h>

namespace titan {

constexpr int ring_slot(int j, int stages) { return j % stages; }
constexpr uint32_t ring_parity(int j, int stages) { return (uint32_t)(j / stages) & 1u; }

// Of n items, the first whose arrival nobody may have waited for yet (an item is
// started only once the one `stages` before it has arrived).
constexpr int ring_tail(int n, int stages) { return n > stages ? n - stages : 0; }

// What the leading CTA of a pair does to its barrier of k-block j, so that the
// phase completes with the copies that really are under way: the leader issued
// its copies of k-blocks 0 .. issued0 - 1 (and with each arrived, expecting the
// bytes of both CTAs), the other CTA those of 0 .. issued1 - 1, `each` bytes a
// CTA.  expect: arrive and expect that many; cancel: that many never come.
struct PairSettle {
    uint32_t expect, cancel;
};
constexpr PairSettle pair_settle(int j, int issued0, int issued1, uint32_t each) {
    return j >= issued0 ? PairSettle{j < issued1 ? each : 0u, 0u} : PairSettle{0u, j < issued1 ? 0u : each};
}

}  // namespace titan
