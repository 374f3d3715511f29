// mlp_layout.h -- where the surrogate's parameters lie in their flat array, and
// which of them a block of the gradient kernels forms (mlp.cu).  Host code.  A
// network may have more than 2^32 parameters: offsets, counts and indexes are 64-bit.
#pragma once

#include <stddef.h>
#include <stdint.h>

namespace titan {

// [W1^T (hid x in), b1, W2^T (hid x hid), b2, W3^T, b3, w4 (hid), b4 (1)]
struct MlpLayout {
    size_t w[3] = {0, 0, 0}, n_w[3] = {0, 0, 0};      // first entry and count of W_l^T
    size_t b[3] = {0, 0, 0}, w4 = 0, b4 = 0, total = 0;
};

constexpr MlpLayout mlp_layout(uint32_t in, uint32_t hid) {
    MlpLayout m;
    size_t at = 0;
    for (int l = 0; l < 3; ++l) {
        m.w[l] = at;
        m.n_w[l] = (size_t)hid * (l == 0 ? in : hid);
        at += m.n_w[l];
        m.b[l] = at;
        at += hid;
    }
    m.w4 = at;
    m.b4 = at + hid;
    m.total = m.b4 + 1;
    return m;
}

// The weights of a layer are formed 1,024 to a block, four to a thread.
constexpr uint32_t kGradBlock = 1024;
constexpr uint32_t grad_blocks(size_t n_w) { return (uint32_t)(n_w / kGradBlock); }       // n_w: a multiple of 128 x 128
constexpr size_t grad_index(uint32_t block, uint32_t thread) { return (size_t)kGradBlock * block + 4 * thread; }

}  // namespace titan
