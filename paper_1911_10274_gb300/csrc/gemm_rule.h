// gemm_rule.h -- which kernel of mlp.cu multiplies a shape.  Host code.
#pragma once

#include <stdint.h>

namespace titan {

// Whether C[M, N] = A[M, K] B[N, K]^T is left to persistent CTA pairs (256 x 256 tiles)
// on a device of `sms` SMs.  Pairs run their products faster (a k-block needs less shared
// memory traffic) and hide a tile's epilogue behind the next tile's products - if they get
// a next tile: with one or two each, the one-CTA kernel's smaller tiles fill the device
// better until K is large.  Measured back to back on 152 SMs, one-CTA -> pairs, us, tiles
// of 256 x 256 a pair in parentheses: 2048 x 2560 (1.05) K 64 10.5 -> 14.6, 1024 18.7 ->
// 20.5, 8192 97 -> 80; 2816 x 3072 (1.7) K 512 17.1 -> 17.9, 1024 22.3 -> 20.7, 4096 56 ->
// 46; 3072 x 4096 (2.5) K 64 18.4 -> 20.6, 512 25.0 -> 24.7, 2048 46 -> 38; 4096^2 (3.4) K
// 64 25.1 -> 26.7, 512 34.3 -> 30.9, 4096 102 -> 86; 5120^2 (5.3) K 64 37.2 -> 37.0, 1024
// 64 -> 48; 8192^2 (13.5) K 64 87 -> 74, 8192 818 -> 600.
constexpr bool gemm_takes_pairs(int64_t M, int64_t N, int64_t K, int sms) {
    const int64_t tiles = (M / 256) * (N / 256), pairs = sms / 2;
    return M % 256 == 0 && N % 256 == 0 &&
           (tiles >= 5 * pairs || (K >= 512 && tiles >= 2 * pairs) || (K >= 1024 && 4 * tiles >= 5 * pairs) ||
            (K >= 8192 && tiles >= pairs));
}

// Tile width of the one-CTA kernel (128 rows): 64 columns when 128-wide tiles would not
// fill one wave of 152 SMs; 256 once there are at least two waves of such tiles - but with a
// GELU in the epilogue (gelu), which two CTAs of 128-wide tiles an SM hide better, only from
// K = 4096 on.  128 -> 256 wide, us: forward pass of a hidden layer of 512 at a batch of 32,768
// 161 -> 177, of 2,048 at 16,384 378 -> 384, of 4,096 at 16,384 1,073 -> 1,008, of 8,192 at 4,096
// 995 -> 915.
constexpr int gemm_tile_width(int64_t M, int64_t N, int64_t K, bool gelu) {
    return N % 256 == 0 && (N / 256) * (M / 128) >= 2 * 152 && (!gelu || K >= 4096) ? 256
           : (N / 128) * (M / 128) <= 152                                            ? 64
                                                                                     : 128;
}

}  // namespace titan
