// tile_width.h -- which output tile width (BN of the tensor-core GEMM) a product takes when nothing was tuned.
// The widths change no output bit. Plain C++.
#pragma once

#include <stdint.h>

namespace chemgb {

// Tile widths the library is built with (the autotuner picks among them).
constexpr int kTileWidths[] = {32, 64, 128, 160, 208, 256};
constexpr int kTileRows = 128;

// Fewest padded columns, then the widest tile.
inline int padded_tile_width(int N) {
    int best = 256;
    long best_pad = -1;
    for (int bn : kTileWidths) {
        if (bn < 64 && N > 64) continue;
        const long pad = (long)((N + bn - 1) / bn) * bn - N;
        if (best_pad < 0 || pad < best_pad || (pad == best_pad && bn > best)) { best = bn; best_pad = pad; }
    }
    return best;
}

// For a layer's handle, whose row count is not known: a tile's time is about that of its columns plus 290
// (the operands' k-blocks and the tile's own start and end), so the width with the smallest sum over the N
// tiles. Measured with the GELU epilogue on 262,144 rows of GELU-distributed operands (us at 160 / 208 /
// 256): 800 x 1600 559 / 512 / 532, 1600 x 96 325 / 329 / 293, 400 x 800 193 / 156 / 207, 1024 x 2048 980 / 811 / 772.
inline int default_tile_width(int N) {
    int best = 256;
    long best_cost = -1;
    for (int bn : kTileWidths) {
        const long cost = (long)((N + bn - 1) / bn) * (bn + 290);
        if (best_cost < 0 || cost < best_cost) { best = bn; best_cost = cost; }
    }
    return best;
}

// For one product of M x N x K: of the two widths above, by the tiles that the busiest of `sms` CTAs computes
// times a tile's cost. GELU outputs: columns plus 140. FP32 outputs (linear): the columns it stores, or 0.03 (columns + 200)
// per k-block where the products take longer; the fewest padded columns stay unless the other width gains 14 %.
// Measured over M = 4,096, 20,000 and 126,000, K = 96 to 1,600 and 37 widths N = 32 to 1,600 (us, the fewest
// padded columns / the rule by N alone / this one): linear 4,096 x 1144 x 1144 22.5 / 32.8 / 22.5,
// 126,000 x 640 x 1144 287 / 316 / 287, 126,000 x 704 x 1144 441 / 343 / 343; GELU 4,096 x 1144 x 1144 20.8 / 29.0 /
// 20.8, 126,000 x 704 x 1144 406 / 258 / 258. Over all of them linear products take at most 5 % more than with the
// fewest padded columns (the rule by N alone: up to 62 %), GELU products at most 12 % (40 %).
inline int product_tile_width(int64_t M, int N, int K, bool gelu, int sms) {
    const int pad = padded_tile_width(N), def = default_tile_width(N);
    auto cost = [&](int bn) {
        const int64_t nt = (N + bn - 1) / bn, tiles = (M + kTileRows - 1) / kTileRows * nt;
        const double rounds = (double)((tiles + sms - 1) / sms);
        if (gelu) return rounds * (bn + 140);
        const double products = (K + 63) / 64 * 0.03 * (bn + 200), columns = (double)N / (double)nt;
        return rounds * (products > columns ? products : columns);
    };
    return cost(def) < (gelu ? 1.0 : 0.86) * cost(pad) ? def : pad;
}

}  // namespace chemgb
