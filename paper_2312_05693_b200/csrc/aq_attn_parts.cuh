// How many runs of tiles of B rows an item of the attention products is cut into (host code only).
#pragma once

namespace aq {

// As few runs as give the busiest CTA the fewest tiles. (Whole, the 512 items of 16 tiles that 32 heads of 2048 x 2048 scores have
// are four rounds, 64 tiles, on 148 SMs whose share is 55.4; in halves 56.)
// A call asks every time, so only cuts that can win are tried: the fewest runs of each length, from whole items on, and none once
// an SM has no more than its share. (One by one, in the mean over item counts, against this: 16 tiles 56 / 47 ns, 512 tiles (65536 keys) 1.27 /
// 0.42 us, the most that a call takes, 65535 tiles, 141 / 5.3 us.)
inline int attn_parts(long row_items, int tiles, int sms) {
    const long share = (row_items * tiles + sms - 1) / sms;
    int best = 1;
    long best_tiles = (row_items + sms - 1) / sms * tiles;
    for (int per = tiles; per > 1 && best_tiles > share;) {
        const int p = (tiles + per - 2) / (per - 1);                         // the fewest runs that are shorter than `per`
        if (row_items * p > 0x7FFFFFFFl) break;
        per = (tiles + p - 1) / p;
        const long most = (row_items * p + sms - 1) / sms * per;
        if (most < best_tiles) { best_tiles = most; best = p; }
    }
    return best;
}

}  // namespace aq
