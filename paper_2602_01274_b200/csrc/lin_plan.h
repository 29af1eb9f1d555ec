// How the stand-alone product is cut, and which of its two kernels takes a shape: plain functions of the sizes.
#pragma once

constexpr int LIN_SMS = 148;
constexpr int LW_ROWS = 32;      // weight rows of a pass of k_linear_wide at most

struct LinPlan {
    int S, groups, NW, TT;
};

// The split with the least weight bytes per block: S = 1 or 2 slices over all SMs (every pair of SMs can hold a
// cluster of two); 4 or 8 only while few clusters are needed (an odd number of SMs per GPC strands some otherwise).  A
// block keeps at least eight chunks of k, and the smaller S wins ties: 17 x 4096 x 11008 (with activations that are not 16-byte
// aligned) runs as 74 clusters of two, 7 tiles each (full 98.9 %), where one slice would leave 4 tiles on some SMs against a mean
// of 3.46.  More than eight tiles a block without slices: slices could even out 5 % at most, and the sums of twice the tiles
// through the cluster cost 1 to 7 us (both measured with k_linear, whichever kernel takes the shape now: 32 x 12210 x 512 16.2 us
// with two slices, 9.5 without; 32 x 11008 x 4096 33.3, 26.9).
static inline LinPlan lin_plan(int N, int K) {
    const int MT = (N + 7) / 8, nch = K / 32;
    LinPlan best{};
    double best_cost = 1e30;
    const int cap[4] = {LIN_SMS, LIN_SMS / 2, 32, 16};
    for (int i = 0; i < 4; ++i) {
        const int S = 1 << i;
        if (S > 1 && (nch / S < 8 || best.NW > 1)) break;           // (NW > 1: more than eight tiles a block without slices)
        const int waves = (MT + cap[i] * 64 - 1) / (cap[i] * 64);   // at most 64 tiles per block
        if (S > 1 && waves > 1) break;
        const int groups = MT < cap[i] * waves ? MT : cap[i] * waves, tiles = (MT + groups - 1) / groups;
        const double cost = (double)waves * tiles / S;
        if (cost < best_cost * 0.97) {
            best_cost = cost;
            best.S = S; best.groups = groups;
            best.NW = 1;
            while ((tiles + best.NW - 1) / best.NW > 8) best.NW *= 2;
            best.TT = (tiles + best.NW - 1) / best.NW;
        }
    }
    return best;
}

// Passes of a k_linear_wide block over its weight rows, and the rows of one, a multiple of two and as even as they come.  Every
// block has the same number of passes (blocks differ by two rows, and no such pair lies on both sides of a multiple of `per`).
struct LinPasses {
    int np, per;
};
static inline LinPasses lin_wide_passes(int N) {
    const int units = (N + 1) / 2, most = (units + LIN_SMS - 1) / LIN_SMS, np = (2 * most + LW_ROWS - 1) / LW_ROWS;
    return LinPasses{np, 2 * ((most + np - 1) / np)};
}

// Whether k_linear_wide takes a shape that k_linear would cut into S slices of k (rows x weight rows x k: us with k_linear / with
// k_linear_wide; graphs of launches on weights that do not fit L2.  Of 9659 measured shapes of up to 14 208 weight rows, 69 are
// 4 to 8 % slower than with the other kernel, 53 are 4 to 12 %; with k_linear_wide for all of them 648 were, by up to 45 %.)
//   - Four and eight slices, and two with fewer than 2048 weight rows, stay with k_linear.  (Two slices, 1409 to 1776 weight rows:
//     k_linear wins at k = 11 008, 17 x 1536 14.4 / 15.2, and loses below, 17 x 1536 x 2048 6.4 / 5.0.  From 2433 weight rows on
//     k_linear_wide wins nearly everywhere: 17 x 2560 x 4096 10.9 / 9.1, 17 x 2560 x 11008 18.7 / 19.0, 17 x 4096 x 11008 24.5 / 21.3;
//     the exception is 17 x 2433 x 11008, 18.2 / 20.4.)
//   - More than three passes of 32 rows stay with k_linear: 17 x 32000 x 1408 24.6 / 26.5.
//   - One pass: always k_linear_wide.
//   - A pass costs about 0.5 us (its sums) and fetches the activations again; what k_linear takes beside the weights grows with
//     token rows x weight rows (its sums).  So with few token rows and a short k the one pass of k_linear is faster: 1 x 13824 x 32
//     3.3 / 4.5, 8 x 5632 x 256 3.7 / 4.0, 17 x 5632 x 640 5.5 / 5.8, 1 x 10240 x 384 4.7 / 5.3, 17 x 10240 x 96 5.1 / 5.7; but
//     32 x 10240 x 32 5.9 / 5.7, 1 x 9472 x 256 4.3 / 4.0 (full passes), 8 x 8192 x 320 4.2 / 4.2.
//   - Two passes of 18 to 24 rows are computed as 32 each, and with 16 and more token rows that bounds a long k: 17 x 5632 x 11008
//     30.7 / 35.6, 32 x 5632 x 4096 15.9 / 16.5, 16 x 5632 x 8192 21.2 / 23.1, 17 x 5120 x 11008 (two slices) 31.8 / 35.6; but
//     17 x 5120 x 4096 16.7 / 15.6, 17 x 8192 x 4096 (two passes of 28) 19.1 / 17.8.
static inline bool lin_wide_takes(int rows, int N, int K, int S) {
    if (S > 2 || (S == 2 && N < 2048) || N > 3 * LW_ROWS * LIN_SMS) return false;
    const LinPasses q = lin_wide_passes(N);
    if (q.np == 1) return true;
    int short_k = 0;                                     // k_linear up to this k
    if (S == 1 && rows <= 24) {
        if (q.per <= 20 || (q.np == 3 && q.per <= 26 && rows <= 8)) short_k = 640;
        else if (q.np == 3 || q.per <= 28) short_k = rows <= 8 ? 288 : 128;
    }
    int long_k = 1 << 30;                                // k_linear from this k on
    if (q.np == 2 && q.per <= 24 && rows > 16 && S == 1) long_k = 4096;
    else if (q.np == 2 && q.per <= 20 && rows >= 16) long_k = 8192;
    return K > short_k && K < long_k;
}
