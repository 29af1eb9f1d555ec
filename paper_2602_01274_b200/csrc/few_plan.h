// Which variant of the few-row kernel a forward takes: plain functions of the sizes.
#pragma once
#include <initializer_list>

constexpr int FEW_SHORT = 16, FEW_LONG = 24, FEW_LONGER = 26;     // 8-row weight atoms of a pass at most, up to eight live rows

// Passes of the block with the most weight rows, dealt out in units of 16 (gate/up) or 2 rows (these may begin inside an atom).
static inline int few_passes(int rows, int unit, int ncta, int atoms) {
    const int most = ((rows + unit - 1) / unit + ncta - 1) / ncta * unit, span = unit == 16 ? most / 8 : (most + 13) / 8;
    return (span + atoms - 1) / atoms;
}

// Atoms of a pass for a forward of these layers (vocab: 0 without LM head).  An additional pass costs 2 to 4 us (its activations
// travel again, its sums meet on their own), but the accumulators of long passes leave the kernel short of registers (16 atoms:
// none spilled, 24: 52 to 84 bytes, 26: 76 to 160), which costs up to 1 us a layer.  So the next longer pass is taken where it saves
// more than one pass for three layers.  Measured (us), 16 / 24 or 26 atoms: drafts of width 4096 and FFN 11 008 (19 atoms, four layers,
// a step of two blocks) 3338 / 3187, 3072 / 8192 (14) 2206 / 2223, 768 / 3072 662 / 678; one row of a target of width 4096 386 / 371,
// 5120 / 27 648 (48, three layers) 787 / 735, 768 / 3072 123.0 / 125.6; 1536 / 8960 with four layers and 151 936 tokens (16; the LM head
// 9 passes or 6) 251.5 / 248.4.  24 / 26 atoms: 8192 / 28 672 (50) 941 / 887, 4096 / 11 008 371.8 / 372.8.  (28 atoms: 130 to 220 bytes
// spilled, 4096 / 11 008 383, 5120 / 27 648 748.)
static inline int few_pass_atoms(int n_layers, int qkv_rows, int gate_up_rows, int vocab, int ncta) {
    auto passes = [&](int atoms) {
        return n_layers * (few_passes(qkv_rows, 2, ncta, atoms) + few_passes(gate_up_rows, 16, ncta, atoms)) + (vocab ? few_passes(vocab, 2, ncta, atoms) : 0);
    };
    int pass = FEW_SHORT;
    for (int next : {FEW_LONG, FEW_LONGER})
        if (3 * (passes(pass) - passes(next)) > n_layers) pass = next;
    return pass;
}
