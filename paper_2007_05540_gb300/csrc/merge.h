// Batched launches of the tensor-core GEMMs (tc_gemm.cu): which batch entries share a tile.  Host and device, no
// CUDA calls.
#pragma once

#include <algorithm>

namespace heff {

// Merged items of a batched launch: the batch entries of one task that share a tile, entry e in
// slot e.  Merge classes of a task:
//   0     one entry per item
//   1-3   GEMM 1: 2, 4 or 8 entries side by side in slots of 128, 64 or 32 columns (the tile's
//         n fits);  GEMM 2: 2 or 4 entries in slots of 64 or 32 rows (its m fits)
//   4, 5  GEMM 1, tiles of at most 64 x 64: 2 or 4 entries in slots of 64 or 32 rows of the
//         transposed tile (A: the vectors, B: the LW rows).  A tile of few LW rows otherwise leaves
//         all its epilogue to the two warps of its tensor-memory lanes
// A launch may merge fewer entries than a class allows (its shift is lowered, its slots widen).
constexpr int MERGE_CLASSES = 6;
struct Merge {
    long item0[MERGE_CLASSES + 1];       // first item of each class
    int task0[MERGE_CLASSES];            // first task
    int shift[MERGE_CLASSES];            // log2 of the entries per item
};

// Items of a merged launch over nb batch entries, at most 2^cap entries each.
inline Merge merge_items(const int* first, int nb, int cap) {
    Merge mg{};
    long items = 0;
    for (int c = 0; c < MERGE_CLASSES; ++c) {
        mg.item0[c] = items;
        mg.task0[c] = first[c];
        mg.shift[c] = std::min(c < 4 ? c : c - 3, cap);
        items += (long)(first[c + 1] - first[c]) * ((nb + (1 << mg.shift[c]) - 1) >> mg.shift[c]);
    }
    mg.item0[MERGE_CLASSES] = items;
    return mg;
}

// log2 of the most entries per item of a batched launch (0: not merged).  A merged item does the work of up
// to 2^class items in the time of about one (electron problem, m = 1000, blocks of 10-120, 16
// vectors: GEMM 1 170k items of 1.0 us), so as many entries are merged as leave every SM two items.  Where that takes
// less than a tenth of the items away (blocks too wide to share a tile) the launch is left to the tile variant
// that the plan has chosen.
inline int merge_cap(const int* first, int nb, int num_sms) {
    if (nb < 2) return 0;
    const long alone = merge_items(first, nb, 0).item0[MERGE_CLASSES];
    for (int cap = 3; cap >= 1; --cap) {
        const long items = merge_items(first, nb, cap).item0[MERGE_CLASSES];
        if (items >= 2L * num_sms) return 10 * items <= 9 * alone ? cap : 0;
    }
    return 0;
}

}  // namespace heff
