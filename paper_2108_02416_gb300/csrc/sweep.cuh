// One pass over the copies in tiles of 128 coordinates: all pairs of copies
// compared, the chosen copies aggregated (R > 1: R copies per file, in the
// file's rows; R = 1: one row per file, only aggregated).
//
// Lower median, exact (IEEE totalOrder through a monotone uint32 key; the key
// map is a bijection, so the output has the chosen element's bits).  Lane l of
// every warp holds four coordinates of the tile, the warps split the files.
//   sample  24 values per coordinate give the span of 255 value bins
//   sweep   every value's bin is counted (8-bit counters, four coordinates per
//           word, 32 banks) and kept as a tag byte
//   search  the bin that holds the median's rank
//   list    the bin's members (about n / 100), found by their tags, copied
//           into the coordinate's list while the next tile is swept
//   rank    the lists are ranked after it
// What this cannot settle (a NaN, an overflowed counter, a crowded bin, no
// spread in the sample) is left open for fixup_kernel.
//
// More than kTagFiles files leave no room for tags: the sweep then only counts,
// and a second pass over the chosen rows lists the members.  (Sharing a tile
// among the blocks of a cluster, counters and members exchanged through
// distributed shared memory, kept one pass but cost 15 to 25 us per tile: 7.0
// against 6.2 ms at 3,003 files of five copies and d = 2^19.)
#pragma once

#include "aspis_internal.cuh"
#include "median_common.cuh"

namespace aspis {

constexpr int64_t kPairFiles = 516;         // most files whose tag bytes let two blocks share an SM
constexpr int64_t kSettleFiles = 256;       // most files whose few tiles settle their open coordinates themselves
constexpr int64_t kLongFiles = 1200;        // most files whose tag bytes leave a block alone room for long lists
constexpr int64_t kTagFiles = 1330;         // most files whose tag bytes leave a tile room in a block
constexpr int64_t kNarrowFiles = 2700;      // most files whose tag bytes fit 64-coordinate tiles (aggregate.cu)
constexpr int kFewFiles = 36;               // most files whose values one thread sorts in registers (few.cu)
constexpr int kUnclean = 16;                // in a guessed sel: copies of the file differ
// Bits of a coordinate that the sweep leaves to fixup_kernel.  They may also
// be a median's own bits (a NaN payload): computing that one again gives it.
constexpr uint32_t kOpen = 0x7FA5C3E1u;

struct SweepArgs {
    const float *copies;
    int64_t d, ld;
    int f;
    const int8_t *sel;
    aspis_detection *det;
    float *out;
    uint32_t *file_neq;              // R > 1: pair words, ORed
    int r;                           // R = 1: row i * r + sel[i] is file i's
    aspis_detection *gate;           // R = 1: run only where a repair was asked for, or NULL
    const uint8_t *slot_mask;        // averages: the copies averaged per file,
    float *means;                    // and where their averages go, [f][ldm]
    int64_t ldm;
};

// Floats of the widest load that every row start allows.
inline int load_width(const float *copies, int64_t ld)
{
    const uintptr_t p = (uintptr_t)copies;
    return p % 16 == 0 && ld % 4 == 0 ? 4 : p % 8 == 0 && ld % 2 == 0 ? 2 : 1;
}

// ok = false where no layout holds f files; open = fixup_kernel has to follow.
template <int R>
cudaError_t launch_sweep(bool &ok, bool &open, const SweepArgs &A, int mode, bool chained, cudaStream_t stream);

// The median of the averages of the copies in slot_mask, which are also written
// to means (R > 1, aligned rows, f <= kTagFiles); nothing is compared.
template <int R>
cudaError_t launch_sweep_averages(bool &ok, const SweepArgs &A, cudaStream_t stream);

}  // namespace aspis
