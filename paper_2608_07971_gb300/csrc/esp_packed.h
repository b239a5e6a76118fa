// The packed screen copy of an option table (internal): what the fp32 screen of
// the evaluation pass reads, bit for bit, in fewer bytes, and the tiles of the packed passes over it.
//
// Per option: one word -v32 (v truncated to fp32 as the screen takes it, negated; +inf for a load-time
// duplicate or padding, so its screen score is +inf), and nw words of two unit fields each: the low
// field in bits 0 .., the high field in the top bits. A field is exactly as wide as the largest unit of
// its column over the table, so every unit is stored as the whole number it is.
//
// Why: the pass over a table larger than L2 streams it every round, and at 4R + 8 bytes per option it
// ran at 0.91-0.995 of the copy bandwidth. R = 6 columns of the cluster workloads hold 86 unit bits: three
// words, 16 bytes per option with -v32 instead of 32. The fp64 values stay in the table for exact scores
// (the units of which come from the words) and for the final pass.
#pragma once

#include <cstdint>

#include "esp_common.h"

namespace esp {

constexpr int kPackMaxWords = 8;   // unit words of an option; tables that need more keep the staged pass
constexpr uint32_t kPackInf = 0x7f800000u;   // +inf: a duplicate or padding option's -v32

struct PackFormat {
    int32_t nw;                          // unit words (an instantiated count: 2, 3, 4, 6 or 8)
    uint32_t mask[kPackMaxWords];        // low field of word k: w & mask[k]
    int32_t shift[kPackMaxWords];        // high field of word k: w >> shift[k] (9 .. 31)
    // with f = funnelshift_r(w, magic[k], shift[k]): the bits of the float 2^23 + high field
    uint32_t magic[kPackMaxWords];
    int8_t col_lo[kPackMaxWords], col_hi[kPackMaxWords];   // table column of each field, -1: none
    int8_t field[kMaxR];                 // of each column: 2 x its word, + 1 for the high field
    // tables with a group column: the last word holds the columns that are priced per group; word g_word
    // also holds, from bit g_shift on, the option's group slot (pack_slot)
    int32_t g_word, g_shift;
    uint32_t g_mask;                     // 0: no group column
    int32_t g_bytes;                     // a warp's shared memory for the groups' prices (pack_group_bytes)
};

// The slot of group g in the warp's table of group prices: every ninth slot is left out, so that the groups
// 8 apart that neighbouring lanes look up lie in different banks.
ESP_HD uint32_t pack_slot(uint32_t g)
{
    return g + (g >> 3);
}
ESP_HD uint32_t pack_slot_group(uint32_t slot)
{
    return slot - slot / 9;
}

// Grouped tables that the packed passes take: one or two columns priced per group (one word), and at
// most kPackMaxPrices prices (the price table is held per warp; more would cost resident CTAs).
constexpr int kPackMaxPrices = 1024;
ESP_HD bool pack_groups_fit(int R, int r_global, int P)
{
    return R - r_global <= 2 && P <= kPackMaxPrices;
}
// Bytes of that table: two fp32 prices per slot; the price update puts P new prices there.
ESP_HD int pack_group_bytes(int P, int n_groups)
{
    const int a = 8 * ((int)pack_slot((uint32_t)n_groups) + 1), b = 8 * P;
    return ((a > b ? a : b) + 15) & ~15;
}

// Steps. A warp screens up to 256 options at once, eight consecutive options of a job per lane as two
// vectors of four (one 16-byte vector per word plane holds four options' words). A step's data are
// contiguous: nw + 1 planes of V vectors, in a plane first the lanes' first vectors, then their second
// ones, without gaps. Three kinds of tile:
//   jobs   3 .. 256 options per job (m = ceil(k / 4) vectors, ca = ceil(m / 2) lanes of a job's
//          2^code-lane group in use, cb = floor(m / 2) of them with a second vector): 32 >> code jobs per
//          step, V = (32 >> code) m; jobs missing from the tile's last step are padding. Narrow (a small
//          table, so that more warps share it): a lane per vector, ca = m <= 2^code and cb = 0
//   tiny   1 or 2 options per job (code kPackTiny, m = k): 256 / k jobs per step, V = 64; lane l holds
//          the step's vectors l and 32 + l
//   large  over 256 options per job (code kPackLarge): nch = ceil(m / 64) steps per job of
//          V = ceil(m / nch) vectors each
// A tile is consecutive jobs (in the packed order) of one scenario with the same kind and m.
struct alignas(16) PackTile {
    uint32_t base;        // plane vectors before the tile: its data start at vector base * (nw + 1)
    uint32_t scenario;
    uint32_t mk;          // m << 3 | code
    uint32_t n_job;
};
static_assert(sizeof(PackTile) == 16, "PackTile is one 16-byte load");
constexpr uint32_t kPackTiny = 6, kPackLarge = 7;
constexpr int kPackStepVecs = 64;   // vectors of a step's plane at most

// Derived shape of a tile.
struct PackShape {
    int code, m;
    int v;            // vectors per plane of a step
    int ca, cb;       // vectors of a job (large: of a step) that are first / second vectors of a lane
    bool narrow;      // a lane holds four options of a job, not eight
    int per_step;     // jobs per step (large: 1 job every nch steps)
    int nch;          // steps per job (1 unless large)
    int steps;
};

ESP_HD PackShape pack_shape(const PackTile &t)
{
    PackShape s;
    s.code = (int)(t.mk & 7u);
    s.m = (int)(t.mk >> 3);
    s.nch = 1;
    s.narrow = false;
    const int n = (int)t.n_job;
    if (s.code == (int)kPackTiny) {
        s.v = 64;
        s.ca = s.cb = 32;
        s.per_step = 256 / s.m;
        s.steps = (n + s.per_step - 1) / s.per_step;
    } else if (s.code == (int)kPackLarge) {
        s.nch = (s.m + 63) / 64;
        s.v = (s.m + s.nch - 1) / s.nch;
        s.ca = (s.v + 1) / 2;
        s.cb = s.v / 2;
        s.per_step = 1;
        s.steps = n * s.nch;
    } else {
        s.per_step = 32 >> s.code;
        s.v = s.per_step * s.m;
        s.narrow = (1 << s.code) >= s.m;   // eight options per lane need fewer lanes than vectors (m = 1: the same)
        s.ca = s.narrow ? s.m : (s.m + 1) / 2;
        s.cb = s.m - s.ca;
        s.steps = (n + s.per_step - 1) >> (5 - s.code);
    }
    return s;
}

}  // namespace esp
