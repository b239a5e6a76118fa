// Host tile planner of the ESP solver (internal).
#pragma once

#include <cstdint>
#include <vector>

#include "esp_common.h"
#include "esp_packed.h"

namespace esp {

struct Plan {
    std::vector<TileDesc> tiles;
    std::vector<int32_t> warp_begin;  // n_warps + 1
    int32_t n_warps = 0;
    int32_t tile_opt = 0;
};

// Splits the jobs of a CSR table (offsets job_off[0 .. S*J]) into at most max_warps contiguous
// warp ranges of about equal option counts (cut at job boundaries), and each range into tiles of
// whole jobs of one scenario with at most tile_opt options; a job with more than tile_opt options
// becomes consecutive chunks of one warp. scen (optional) gives each job's scenario (default j / J);
// runk (optional) gives each job the option count of its run in the sorted layout (0: not in a
// run): tiles never mix runs, and a tile of a run carries tile_run_flags(k). Returns false on
// inconsistent offsets.
bool plan_tiles(const int64_t *job_off, int32_t S, int32_t J, int32_t tile_opt, int32_t max_warps, Plan &out,
                const int32_t *scen = nullptr, const int32_t *runk = nullptr);

// Checks a plan against the table: every job covered exactly once and in order, chunks complete,
// every tile inside the table and inside one scenario (and one run). Returns false on the first
// violation.
bool check_plan(const int64_t *job_off, int32_t S, int32_t J, const Plan &p, const int32_t *scen = nullptr,
                const int32_t *runk = nullptr);

// Sorted layout of a general table (jobs of varying size, no group column), built at load time so
// that most jobs are evaluated as runs of equal size. Per scenario: the jobs of 3 .. kRunMaxK
// options, each padded with never-chosen options to a multiple of 4 and ordered by padded size
// (original order within a size); this part comes first for every scenario, so every run starts on
// a 4-option boundary. Then, per scenario, the jobs of more than kRunMaxK options, then the runs
// of 2-option and of 1-option jobs.
struct SortedLayout {
    std::vector<int64_t> off;    // S*J + 1 padded option offsets in sorted order
    std::vector<int32_t> jmap;   // sorted job -> original global job index
    std::vector<int32_t> scen;   // scenario of each sorted job
    std::vector<int32_t> runk;   // options (padded) of every job of the sorted job's run, 0 for a large job
};

// Returns false when the table is not eligible (more than 2^31 - 1 jobs, or inconsistent offsets).
// run_max_k: the largest padded job of the runs (a multiple of 4; the library uses kRunMaxK).
bool sort_layout(const int64_t *job_off, int32_t S, int32_t J, SortedLayout &out, int32_t run_max_k = kRunMaxK);


// Cost of a step of one- and two-option jobs in the final pass, in tenths of another step's: up to eight winners per
// lane, each with outputs to write and an exact score. (With the round pass's ranges, a few warps held all of them: a
// one-round solve of the heavy-tailed table at 16 scenarios took 1.61 ms, 1.02 with these; 1.43 staged.)
constexpr int64_t kPackFinalTiny = 40;

// Plan of the packed passes over a table (esp_packed.h).
struct PackPlan {
    std::vector<int32_t> job;          // table job of each job in the packed order; empty: the same order
    std::vector<int32_t> job_begin;    // n_tiles + 1: first job (packed order) of each tile
    std::vector<PackTile> tiles;       // by scenario
    std::vector<int32_t> warp_begin;   // n_warps + 1: the round pass's ranges of about equal cost
    std::vector<int32_t> final_begin;  // n_warps + 1: the final pass's
    std::vector<int32_t> scen_tiles;   // S: tiles of each scenario
    int64_t vecs = 0;                  // vectors per plane of the whole copy
    int64_t steps = 0;
    bool narrow = false;               // four options per lane (small tables)
    int32_t n_warps = 0;
};

// Word layout of the unit fields for the largest unit of each column over the table (each below
// 2^23): columns paired so that two fit 32 bits, the widest with the widest that still fits. False when
// the table needs more words than the passes have (kPackMaxWords) or a unit is 2^23 or more. n_groups > 0:
// columns r_global .. R - 1 (one or two) are priced per group and share the last word; the option's group
// slot takes bits that a word leaves free, or a word of its own (3, 4 or 6 words).
bool pack_format(const int32_t *umax, int32_t R, PackFormat &out, int32_t r_global = 0, int32_t n_groups = 0);

// Packed order (per scenario, jobs of the same kind and vector count together), tiles of at most
// kPackTileSteps steps (fewer where the table is small, so that every warp has work; a job of more steps
// is a tile by itself) and ranges for at most max_warps warps. False on inconsistent offsets or a table
// beyond the tile records' 32-bit fields. all_k > 0: every job is known to have that many options.
constexpr int kPackTileSteps = 8;
bool plan_packed(const int64_t *off, int32_t S, int32_t J, int32_t max_warps, PackPlan &out, int64_t all_k = 0);
// Checks a packed plan against the table: every job once, every tile's jobs of its scenario, kind and
// vector count, the tiles' data contiguous, the ranges covering every tile once and in order.
bool check_packed(const int64_t *off, int32_t S, int32_t J, const PackPlan &p, int64_t all_k = 0);

// Slices of the cluster-resident kernel: every scenario's jobs split into cs contiguous runs of about
// equal option counts, run c starting at the first job whose first option lies at least
// floor(c * N_s / cs) options into the scenario (N_s = options of scenario s).
struct ResShape {
    int32_t cs = 0;
    int32_t m_max = 0;                // most jobs in one slice
    int64_t n_max = 0;                // most options in one slice
    std::vector<int32_t> cuts;        // S * (cs + 1) scenario-local job indices
};

// Fills out for cs CTAs per scenario. Returns false on inconsistent offsets.
bool plan_resident(const int64_t *job_off, int32_t S, int32_t J, int32_t cs, ResShape &out);

// One cluster size that fits: its lanes per job, largest slice (jobs, options) and co-resident clusters.
struct ResSize {
    int32_t cs, lanes, m_max, clusters;
    int64_t n_max;
};

// Predicted microseconds of a round of all S scenarios: with clusters of that size (waves of clusters one after
// the other), and streamed (words: unit words of the packed copy, 0: the staged pass).
double resident_round_us(int32_t S, int32_t R, int64_t min_k, int64_t max_k, int32_t sms, const ResSize &o);
double streaming_round_us(int64_t n_opt, int32_t R, int32_t words, int32_t sms);

// The size with the shortest predicted round (-1: none in sizes); ties keep the smaller cluster.
int resident_choice(int32_t S, int32_t R, int64_t min_k, int64_t max_k, int32_t sms, const std::vector<ResSize> &sizes);

}  // namespace esp
