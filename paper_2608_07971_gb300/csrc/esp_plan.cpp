// Host tile planner: static work split of one evaluation pass over tiles and warps.
#include "esp_plan.h"

#include <algorithm>
#include <climits>
#include <cstdint>

namespace esp {

// Estimated cost of evaluating a tile, in SM cycles of one warp, from clock64 probes of the pass on
// GB300. A tile costs a fixed part (stage wait, copy issue, bookkeeping) plus one warp-wide step per
// "row": 128 options four per lane for uniform runs and chunks of large jobs (a run of jobs with K =
// 4m options gives each job 2^ceil(log2 m) lanes, so 32 / that many jobs share a row), 32 options
// one per lane otherwise; closing a chunked job adds its cross-warp reduction and winner read.
static int64_t tile_rows(const TileDesc &d)
{
    if (d.flags & TILE_BIG)
        return (d.n_opt + 127) / 128;
    if ((d.flags & TILE_RUN) && tile_run_k(d.flags) >= 4) {
        const int m = tile_run_k(d.flags) / 4;
        int lanes = 1;
        while (lanes < m)
            lanes <<= 1;
        const int per_row = 32 / lanes;
        return (d.n_job + per_row - 1) / per_row;
    }
    return (d.n_opt + 31) / 32;
}

static int64_t tile_cost(const TileDesc &d)
{
    return 1050 + 1650 * tile_rows(d) + ((d.flags & TILE_BIG_LAST) ? 850 : 0);
}

bool plan_tiles(const int64_t *off, int32_t S, int32_t J, int32_t tile_opt, int32_t max_warps, Plan &out,
                const int32_t *scen, const int32_t *runk)
{
    out.tiles.clear();
    out.warp_begin.clear();
    out.tile_opt = tile_opt;
    const int64_t n_jobs = (int64_t)S * J;
    if (tile_opt < 32 || (tile_opt & 31) || max_warps < 1)
        return false;
    if (n_jobs == 0) {
        out.n_warps = 0;
        out.warp_begin.push_back(0);
        return true;
    }
    const int64_t total = off[n_jobs];
    if (off[0] != 0 || total < n_jobs)
        return false;
    for (int64_t j = 0; j < n_jobs; ++j)   // every job needs at least one option
        if (off[j + 1] <= off[j])
            return false;

    // 1. tiles in job order: whole jobs of one scenario (and one run) up to tile_opt options, or the
    //    chunks of a job larger than a tile. Without scen, job j belongs to scenario j / J, tracked
    //    incrementally (s_cur, s_end) instead of dividing per job.
    out.tiles.reserve((size_t)std::min<int64_t>(n_jobs, total / std::max(1, tile_opt / 4) + S + 1));
    int32_t s_cur = 0;
    int64_t s_end = J;
    int64_t j = 0;
    while (j < n_jobs) {
        while (!scen && j >= s_end) {
            ++s_cur;
            s_end += J;
        }
        const int32_t s = scen ? scen[j] : s_cur;
        const int64_t K = off[j + 1] - off[j];
        if (K > tile_opt || (runk && runk[j] > kPassRunMaxK)) {
            const int64_t nch = (K + tile_opt - 1) / tile_opt;
            for (int64_t c = 0; c < nch; ++c) {
                TileDesc d;
                d.opt_begin = off[j] + c * tile_opt;
                d.job_begin = j;
                d.n_opt = (int32_t)std::min<int64_t>(tile_opt, K - c * tile_opt);
                d.n_job = (c == 0) ? 1 : 0;
                d.scenario = s;
                d.flags = TILE_BIG | (c == 0 ? TILE_BIG_FIRST : 0u) | (c == nch - 1 ? TILE_BIG_LAST : 0u);
                out.tiles.push_back(d);
            }
            ++j;
            continue;
        }
        const int64_t opt0 = off[j];
        const int32_t rk = runk ? runk[j] : 0;
        int64_t jj = j;
        const int64_t jlim = scen ? n_jobs : std::min<int64_t>(n_jobs, s_end);
        while (jj < jlim && (!scen || scen[jj] == s) && (!runk || runk[jj] == rk) && off[jj + 1] - opt0 <= tile_opt)
            ++jj;
        TileDesc d;
        d.opt_begin = opt0;
        d.job_begin = j;
        d.n_opt = (int32_t)(off[jj] - opt0);
        d.n_job = (int32_t)(jj - j);
        d.scenario = s;
        d.flags = rk > 0 ? tile_run_flags(rk) : 0u;
        out.tiles.push_back(d);
        j = jj;
    }

    // 2. warps: contiguous tile ranges of about equal estimated cost, at least one full tile of work
    //    per warp; a range never starts inside the chunks of a large job (its state is per warp)
    const int64_t n_tiles = (int64_t)out.tiles.size();
    std::vector<int64_t> pre(n_tiles + 1, 0);
    for (int64_t k = 0; k < n_tiles; ++k)
        pre[k + 1] = pre[k] + tile_cost(out.tiles[k]);
    const int64_t full = 1050 + 1650;     // one row
    const int64_t want = (pre[n_tiles] + full - 1) / full;
    const int32_t W = (int32_t)std::min<int64_t>(std::min<int64_t>(max_warps, std::max<int64_t>(1, want)), n_tiles);
    out.warp_begin.assign(W + 1, 0);
    out.warp_begin[W] = (int32_t)n_tiles;
    for (int32_t w = 1; w < W; ++w) {
        const int64_t target = (int64_t)((__int128)pre[n_tiles] * w / W);
        int64_t k = std::lower_bound(pre.begin(), pre.end(), target) - pre.begin();
        if (k > 0 && target - pre[k - 1] < pre[k] - target)   // the nearer tile boundary
            --k;
        if (k < n_tiles && (out.tiles[k].flags & TILE_BIG) && !(out.tiles[k].flags & TILE_BIG_FIRST)) {
            int64_t a = k, b = k;                            // the chunked job's first tile, the next job's
            while (!(out.tiles[a].flags & TILE_BIG_FIRST))
                --a;
            while (b < n_tiles && (out.tiles[b].flags & TILE_BIG) && !(out.tiles[b].flags & TILE_BIG_FIRST))
                ++b;
            k = (target - pre[a] < pre[b] - target) ? a : b;
        }
        k = std::min<int64_t>(std::max<int64_t>(k, out.warp_begin[w - 1]), n_tiles);
        out.warp_begin[w] = (int32_t)k;
    }
    out.n_warps = W;
    return true;
}

bool check_plan(const int64_t *off, int32_t S, int32_t J, const Plan &p, const int32_t *scen,
                const int32_t *runk)
{
    auto scen_of = [&](int64_t j) -> int64_t { return scen ? scen[j] : j / J; };
    const int64_t n_jobs = (int64_t)S * J;
    if ((int32_t)p.warp_begin.size() != p.n_warps + 1)
        return false;
    if (p.warp_begin.front() != 0 || p.warp_begin.back() != (int32_t)p.tiles.size())
        return false;
    for (int32_t w = 0; w < p.n_warps; ++w)
        if (p.warp_begin[w] > p.warp_begin[w + 1])
            return false;
    int64_t next_job = 0;
    int64_t big_next_opt = -1;  // expected opt_begin of the next chunk of an open big job
    for (const TileDesc &d : p.tiles) {
        if (d.n_opt < 1 || d.n_opt > p.tile_opt)
            return false;
        if (d.scenario < 0 || d.scenario >= S)
            return false;
        if (d.flags & TILE_BIG) {
            const int64_t j = d.job_begin;
            if (d.flags & TILE_BIG_FIRST) {
                if (big_next_opt >= 0 || j != next_job || d.opt_begin != off[j] || d.n_job != 1)
                    return false;
            } else if (d.opt_begin != big_next_opt || d.n_job != 0 || j != next_job) {
                return false;
            }
            if (scen_of(j) != d.scenario || d.opt_begin + d.n_opt > off[j + 1])
                return false;
            if (d.flags & TILE_BIG_LAST) {
                if (d.opt_begin + d.n_opt != off[j + 1])
                    return false;
                big_next_opt = -1;
                next_job = j + 1;
            } else {
                if (d.n_opt != p.tile_opt)
                    return false;
                big_next_opt = d.opt_begin + d.n_opt;
            }
        } else {
            if (big_next_opt >= 0 || d.job_begin != next_job || d.n_job < 1)
                return false;
            const int64_t j1 = d.job_begin + d.n_job;
            if (j1 > n_jobs || d.opt_begin != off[d.job_begin] || d.opt_begin + d.n_opt != off[j1])
                return false;
            if (!scen) {   // a contiguous range lies in one scenario iff its ends do
                if (scen_of(d.job_begin) != d.scenario || scen_of(j1 - 1) != d.scenario)
                    return false;
            }
            if (scen || runk) {
                for (int64_t j = d.job_begin; j < j1; ++j) {
                    if (scen && scen[j] != d.scenario)
                        return false;
                    if (d.flags & TILE_RUN) {
                        const int k = tile_run_k(d.flags);
                        if (!runk || runk[j] != k || off[j + 1] - off[j] != k || k > kPassRunMaxK)
                            return false;
                    } else if (runk && runk[j] != 0) {
                        return false;
                    }
                }
            } else if (d.flags & TILE_RUN) {
                return false;
            }
            if ((d.flags & TILE_RUN) && (d.opt_begin & 3) != 0 && tile_run_k(d.flags) >= 4)
                return false;   // a run of 4m-option jobs starts on a 4-option boundary
            next_job = j1;
        }
    }
    return big_next_opt < 0 && next_job == n_jobs;
}

bool plan_resident(const int64_t *off, int32_t S, int32_t J, int32_t cs, ResShape &out)
{
    out.cs = cs;
    out.m_max = 0;
    out.n_max = 0;
    out.cuts.assign((size_t)S * (cs + 1), 0);
    if (cs < 1 || S < 1 || J < 1)
        return false;
    for (int32_t s = 0; s < S; ++s) {
        const int64_t *o = off + (int64_t)s * J;   // o[0 .. J]
        const int64_t N = o[J] - o[0];
        if (N < J)
            return false;
        int32_t *cut = out.cuts.data() + (size_t)s * (cs + 1);
        cut[0] = 0;
        cut[cs] = J;
        for (int32_t c = 1; c < cs; ++c) {
            const int64_t target = o[0] + (int64_t)((__int128)N * c / cs);
            int32_t j = (int32_t)(std::lower_bound(o, o + J, target) - o);
            cut[c] = std::max(j, cut[c - 1]);
        }
        for (int32_t c = 0; c < cs; ++c) {
            out.m_max = std::max(out.m_max, cut[c + 1] - cut[c]);
            out.n_max = std::max<int64_t>(out.n_max, o[cut[c + 1]] - o[cut[c]]);
        }
    }
    return true;
}

bool sort_layout(const int64_t *off, int32_t S, int32_t J, SortedLayout &out, int32_t run_max_k)
{
    const int32_t kmax = run_max_k;
    if (kmax < 4 || (kmax & 3))
        return false;
    const int64_t n_jobs = (int64_t)S * J;
    out.off.assign(1, 0);
    out.jmap.clear();
    out.scen.clear();
    out.runk.clear();
    if (n_jobs < 1 || n_jobs >= INT32_MAX)
        return false;
    out.off.reserve(n_jobs + 1);
    out.jmap.reserve(n_jobs);
    out.scen.reserve(n_jobs);
    out.runk.reserve(n_jobs);
    auto push = [&](int64_t j, int32_t s, int64_t kp, int32_t rk) {
        out.off.push_back(out.off.back() + kp);
        out.jmap.push_back((int32_t)j);
        out.scen.push_back(s);
        out.runk.push_back(rk);
    };
    std::vector<std::vector<int32_t>> bucket(kmax / 4 + 1);
    for (int32_t s = 0; s < S; ++s) {       // jobs of 3 .. kmax options, padded to 4m
        for (auto &b : bucket)
            b.clear();
        for (int64_t j = (int64_t)s * J; j < (int64_t)(s + 1) * J; ++j) {
            const int64_t K = off[j + 1] - off[j];
            if (K < 1)
                return false;
            if (K >= 3 && K <= kmax)
                bucket[(K + 3) / 4].push_back((int32_t)j);
        }
        for (int b = 1; b <= kmax / 4; ++b)
            for (int32_t j : bucket[b])
                push(j, s, 4 * b, 4 * b);
    }
    for (int32_t s = 0; s < S; ++s)         // large jobs, unpadded
        for (int64_t j = (int64_t)s * J; j < (int64_t)(s + 1) * J; ++j)
            if (off[j + 1] - off[j] > kmax)
                push(j, s, off[j + 1] - off[j], 0);
    for (int32_t s = 0; s < S; ++s)         // runs of 2- and 1-option jobs
        for (int64_t k = 2; k >= 1; --k)
            for (int64_t j = (int64_t)s * J; j < (int64_t)(s + 1) * J; ++j)
                if (off[j + 1] - off[j] == k)
                    push(j, s, k, (int32_t)k);
    return (int64_t)out.jmap.size() == n_jobs;
}

// Fitted to rounds measured on GB300: 912 tables (64 to 20000 jobs of 2 to 200 options, uniform and ragged, R = 3 to
// 12, 1 to 256 scenarios), each streamed and with every cluster size that fits. The size it picks, or streaming where that
// is predicted shorter, is within 1% of the best of all on average and 1.23x at worst (R = 12, 64 scenarios of 1000 x
// 16); the rule before it, scenarios in flight over a fitted round, was within 3.7% and 2.8x: it counted the
// scenarios that fit at once but not the waves (16 scenarios of 2048 x 16, R = 4: 5.8 us in two waves of 16 CTAs where
// one wave of 8 takes 3.8).
double resident_round_us(int32_t S, int32_t R, int64_t min_k, int64_t max_k, int32_t sms, const ResSize &o)
{
    const bool same = min_k == max_k;
    // a lane's turns of a job, each its share of the job's options one after the other, and 8 options' worth for
    // the job's end; a warp of jobs of different sizes waits for its largest
    const double turns = (double)(((int64_t)o.m_max * o.lanes + 255) / 256);
    double k = (double)((max_k + o.lanes - 1) / o.lanes);
    if (!same)
        k = std::min(k, 3.8 * (double)o.n_max / ((double)o.m_max * o.lanes) + 0.15 * k);
    // per option: wider tables take longer, and widths without an instantiation, and slices in CSR order
    const double per = (R == 4 || R == 6 || R == 8 ? 0.018 + 0.0059 * R : 0.039 + 0.0141 * R) * (same ? 1.0 : 1.13);
    double t = 1.6 + (o.cs == 1 ? 0.0 : 0.26 + 0.028 * o.cs) + per * turns * (k + 8.35);
    // the slice's options at the SM's rate: where two CTAs share one, and for the bank conflicts of CSR order
    t += per * (double)o.n_max / 256.0 * ((std::min(S, o.clusters) * o.cs > sms ? 0.53 : 0.0) + (same ? 0.0 : 0.47));
    return t * (double)((S + o.clusters - 1) / o.clusters);
}

// A launch and the update (7.6), filling the GPU's warps, then the bytes and the options; the staged pass has more
// work per option.
double streaming_round_us(int64_t n_opt, int32_t R, int32_t words, int32_t sms)
{
    const double n = (double)n_opt, full = std::min(1.0, n / (256.0 * 20.0 * sms));
    if (words > 0)
        return 7.6 + 4.9 * full + n * 4.0 * (words + 1) / 8.2e6 + 0.63e-6 * n;
    return 8.5 + 14.0 * full + n * (4.0 * R + 8.0) / 7e6;
}

int resident_choice(int32_t S, int32_t R, int64_t min_k, int64_t max_k, int32_t sms, const std::vector<ResSize> &sizes)
{
    int best = -1;
    double us = 0.0;
    for (size_t i = 0; i < sizes.size(); ++i) {
        const double t = resident_round_us(S, R, min_k, max_k, sms, sizes[i]);
        if (best < 0 || t < us) {
            us = t;
            best = (int)i;
        }
    }
    return best;
}

bool pack_format(const int32_t *umax, int32_t R, PackFormat &out, int32_t r_global, int32_t n_groups)
{
    out = PackFormat{};
    if (R < 1 || R > kMaxR)
        return false;
    const int32_t flat = n_groups > 0 ? r_global : R;   // columns priced alike for every option
    struct Col {
        int bits, col;
    };
    std::vector<Col> cols;
    for (int32_t r = 0; r < R; ++r) {
        int b = 0;
        while (b < 31 && (umax[r] >> b) != 0)
            ++b;
        if (umax[r] < 0 || b > 23)
            return false;
        cols.push_back({std::max(b, 1), r});
    }
    std::stable_sort(cols.begin(), cols.begin() + flat, [](const Col &x, const Col &y) { return x.bits > y.bits; });
    std::vector<char> used(cols.size(), 0);
    int nw = 0, taken[kPackMaxWords] = {}, high[kPackMaxWords] = {};   // bits of a word's low and high field
    for (int k = 0; k < kPackMaxWords; ++k) {   // empty words: nothing low, one bit high
        out.mask[k] = 0u;
        out.shift[k] = 31;
        out.magic[k] = 0x4b000000u >> 1;
        out.col_lo[k] = out.col_hi[k] = -1;
    }
    auto put = [&](int k, const Col &lo, const Col *hi) {
        taken[k] = lo.bits;
        out.mask[k] = (1u << lo.bits) - 1u;
        out.col_lo[k] = (int8_t)lo.col;
        out.field[lo.col] = (int8_t)(2 * k);
        if (hi) {
            out.field[hi->col] = (int8_t)(2 * k + 1);
            high[k] = hi->bits;
            out.shift[k] = 32 - hi->bits;
            out.magic[k] = 0x4b000000u >> hi->bits;   // exact: its low 24 bits are zero
            out.col_hi[k] = (int8_t)hi->col;
        }
    };
    for (int32_t i = 0; i < flat; ++i) {
        if (used[i])
            continue;
        if (nw == kPackMaxWords)
            return false;
        const Col *hi = nullptr;
        for (int32_t j = i + 1; j < flat; ++j)
            if (!used[j] && cols[i].bits + cols[j].bits <= 32) {
                used[j] = 1;
                hi = &cols[j];
                break;
            }
        put(nw++, cols[i], hi);
    }
    if (n_groups <= 0) {
        for (int n : {2, 3, 4, 6, 8})
            if (nw <= n) {
                out.nw = n;
                return true;
            }
        return false;
    }
    const Col *hi = R - flat == 2 ? &cols[flat + 1] : nullptr;
    if (R - flat < 1 || R - flat > 2 || cols[flat].bits + (hi ? hi->bits : 0) > 32)
        return false;
    int slot_bits = 1;
    while ((pack_slot((uint32_t)(n_groups - 1)) >> slot_bits) != 0)
        ++slot_bits;
    for (int n : {3, 4, 6}) {
        if (nw + 1 > n)
            continue;
        put(n - 1, cols[flat], hi);
        for (int k = 0; k < n; ++k) {
            // an empty word's high field is a zero bit of no column
            if (taken[k] + std::max(high[k], out.col_hi[k] < 0 ? 1 : 0) + slot_bits <= 32) {
                out.nw = n;
                out.g_word = k;
                out.g_shift = taken[k];
                out.g_mask = (1u << slot_bits) - 1u;
                return true;
            }
        }
        out.mask[n - 1] = 0u;   // no room for the slot: one more word
        out.shift[n - 1] = 31;
        out.magic[n - 1] = 0x4b000000u >> 1;
        out.col_lo[n - 1] = out.col_hi[n - 1] = -1;
        taken[n - 1] = high[n - 1] = 0;
    }
    return false;
}

// Kind and vector count of a job of k options, as a tile's mk. narrow: four options per lane (jobs of up to
// 128 options).
static uint32_t pack_kind(int64_t k, bool narrow)
{
    if (k <= 2)
        return (uint32_t)k << 3 | kPackTiny;
    const int64_t m = (k + 3) / 4;
    if (m > 64)
        return (uint32_t)m << 3 | kPackLarge;
    const int64_t lanes = narrow && m <= 32 ? m : (m + 1) / 2;
    uint32_t code = 0;
    while ((1 << code) < lanes)
        ++code;
    return (uint32_t)m << 3 | code;
}

bool plan_packed(const int64_t *off, int32_t S, int32_t J, int32_t max_warps, PackPlan &out, int64_t all_k)
{
    out = PackPlan();
    out.scen_tiles.assign((size_t)std::max(S, 1), 0);
    const int64_t n_jobs = (int64_t)S * J;
    if (S < 1 || J < 0 || max_warps < 1 || n_jobs >= INT32_MAX || off[0] != 0)
        return false;
    // 1. the order: within a scenario by kind and vector count (a counting sort over the kinds of at most
    //    256 options keeps the table's order inside each; larger jobs are sorted by vector count)
    struct Seg {
        int32_t job, n, scen;
        uint32_t mk;
    };
    std::vector<Seg> segs;
    bool same = true;
    if (all_k >= (int64_t)1 << 30)
        return false;
    if (all_k > 0)
        for (int32_t s = 0; s < S && J > 0; ++s)
            segs.push_back({s * J, J, s, pack_kind(all_k, false)});
    std::vector<int32_t> count(67), at(67), order(all_k > 0 ? 0 : (size_t)J), big;
    auto cls = [](uint32_t mk) { return (mk & 7u) == kPackTiny ? (int)(mk >> 3) - 1 : (int)(mk >> 3) + 1; };   // 0, 1, 2 .. 65
    std::vector<int32_t> perm;
    perm.reserve(all_k > 0 ? 0 : (size_t)n_jobs);
    std::vector<uint32_t> kind(order.size());
    for (int32_t s = 0; s < S && all_k == 0; ++s) {
        const int64_t j0 = (int64_t)s * J;
        std::fill(count.begin(), count.end(), 0);
        big.clear();
        for (int32_t j = 0; j < J; ++j) {
            const int64_t k = off[j0 + j + 1] - off[j0 + j];
            if (k < 1 || k >= (int64_t)1 << 30)
                return false;
            kind[(size_t)j] = pack_kind(k, false);
            if ((kind[(size_t)j] & 7u) == kPackLarge)
                big.push_back(j);
            else
                ++count[(size_t)cls(kind[(size_t)j])];
        }
        int32_t sum = 0;
        for (int c = 66; c >= 0; --c) {   // large vector counts first
            at[(size_t)c] = sum;
            sum += count[(size_t)c];
        }
        for (int32_t j = 0; j < J; ++j)
            if ((kind[(size_t)j] & 7u) != kPackLarge)
                order[(size_t)at[(size_t)cls(kind[(size_t)j])]++] = j;
        std::stable_sort(big.begin(), big.end(), [&](int32_t x, int32_t y) { return kind[(size_t)x] > kind[(size_t)y]; });
        std::copy(big.begin(), big.end(), order.begin() + sum);
        for (int32_t i = 0; i < J; ++i) {
            const int32_t j = order[(size_t)i];
            same = same && j == i;
            if (i == 0 || kind[(size_t)j] != segs.back().mk)
                segs.push_back({(int32_t)perm.size(), 0, s, kind[(size_t)j]});
            ++segs.back().n;
            perm.push_back((int32_t)(j0 + j));
        }
    }
    if (!same)
        out.job = std::move(perm);
    // 2. tiles: about three per warp where the table has the steps, else single steps
    for (const Seg &g : segs)
        out.steps += pack_shape(PackTile{0, 0, g.mk, (uint32_t)g.n}).steps;
    // a table of at most half a step per warp: four options per lane, twice the steps and each shorter
    // (one 2048-job cluster of 16 options per job: 128 steps of eight options per lane took 12.8 us per
    // round, 256 of four 12.2)
    out.narrow = 2 * out.steps <= max_warps;
    if (out.narrow) {
        out.steps = 0;
        for (Seg &g : segs) {
            const int64_t m = g.mk >> 3;
            if ((g.mk & 7u) < kPackTiny)
                g.mk = pack_kind(4 * m, true);
            out.steps += pack_shape(PackTile{0, 0, g.mk, (uint32_t)g.n}).steps;
        }
    }
    const int64_t steps_max = std::min<int64_t>(kPackTileSteps, std::max<int64_t>(1, out.steps / (3LL * max_warps)));
    const size_t tiles_max = segs.size() + (size_t)(out.steps / steps_max) + 1;   // about (jobs of many steps are rare)
    out.tiles.reserve(tiles_max);
    out.job_begin.reserve(tiles_max + 1);
    std::vector<int64_t> cost(1, 0), final_cost(1, 0);   // of the tiles so far, in tenths of a step
    cost.reserve(tiles_max + 1);
    final_cost.reserve(tiles_max + 1);
    for (const Seg &g : segs) {
        const PackShape one = pack_shape(PackTile{0, 0, g.mk, 1});
        const int64_t jobs_max = std::max<int64_t>(1, steps_max / one.nch) * one.per_step;
        for (int64_t a = 0; a < g.n; a += jobs_max) {
            PackTile t;
            t.base = (uint32_t)out.vecs;
            t.scenario = (uint32_t)g.scen;
            t.mk = g.mk;
            t.n_job = (uint32_t)std::min<int64_t>(jobs_max, g.n - a);
            const PackShape sh = pack_shape(t);
            out.job_begin.push_back((int32_t)(g.job + a));
            out.vecs += (int64_t)sh.steps * sh.v;
            if (out.vecs > (int64_t)UINT32_MAX)
                return false;
            ++out.scen_tiles[(size_t)g.scen];
            out.tiles.push_back(t);
            cost.push_back(cost.back() + 5 + 10LL * sh.steps);
            final_cost.push_back(final_cost.back() + 5 + (sh.code == (int)kPackTiny ? kPackFinalTiny : 10) * sh.steps);
        }
    }
    out.job_begin.push_back((int32_t)n_jobs);
    if (out.tiles.size() >= (size_t)INT32_MAX)
        return false;
    // 3. the passes' ranges: contiguous tiles of about equal cost. In the final pass a lane of a step of one- and
    //    two-option jobs writes the outputs of up to eight winners, others of one at most.
    const int64_t n_tiles = (int64_t)out.tiles.size();
    const int32_t W = (int32_t)std::min<int64_t>(max_warps, n_tiles);
    out.n_warps = W;
    auto split = [&](const std::vector<int64_t> &pre, std::vector<int32_t> &begin) {
        begin.assign((size_t)W + 1, 0);
        int64_t at = 0;   // first tile boundary at or beyond the target, which only grows
        for (int32_t w = 1; w < W; ++w) {
            const int64_t target = (int64_t)((__int128)pre[n_tiles] * w / W);
            while (pre[at] < target)
                ++at;
            int64_t i = at;
            if (i > 0 && target - pre[i - 1] < pre[i] - target)
                --i;
            begin[w] = (int32_t)std::min<int64_t>(std::max<int64_t>(i, begin[w - 1]), n_tiles);
        }
        begin[W] = (int32_t)n_tiles;
    };
    split(cost, out.warp_begin);
    split(final_cost, out.final_begin);
    return true;
}

bool check_packed(const int64_t *off, int32_t S, int32_t J, const PackPlan &p, int64_t all_k)
{
    const int64_t n_jobs = (int64_t)S * J, n_tiles = (int64_t)p.tiles.size();
    if ((int64_t)p.job_begin.size() != n_tiles + 1 || p.job_begin.front() != 0 || p.job_begin.back() != n_jobs ||
        (!p.job.empty() && (int64_t)p.job.size() != n_jobs))
        return false;
    std::vector<char> seen(p.job.empty() ? 0 : (size_t)n_jobs, 0);
    std::vector<int32_t> count((size_t)S, 0);
    int64_t vecs = 0;
    int32_t last = 0;
    for (int64_t i = 0; i < n_tiles; ++i) {
        const PackTile &t = p.tiles[(size_t)i];
        if (t.base != (uint64_t)vecs || t.n_job < 1 || (int64_t)p.job_begin[i] + t.n_job != p.job_begin[i + 1] ||
            (int32_t)t.scenario < last || (int32_t)t.scenario >= S)
            return false;
        last = (int32_t)t.scenario;
        if (all_k > 0) {   // every job alike, in the table's order: the ends tell
            if (!p.job.empty() || p.job_begin[i] / J != (int32_t)t.scenario || (p.job_begin[i + 1] - 1) / J != (int32_t)t.scenario ||
                pack_kind(all_k, p.narrow) != t.mk)
                return false;
        }
        for (int64_t q = p.job_begin[i]; q < p.job_begin[i + 1] && all_k == 0; ++q) {
            const int64_t j = p.job.empty() ? q : p.job[(size_t)q];
            if (j < (int64_t)t.scenario * J || j >= (int64_t)(t.scenario + 1) * J || pack_kind(off[j + 1] - off[j], p.narrow) != t.mk)
                return false;
            if (!p.job.empty()) {
                if (seen[(size_t)j])
                    return false;
                seen[(size_t)j] = 1;
            }
        }
        const PackShape sh = pack_shape(t);
        if (sh.v < 1 || sh.v > kPackStepVecs || sh.steps < 1 ||
            (sh.code < (int)kPackTiny && (sh.code > 5 || sh.ca > (1 << sh.code))))
            return false;
        ++count[(size_t)t.scenario];
        vecs += (int64_t)sh.steps * sh.v;
    }
    if (vecs != p.vecs || count != p.scen_tiles)
        return false;
    for (const std::vector<int32_t> *b : {&p.warp_begin, &p.final_begin}) {
        if ((int32_t)b->size() != p.n_warps + 1 || b->front() != 0 || b->back() != n_tiles)
            return false;
        for (int32_t w = 0; w < p.n_warps; ++w)
            if ((*b)[w] > (*b)[w + 1])
                return false;
    }
    return true;
}

}  // namespace esp
