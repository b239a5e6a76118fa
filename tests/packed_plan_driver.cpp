// Test driver for the packed passes' host planner (compiled by tests/test_packed_plan.py with the
// sanitizers): reads int64 words n_cases, then per case S, J, R, max_warps, all_k, job offsets [S*J + 1],
// umax [R]; writes per case: format ok, nw, then per word mask, shift, magic, col_lo, col_hi; plan ok, check ok,
// n_tiles, n_warps, vecs, steps, narrow, per tile base, scenario, mk, n_job, job_begin; the packed order [S*J];
// warp_begin [n_warps + 1]; and whether the check refuses the plan with its last job range shifted.
#include <cstdint>
#include <cstdio>
#include <vector>

#include "esp_plan.h"

int main(int argc, char **argv)
{
    if (argc != 3)
        return 2;
    std::FILE *f = std::fopen(argv[1], "rb");
    std::vector<int64_t> w;
    int64_t x;
    while (f && std::fread(&x, 8, 1, f) == 1)
        w.push_back(x);
    if (f)
        std::fclose(f);
    size_t at = 0;
    std::vector<int64_t> out;
    const int64_t n = w.at(at++);
    for (int64_t c = 0; c < n; ++c) {
        const int32_t S = (int32_t)w.at(at), J = (int32_t)w.at(at + 1), R = (int32_t)w.at(at + 2);
        const int32_t warps = (int32_t)w.at(at + 3);
        const int64_t all_k = w.at(at + 4);
        at += 5;
        std::vector<int64_t> off(w.begin() + (long)at, w.begin() + (long)at + (long)S * J + 1);
        at += off.size();
        std::vector<int32_t> um;
        for (int32_t r = 0; r < R; ++r)
            um.push_back((int32_t)w.at(at++));
        esp::PackFormat fm;
        out.push_back(esp::pack_format(um.data(), R, fm));
        out.push_back(fm.nw);
        for (int k = 0; k < esp::kPackMaxWords; ++k)
            for (int64_t v : {(int64_t)fm.mask[k], (int64_t)fm.shift[k], (int64_t)fm.magic[k], (int64_t)fm.col_lo[k],
                              (int64_t)fm.col_hi[k]})
                out.push_back(v);
        esp::PackPlan p;
        const bool ok = esp::plan_packed(off.data(), S, J, warps, p, all_k);
        out.push_back(ok);
        if (!ok)
            continue;
        out.push_back(esp::check_packed(off.data(), S, J, p, all_k));
        for (int64_t v : {(int64_t)p.tiles.size(), (int64_t)p.n_warps, p.vecs, p.steps, (int64_t)p.narrow})
            out.push_back(v);
        for (size_t i = 0; i < p.tiles.size(); ++i)
            for (int64_t v : {(int64_t)p.tiles[i].base, (int64_t)p.tiles[i].scenario, (int64_t)p.tiles[i].mk,
                              (int64_t)p.tiles[i].n_job, (int64_t)p.job_begin[i]})
                out.push_back(v);
        for (int64_t j = 0; j < (int64_t)S * J; ++j)
            out.push_back(p.job.empty() ? j : p.job[(size_t)j]);
        for (int32_t v : p.warp_begin)
            out.push_back(v);
        esp::PackPlan q = p;
        ++q.tiles.back().n_job;
        out.push_back(!esp::check_packed(off.data(), S, J, q, all_k));
    }
    f = std::fopen(argv[2], "wb");
    if (!f || std::fwrite(out.data(), 8, out.size(), f) != out.size())
        return 2;
    return std::fclose(f) ? 2 : 0;
}
