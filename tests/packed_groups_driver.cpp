// Test driver for the word layout of grouped tables (compiled by tests/test_packed_groups.py with the
// sanitizers): reads int64 words n_cases, then per case R, r_global, n_groups, umax [R]; writes per case ok,
// nw, g_word, g_shift, g_mask, then per word mask, shift, magic, col_lo, col_hi; and at the end whether every
// group below 65536 comes back from its slot.
#include <cstdint>
#include <cstdio>
#include <vector>

#include "esp_plan.h"

int main(int argc, char **argv)
{
    if (argc != 3)
        return 2;
    std::FILE *f = std::fopen(argv[1], "rb");
    std::vector<int64_t> w, out;
    int64_t x;
    while (f && std::fread(&x, 8, 1, f) == 1)
        w.push_back(x);
    if (f)
        std::fclose(f);
    size_t at = 0;
    for (int64_t c = w.at(at++); c > 0; --c) {
        const int32_t R = (int32_t)w.at(at), rg = (int32_t)w.at(at + 1), ng = (int32_t)w.at(at + 2);
        at += 3;
        std::vector<int32_t> um;
        for (int32_t r = 0; r < R; ++r)
            um.push_back((int32_t)w.at(at++));
        esp::PackFormat fm;
        out.push_back(esp::pack_format(um.data(), R, fm, rg, ng));
        for (int64_t v : {(int64_t)fm.nw, (int64_t)fm.g_word, (int64_t)fm.g_shift, (int64_t)fm.g_mask})
            out.push_back(v);
        for (int k = 0; k < esp::kPackMaxWords; ++k)
            for (int64_t v : {(int64_t)fm.mask[k], (int64_t)fm.shift[k], (int64_t)fm.magic[k], (int64_t)fm.col_lo[k],
                              (int64_t)fm.col_hi[k]})
                out.push_back(v);
    }
    bool back = true;
    for (uint32_t g = 0; g < 65536; ++g)
        back = back && esp::pack_slot_group(esp::pack_slot(g)) == g && (g == 0 || esp::pack_slot(g) > esp::pack_slot(g - 1));
    out.push_back(back);
    f = std::fopen(argv[2], "wb");
    if (!f || std::fwrite(out.data(), 8, out.size(), f) != out.size())
        return 2;
    return std::fclose(f) ? 2 : 0;
}
