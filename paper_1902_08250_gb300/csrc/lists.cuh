// lists.cuh -- rules of the uniform tree's interaction lists, shared by the device
// list builder and the host code that enumerates them.
#pragma once
#include <map>
#include <tuple>
#include <vector>

#include "internal.h"

// inverse: source row whose image row is ri
__host__ __device__ inline int64_t src_row(int term, int64_t ri, int64_t nrow)
{
    switch (term) {
    case 0: return ri;
    case 1: return -1 - ri;
    case 2: return 2 * nrow - 1 - ri;
    case 3: return ri + 2 * nrow;
    default: return ri - 2 * nrow;
    }
}
__host__ __device__ inline int64_t floordiv2(int64_t a) { return a >= 0 ? a / 2 : -((-a + 1) / 2); }
__host__ __device__ inline bool adj(int64_t c1, int64_t r1, int64_t c2, int64_t r2)
{
    return (c1 - c2 <= 1 && c2 - c1 <= 1) && (r1 - r2 <= 1 && r2 - r1 <= 1);
}
__host__ __device__ inline bool v_rule(int l, int64_t ct, int64_t rt, int64_t cs, int64_t ri)
{
    if (adj(ct, rt, cs, ri)) return false;
    if (l == 0) return true;
    return adj(ct / 2, floordiv2(rt), cs / 2, floordiv2(ri));
}

// An interior box's V list depends only on its row and its column's parity (levels >= 1): the entry
// lists of every (row, parity) class of a level, [2 row + parity], e0 their offsets.  A source column
// c - dc outside the level is an entry that the target does not have.  Level 0 is one row of boxes whose
// lists hold every class: one list.
struct RowEnt {
    int32_t slot, dc, rs, pad; // table slot, target column - source column, source row
};
inline lm_status lm_row_entries(const Level &lv, std::vector<RowEnt> &ents, std::vector<int32_t> &e0)
{
    std::map<std::tuple<int, int, int>, int> slot;
    for (size_t i = 0; i < lv.cls_term.size(); ++i) slot[{lv.cls_term[i], lv.cls_dc[i], lv.cls_dr[i]}] = (int)i;
    ents.clear();
    e0.clear();
    if (lv.l == 0) {
        e0 = {0, (int32_t)lv.cls_term.size()};
        for (size_t i = 0; i < lv.cls_term.size(); ++i) ents.push_back(RowEnt{(int32_t)i, lv.cls_dc[i], 0, 0});
        return LM_OK;
    }
    for (int64_t rt = 0; rt < lv.nrow; ++rt)
        for (int par = 0; par < 2; ++par) {
            e0.push_back((int32_t)ents.size());
            const int64_t ct = 8 + par; // an interior column
            for (int term = 0; term < 5; ++term) {
                const int64_t a = src_row(term, rt - 3, lv.nrow), b = src_row(term, rt + 3, lv.nrow);
                const int64_t rlo = a < b ? a : b, rhi = a < b ? b : a;
                for (int64_t rs = rlo > 0 ? rlo : 0; rs <= rhi && rs < lv.nrow; ++rs) {
                    const int64_t ri = img_row(term, rs, lv.nrow);
                    for (int64_t cs = ct - 3; cs <= ct + 3; ++cs) {
                        if (!v_rule(lv.l, ct, rt, cs, ri)) continue;
                        auto f = slot.find({term, (int)(ct - cs), (int)(rt - ri)});
                        if (f == slot.end()) {
                            lm_set_error("build_tree: internal error, an interaction has no translation class");
                            return LM_ECUDA;
                        }
                        ents.push_back(RowEnt{f->second, (int32_t)(ct - cs), (int32_t)rs, 0});
                    }
                }
            }
        }
    e0.push_back((int32_t)ents.size());
    return LM_OK;
}
