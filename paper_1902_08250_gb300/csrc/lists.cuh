// lists.cuh -- rules of the uniform tree's interaction lists, shared by the device
// list builder and the host code that enumerates them.
#pragma once
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
