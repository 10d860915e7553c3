// Host check of the row sweep's shared-memory layout (paper_0706_3293_gb300/csrc/hm_row.cuh, row_stage): every table
// starts on its type's alignment from a 16-byte aligned base.  Prints the violations and returns their number.
#include <cstdio>

#include "hm_row.cuh"

template <class I, class Acc>
static int check(int nc, int S2, int cd_len) {
    hm::RowPlan P{};
    hm::SectorView sv{};
    P.nc = nc;
    sv.S2 = S2;
    sv.cd_len = cd_len;
    const size_t coef = hm::row_coef_bytes(P, S2, sizeof(Acc)), g = coef + 4 * (size_t)cd_len * sizeof(I);
    const size_t cd = coef + 6 * (size_t)cd_len * sizeof(I), slots = coef + hm::row_tab_bytes<I>(sv);
    const bool ok = alignof(hm::RowEF<I>) <= 16 && alignof(hm::RowG<I>) <= 16 && coef % alignof(hm::RowEF<I>) == 0 &&
                    g % alignof(hm::RowG<I>) == 0 && cd % alignof(I) == 0 && slots % alignof(hm::RowG<I>) == 0;
    if (!ok) printf("index %zu bytes, sums %zu bytes, %d classes, 2s = %d, %d entries\n", sizeof(I), sizeof(Acc), nc, S2, cd_len);
    return ok ? 0 : 1;
}

int main() {
    int bad = 0;
    for (int nc = 1; nc <= 5; ++nc)
        for (int S2 = 1; S2 <= 7; ++S2)
            for (int len : {3, 4, 5, 6, 7, 100, 101})
                bad += check<uint32_t, float>(nc, S2, len) + check<uint32_t, double>(nc, S2, len) +
                       check<uint64_t, float>(nc, S2, len) + check<uint64_t, double>(nc, S2, len);
    return bad != 0;
}
