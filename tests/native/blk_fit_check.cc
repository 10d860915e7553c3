// Prints blk_fitting_K (paper_0706_3293_gb300/csrc/blk_fit.h, compiled here as plain C++) for bond lists from
// standard input: "nb own k0 kmax sl sx sg", then nb times "p q class".
#include <cstdio>
#include <vector>

#include "blk_fit.h"

int main() {
    int nb, own, k0, kmax, sl, sx, sg;
    while (scanf("%d %d %d %d %d %d %d", &nb, &own, &k0, &kmax, &sl, &sx, &sg) == 7) {
        std::vector<unsigned char> p(nb), q(nb);
        std::vector<int> c(nb);
        for (int t = 0; t < nb; ++t)
            if (scanf("%hhu %hhu %d", &p[t], &q[t], &c[t]) != 3) return 1;
        const int K = hm::blk_fitting_K(nb, p.data(), q.data(), c.data(), own != 0, k0, kmax, sl, sx, sg);
        printf("%d %d\n", K, (int)(K >= 0 && hm::blk_slots_fit(nb, p.data(), q.data(), c.data(), own != 0, K, sl, sx, sg)));
    }
    return 0;
}
