// fx_host.cu -- host-side checks of the fixed-point kernels' code
// (tests/test_fixed_point_host.py): what can be shown without a GPU.
#include <stdio.h>

#include <set>
#include <vector>

#include "gsm_fx3.cuh"

using namespace gsm;

// Shared words that each sync group of the 64 R kernels touches, in the
// reductions of the first stage and in the conv's sums: no word may belong to
// two groups, and all must lie in the arrays.
template <int R>
int groups_share_words()
{
    using F = F3<R>;
    const int count = sizeof(F3Shared<R>::r1) / sizeof(int), groups = F::NL / F::LG;
    std::vector<std::set<int>> words(groups);
    for (int tid = 0; tid < F::THREADS; ++tid) {
        const int line = tid / F::NB, b = tid % F::NB;
        if (F::SEG > 1 && b % F::W == 0) words[tid / F::SG].insert(F::reduce_word(line, b / F::W));
        for (int k = 0; k < F::KC && !F::TWO; ++k) {   // F3Thread::last_bfly
            const int q = tid % F::SG + k * F::SG, ln = tid / F::SG * F::LG + q / F::BC, bc = q % F::BC;
            if (q >= F::BC * F::LG) continue;
            for (int half = 0; half < 2; ++half) words[tid / F::SG].insert(F::conv_word(ln, half));
            if (bc >> 5 > 1) return 1;
        }
    }
    std::set<int> seen;
    for (const auto &w : words)
        for (int i : w)
            if (i < 0 || i >= count || !seen.insert(i).second) return 1;
    return 0;
}

int main()
{
    const int bad[] = {groups_share_words<1>(), groups_share_words<2>(), groups_share_words<3>(), groups_share_words<4>(),
                       groups_share_words<5>(), groups_share_words<6>(), groups_share_words<8>()};
    for (int b : bad) printf("%d ", b);
    printf("\n");
    return 0;
}
