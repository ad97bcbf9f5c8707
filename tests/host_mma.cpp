// The host side of the tensor-core base conversion (mmaplan.cpp) for
// test_host_mma.py: the rule that chooses the form.
#include <algorithm>

#include "internal.h"

namespace catfhe {
bool plan_fits_mont(const PlanSpec &) { return true; }
}  // namespace catfhe

using namespace catfhe;

// `plans` conversions of K[i] sources and T[i] targets, split weights or not.
extern "C" int mma_rule(int plans, const int *K, const int *T, int split, uint64_t coeffs,
                        int sms, int beside) {
    ConvPlans cp{};
    cp.mma = true;
    cp.l.n = cp.m.n = uint32_t(plans);
    cp.l.mont = 1;
    cp.l.split = uint32_t(split);
    cp.l.kmin = cp.l.kmax = uint32_t(K[0]);
    for (int i = 0; i < plans; i++) {
        cp.m.head[i] = uint64_t(K[i]);
        for (int t = 0; t < T[i]; t += 3)
            cp.m.counts[i] |= uint64_t(T[i] - t < 3 ? T[i] - t : 3) << (4 * (t / 3));
        cp.l.kmin = std::min(cp.l.kmin, uint32_t(K[i]));
        cp.l.kmax = std::max(cp.l.kmax, uint32_t(K[i]));
    }
    return mma_is_faster(cp, coeffs, sms, beside != 0);
}
