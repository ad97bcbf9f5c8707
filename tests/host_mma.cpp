// The host side of the tensor-core base conversion (mmaplan.cpp) for
// test_host_mma.py: the rule that chooses the form, and the image of a plan.
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

// The image for sources src (factors pre), targets dst (factors post): its
// words, -1 if there is none.
extern "C" int mma_plan(int K, const uint64_t *src, const uint64_t *pre, int T, const uint64_t *dst,
                        const uint64_t *post, uint64_t *img, int cap) {
    PlanSpec s;
    for (int i = 0; i < K; i++) {
        s.src_mod.push_back(src[i]);
        s.src_off.push_back(uint32_t(i));
        s.pre.push_back(pre[i]);
    }
    for (int t = 0; t < T; t++) {
        s.dst_mod.push_back(dst[t]);
        s.dst_off.push_back(uint32_t(t));
        s.post.push_back(post[t]);
    }
    const std::vector<uint64_t> v = build_mma_plan(s, 1, 1);
    if (v.empty() || int(v.size()) > cap) return -1;
    std::copy(v.begin(), v.end(), img);
    return int(v.size());
}
