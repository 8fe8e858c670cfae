// Which form an Arnoldi step of F3R takes. Host code without CUDA, so that the
// rule is checked on a machine with no GPU.
#pragma once

#include <stdint.h>

#include <algorithm>

namespace packsell {

struct StepPlan {
    int elems = 0;   // elements per thread of the cooperative kernel; 0: the three separate kernels
    int blocks = 0;  // of the cooperative kernel
};

// The cooperative kernel needs all its blocks resident at once and the whole
// vector in their registers: 16 elements per thread where that is enough (up
// to 2.49M unknowns on 152 SMs), else 32 (up to 4.98M). Small vectors get one
// vector of four per thread, on as few blocks as that takes. per_sm(E): blocks
// of the E-element kernel that fit on an SM (0: unknown). fits(E, blocks):
// whether such a launch is accepted; the device may grant this process fewer
// SMs than it reports, and then the separate kernels run instead.
template <typename PerSm, typename Fits>
StepPlan plan_step(int64_t n, int sms, int threads, PerSm per_sm, Fits fits) {
    for (int e : {16, 32}) {
        const int64_t most = (int64_t)sms * std::min(per_sm(e), 4);
        const int64_t want = std::max<int64_t>(1, (n / 4 + threads - 1) / threads);
        const int64_t blocks = std::min(most, want);
        if (blocks < 1 || n / 4 > blocks * threads * (e / 4)) continue;
        if (fits(e, (int)blocks)) return StepPlan{e, (int)blocks};
    }
    return StepPlan{};
}

}  // namespace packsell
