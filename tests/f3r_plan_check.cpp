// csrc/f3r_plan.h: prints "elems blocks trials" for n, SMs, blocks per SM of the two kernels and
// the most blocks that a launch may have.
#include <cstdio>
#include <cstdlib>

#include "f3r_plan.h"

int main(int argc, char **argv) {
    for (int i = 1; i + 4 < argc; i += 5) {
        const long long n = atoll(argv[i]);
        const int sms = atoi(argv[i + 1]), per16 = atoi(argv[i + 2]), per32 = atoi(argv[i + 3]);
        const int granted = atoi(argv[i + 4]);
        int trials = 0;
        const packsell::StepPlan p = packsell::plan_step(
            n, sms, 256, [&](int e) { return e == 16 ? per16 : per32; },
            [&](int, int blocks) { return ++trials, blocks <= granted; });
        std::printf("%d %d %d\n", p.elems, p.blocks, trials);
    }
}
