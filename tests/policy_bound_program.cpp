/* policy_bound on the weights of stdin (float32): argv[1] hidden units, argv[2] 1 with a second hidden layer,
 * argv[3] roundings per term. Prints the base, the bound and the largest |w1[j] - w0[j]|.
 * With argv[1] "rounds": the roundings stated for argv[2] units, argv[3] 1 with a second hidden layer, over argv[4]
 * lanes, 0 where one lane reads the paired layout. */
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "../paper_2301_13062_b200/csrc/policy_bound.h"

int main(int, char **argv) {
    if (!strcmp(argv[1], "rounds")) {
        const int units = atoi(argv[2]), lanes = atoi(argv[4]);
        printf("%d\n", lanes ? cp::lanes_rounds(units, lanes) : cp::units_rounds(units, atoi(argv[3]) != 0));
        return 0;
    }
    const int units = atoi(argv[1]);
    const bool deep = atoi(argv[2]) != 0;
    std::vector<float> w(7 * units + 2 + (deep ? units * (units + 1) : 0)), steps(units);
    if (fread(w.data(), sizeof(float), w.size(), stdin) != w.size()) return 1;
    const cp::PolicyBound b = cp::policy_bound(w.data(), units, deep, atoi(argv[3]), steps.data());
    float largest = 0.0f;
    for (float v : steps) largest = std::fmax(largest, std::fabs(v));
    printf("%.9g %.9g %.9g\n", b.base, b.bound, largest);
    return 0;
}
