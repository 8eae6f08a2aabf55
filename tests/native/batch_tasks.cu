// Steps a CTA's groups through its sequence of tasks (TaskCursor) from a given sweep on and compares
// every task with the quotient and remainder in 64 bits. The counter is the kernel's: 32 bits.
// Arguments: chains, sweeps, first sweep, tasks to take, groups.
// Prints the tasks compared, or the first difference.
#include <stdio.h>
#include <stdlib.h>

#include <vector>

#include "pt_internal.h"

int main(int argc, char** argv) {
    if (argc != 6) return 1;
    const int count = atoi(argv[1]), n_groups = atoi(argv[5]);
    const long long sweeps = atoll(argv[2]), first = atoll(argv[3]), tasks = atoll(argv[4]);
    unsigned long long number = (unsigned long long)first * count;
    std::vector<ptq::TaskCursor> at;
    for (int g = 0; g < n_groups; ++g, ++number) {  // where the groups stand in that sweep
        at.emplace_back(g);
        at[g].task = (unsigned)number;
        at[g].s = (int)first;
    }
    unsigned draw = 12345u;
    long long done = 0;
    for (; done < tasks && number < (unsigned long long)(sweeps + 1) * count; ++done, ++number) {
        draw = draw * 1664525u + 1013904223u;
        ptq::TaskCursor& a = at[(draw >> 16) % n_groups];
        a.move_to((unsigned)number, count);
        const unsigned long long s = number / count;
        if (a.s < 0 || a.s > sweeps || (unsigned long long)a.s != s || a.lc < 0 ||
            (unsigned long long)a.lc != number - s * count) {
            printf("task %llu: sweep %d chain %d\n", number, a.s, a.lc);
            return 2;
        }
    }
    printf("%lld\n", done);
    return 0;
}
