// Steps a CTA's groups through its sequence of tasks (TaskCursor) and compares every task with the
// quotient and remainder in 64 bits. Arguments: chains, sweeps, first sweep, tasks to take.
// Prints the tasks compared, or the first difference.
#include <stdio.h>
#include <stdlib.h>

#include "pt_internal.h"

int main(int argc, char** argv) {
    if (argc != 5) return 1;
    const int count = atoi(argv[1]), n_groups = 16;
    const long long sweeps = atoll(argv[2]), first = atoll(argv[3]), tasks = atoll(argv[4]);
    unsigned long long next = (unsigned long long)first * count;
    ptq::TaskCursor at[n_groups];
    unsigned draw = 12345u;
    long long done = 0;
    for (; done < tasks && next < (unsigned long long)(sweeps + 1) * count; ++done, ++next) {
        draw = draw * 1664525u + 1013904223u;
        ptq::TaskCursor& a = at[(draw >> 16) % n_groups];
        a.move_to(next, count);
        const unsigned long long s = next / count;
        if (a.s < 0 || a.s > sweeps || (unsigned long long)a.s != s || a.lc < 0 ||
            (unsigned long long)a.lc != next - s * count) {
            printf("task %llu: sweep %d chain %d\n", next, a.s, a.lc);
            return 2;
        }
    }
    printf("%lld\n", done);
    return 0;
}
