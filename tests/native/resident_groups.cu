// Layouts of resident chains with a given group width (kernel path 7), host code only. Input lines:
//   N P R Lmax dc n_levels cluster group_threads; output per line: groups and bytes, or 0 0.
#include <stdio.h>

#include "pt_internal.h"

int main() {
    const size_t cap = 227 * 1024 - 1024;
    ptq::BatchInstance I = {};
    int cluster, group;
    while (scanf("%d %d %d %d %d %d %d %d", &I.N, &I.P, &I.R, &I.Lmax, &I.dc, &I.n_levels, &cluster, &group) == 8) {
        I.nL3 = 3 * (2 * I.Lmax + 1);
        I.slot_stride = (I.N * I.P + 15) / 16 * 16;
        ptq::BatchInstance T = I;
        if (ptq::resident_groups(T, cluster, 512, cap, group, 1))
            printf("%d %d\n", T.n_groups, (int)ptq::batch_smem_bytes(T, cluster, 512));
        else
            printf("0 0\n");
    }
    return 0;
}
