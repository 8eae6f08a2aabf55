// Compares the least shared memory each kernel path asks for with what a chain of that path may
// need at most: its spins and one row more, descriptors, schedule, one threshold row as the caller
// gives it, random words, and 800 bytes of scratch. Host code only; prints the layouts compared, or
// every one that asks for more.
#include <stdio.h>
#include <string.h>

#include "pt_internal.h"

static size_t up16(size_t x) { return (x + 15) & ~(size_t)15; }

int main() {
    using namespace ptq;
    int compared = 0, over = 0;
    for (int Lmax = 1; Lmax <= 127; ++Lmax)
        for (int P = 8; P <= 256; P += P < 64 ? 8 : 64)
            for (int N : {1, 3, 97, 1000, 4100})
                for (int dc : {4, 8})
                    for (int path : {kPathPackedInline, kPathPacked, kPathBits, kPathSplit, kPathSplitInline, kPathPeer}) {
                        if (P % 16 && (path == kPathSplit || path == kPathSplitInline)) continue;
                        DevProblem p;
                        memset(&p, 0, sizeof(p));
                        p.N = N;
                        p.P = P;
                        p.R = 4;
                        p.Lmax = Lmax;
                        p.nL3 = 3 * (2 * Lmax + 1);
                        p.n_levels = N + 1 < 20 ? N + 1 : 20;
                        const bool split = path == kPathSplit || path == kPathSplitInline;
                        const size_t W = P / 16, row = split ? 8 * W + 16 : (path == kPathBits ? P / 8 : P);
                        size_t most = split ? up16((N + 1) * row) : up16(N * row) + up16(row);
                        if (path == kPathBits) most += 2048;
                        most += (size_t)N * (dc == 4 ? 32 : 48) + up16(8 * (size_t)N) + up16(4 * (p.n_levels + 1)) +
                                up16(4 * (size_t)p.nL3) + 800 + (split ? 64 : 0);
                        if (path == kPathPacked || path == kPathPeer) most += 64 * (size_t)N * (P / 8);
                        if (path == kPathSplit) most += 64 * (size_t)N * (W + 1);
                        const size_t need = sweep_smem_bytes(p, path, dc);
                        ++compared;
                        if (need > most) {
                            if (++over < 20)
                                printf("path %d N %d P %d Lmax %d dc %d: %zu > %zu\n", path, N, P, Lmax, dc, need, most);
                        }
                    }
    printf("%d %d\n", compared, over);
    return over != 0;
}
