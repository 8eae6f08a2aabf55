// Prints the layouts choose_groups gives requests on clusters of each size, and what every CTA does
// with its share of the chains (host code only). Input, per request: n edges P R lmax-free couplings:
//   n n_edges P R, then ei ej J per edge, then h per site; ends with n = 0.
// Output, per request and cluster: P R lmax cluster form group_threads n_groups resident buffers bytes
//   | count keep in_place of every CTA.
#include <stdio.h>

#include <vector>

#include "pt_internal.h"

int main() {
    const size_t cap = 227 * 1024 - 1024;
    int n, ne, P, R;
    while (scanf("%d %d %d %d", &n, &ne, &P, &R) == 4 && n > 0) {
        std::vector<int32_t> ei(ne), ej(ne), J(ne), h(n);
        for (int k = 0; k < ne; ++k)
            if (scanf("%d %d %d", &ei[k], &ej[k], &J[k]) != 3) return 1;
        for (int i = 0; i < n; ++i)
            if (scanf("%d", &h[i]) != 1) return 1;
        std::vector<pt_rung> ladder(R, pt_rung{1.0, 1.0});
        pt_request r = {};
        r.inst = {n, ne, ei.data(), ej.data(), J.data(), h.data()};
        r.P = P;
        r.R = R;
        r.ladder = ladder.data();
        r.n_sweeps = 1;
        ptq::Prepared pr;
        char why[200];
        if (ptq::prepare_request(r, pr, why, sizeof(why), 32 / (P / 8) > 1 ? 32 / (P / 8) : 1)) {
            fprintf(stderr, "%s\n", why);
            return 1;
        }
        ptq::request_block_layout(pr);
        for (int K = 1; K <= 16; ++K) {
            ptq::BatchInstance I = {};
            ptq::fill_instance(I, pr, nullptr, r);
            ptq::choose_groups(I, K, 512, cap);
            const size_t bytes = ptq::batch_smem_bytes(I, K, 512);
            printf("%d %d %d %d %d %d %d %d %d %d |", P, R, I.Lmax, K, I.form, I.group_threads, I.n_groups, I.resident,
                   ptq::CtaShare::buffers(I, K), bytes <= cap ? (int)bytes : -1);
            for (int rank = 0; rank < K; ++rank) {
                const ptq::CtaShare s(I, rank, K);
                printf(" %d %d %d", s.count, (int)s.keep, (int)s.in_place);
            }
            printf("\n");
        }
    }
    return 0;
}
