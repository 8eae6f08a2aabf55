// pt_batch.cu -- many independent PT-QMC problems in one persistent launch.
//
// Each thread-block cluster pulls a whole problem from a work counter (problems sorted by
// work, largest first) and owns it until every sweep is done: CTA r of the cluster sweeps
// chains [r*C, (r+1)*C), C = ceil(R / cluster). Within a CTA the chains are "packed" onto
// groups of threads (the paper's chain packing, Sec. 5): a group sweeps one chain at a time
// with the same level schedule, random-number counters and update arithmetic as the
// single-problem kernel, so every problem gets exactly the bits it would get alone.
//
// Nothing waits for a whole sweep of the problem. A CTA's work is the sequence of tasks
// (sweep, chain), sweep by sweep; its groups take the next task as they come free (or, with
// no more chains than groups, each group keeps its chain). A task needs its chain's previous
// sweep, and the swap decision that follows it: the chain's (E, M) and its partner's, which
// every chain publishes after its sweep in mailboxes that all CTAs of the cluster hold (as
// path 9 does), so partners evaluate the same decision and no barrier orders the passes. A
// task waits only for tasks of an earlier sweep, and those are taken first, so some task can
// always run; the waits have a time limit all the same. Only the CTAs of one cluster wait
// for one another, and those are resident together.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdarg.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <cmath>
#include <map>
#include <mutex>
#include <string>
#include <thread>
#include <vector>

#include "pt.h"
#include "pt_device.cuh"
#include "pt_internal.h"

namespace cg = cooperative_groups;

namespace ptq {

// Shared memory of one CTA while it owns problem I.
struct BatchLayout {
    size_t sdesc, items, loff, rung, seq, E, M, mail, thr, red, ctl, chains, total;
    int C, ngroups, chain_stride, nbufs, DW, thr_words;
    __host__ __device__ BatchLayout(const BatchInstance& I, int K, int threads) {
        DW = I.dc == 4 ? 8 : 12;
        C = (I.R + K - 1) / K;
        ngroups = I.n_groups;
        chain_stride = (int)up16((size_t)I.N * form_row_bytes(I.form, I.P));
        nbufs = CtaShare::buffers(I, K);
        thr_words = (int)(up16((size_t)IndexRule(I.Lmax).row_words() * 4) / 4);
        size_t o = 0;
        sdesc = o;  o += (size_t)I.N * DW * 4;
        items = o;  o += up16((size_t)2 * I.N * 4);
        loff = o;   o += up16((size_t)(I.n_levels + 1) * 4);
        rung = o;   o += up16((size_t)C * 4);
        seq = o;    o += up16((size_t)C * 4);
        E = o;      o += up16((size_t)C * 8);
        M = o;      o += up16((size_t)C * 8);
        mail = o;   o += I.mail_smem ? (size_t)kClusterMailPasses * I.R * 16 : 0;
        thr = o;    o += (size_t)(I.thr_resident ? I.R : ngroups) * thr_words * 4;
        red = o;    o += up16((size_t)ngroups * (I.group_threads / 32) * 3 * 4);
        ctl = o;    o += up16((size_t)ngroups * 16);
        chains = o; o += (size_t)nbufs * chain_stride;
        total = o;
    }
};

// Shared memory of the persistent kernel that outlives a problem.
struct BatchShared {
    unsigned long long mbar[16];  // per group: arrival of a streamed chain
    long long limit_ns;           // the time limit of every wait ...
    int* status;                  // ... and the word that says PT_ETIMEDOUT when one ran out
    uint32_t phase[16];           // per group: parity of the next arrival
    unsigned next;                // next task of this CTA (TaskCursor)
    int abort;                    // a wait gave up
    int job;
};

size_t batch_smem_bytes(const BatchInstance& I, int cluster, int threads) {
    return BatchLayout(I, cluster, threads).total;
}

// A chain group's barrier: a named barrier of its warps, or just the warp for one-warp groups.
__device__ __forceinline__ void group_sync(int bar, int gsize) {
    if (gsize == 32)
        __syncwarp();
    else
        named_barrier(bar, gsize);
}

// ---- asynchronous copies of whole chains between global and shared memory
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned long long* m) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(m)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long* m, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(m)), "r"(parity)
        : "memory");
    return ok != 0u;
}
// One thread: `bytes` (a multiple of 16, both addresses 16-byte aligned) into shared memory,
// completing on m ...
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, unsigned long long* m) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(m)), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(m))
                 : "memory");
}
// ... and out of it, as one bulk group of that thread.
__device__ __forceinline__ void bulk_store(void* dst, const void* src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n\tcp.async.bulk.commit_group;" ::"l"(dst),
                 "r"(smem_u32(src)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void bulk_stores_done() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void fence_async() { asm volatile("fence.proxy.async;" ::: "memory"); }

// Polls ready() until it holds, with a time limit (then the status and sh.abort say so) and back-off;
// false when some wait of this CTA gave up. The whole warp, converged.
template <typename Ready>
__device__ __forceinline__ bool wait_for(BatchShared& sh, Ready ready) {
    unsigned long long start = 0;
    unsigned int nap = 0;
    for (int polls = 0;; ++polls) {
        if (__all_sync(0xFFFFFFFFu, ready())) return true;
        if (polls >= 32) {  // (the clock is read only once the first polls have failed)
            if (polls == 32) start = globaltimer_ns();
            nap = nap ? min(2u * nap, 256u) : 16u;
            __nanosleep(nap);
            if (*(volatile int*)&sh.abort) return false;
            if ((long long)(globaltimer_ns() - start) > sh.limit_ns) {
                if ((threadIdx.x & 31) == 0) {
                    atomicCAS(sh.status, 0, PT_ETIMEDOUT);
                    *(volatile int*)&sh.abort = 1;
                }
                return false;
            }
        }
    }
}

// One sweep of one chain by one group. A function of its own, so that its registers are the
// unit loop's alone and not the task loop's as well (which the call saves once a sweep): with
// both in one body the loop took 117 instructions a unit on N=512, P=64 against 88 in isolation.
struct ChainSweep {
    uint32_t sdesc, items, loff, thr;  // byte offsets in shared memory
    uint32_t buf;
    uint32_t key0, key1, t, rho;
    int n_levels, Lmax, P, gsize, gtid, bar;
};
struct ChainChange {
    int dE, dM, flips;  // this thread's share
};
// The levels of one sweep: unit(item, column) for every item and column g < cols of the
// group's rows, a barrier of the group after each level.
template <typename Offsets, typename Unit>
__device__ __forceinline__ void run_levels(const ChainSweep& c, const uint32_t* s_items, const int32_t* s_loff,
                                           int cols, Offsets offsets, Unit unit) {
    if (c.gsize >= cols) {
        // this thread's column never changes: its row offsets are loop invariants
        const int q_step = c.gsize / cols, q_lane = c.gtid / cols, g = c.gtid - q_lane * cols;
        const bool lane_ok = q_lane < q_step;
        const UnitOffsets off = offsets((uint32_t)g);
        int base = s_loff[0];
        for (int lev = 0; lev < c.n_levels; ++lev) {
            const int end = s_loff[lev + 1];
            if (lane_ok)
                for (int q = base + q_lane; q < end; q += q_step) unit(s_items[q], (uint32_t)g, off);
            base = end;
            group_sync(c.bar, c.gsize);
        }
    } else {
        for (int lev = 0; lev < c.n_levels; ++lev) {
            const int base = s_loff[lev], units = (s_loff[lev + 1] - base) * cols;
            for (int u = c.gtid; u < units; u += c.gsize) {
                const int q = u / cols, g = u - q * cols;
                unit(s_items[base + q], (uint32_t)g, offsets((uint32_t)g));
            }
            group_sync(c.bar, c.gsize);
        }
    }
}
// int8 rows, units of W words of four copies.
template <int DC, int W, bool WIDE>
__device__ __noinline__ ChainChange sweep_chain(const ChainSweep c) {
    extern __shared__ __align__(16) unsigned char smem[];
    int8_t* buf = reinterpret_cast<int8_t*>(smem + c.buf);
    const uint32_t* s_sdesc = reinterpret_cast<const uint32_t*>(smem + c.sdesc);
    const UnitRule<WIDE> rule(c.Lmax);
    const PhiloxKey key = philox_schedule(c.key0, c.key1);
    const uint32_t half = (uint32_t)c.P >> 1, thr = thr_base<WIDE>(c.thr, c.Lmax);
    FlipSums sums;
    sums.clear();
    run_levels(
        c, reinterpret_cast<const uint32_t*>(smem + c.items), reinterpret_cast<const int32_t*>(smem + c.loff),
        c.P / (8 * W), [&](uint32_t g) { return row_offsets<W>(g, half); },
        [&](uint32_t item, uint32_t g, const UnitOffsets& off) {
            const UnitEval<W> e =
                unit_eval<DC, W, false, WIDE>(buf, s_sdesc, item, off, nullptr, c.t, c.rho, W * g, rule, key);
            uint32_t F[W];
            unit_flips<W, false, WIDE>(e, smem, rule, thr, F);
            unit_commit<W>(e, F, sums);
        });
    return ChainChange{sums.dE(rule), sums.dM(rule), sums.flips()};
}
// Bit words of U units.
template <int DC, int U>
__device__ __noinline__ ChainChange sweep_chain_bits(const ChainSweep c) {
    extern __shared__ __align__(16) unsigned char smem[];
    int8_t* buf = reinterpret_cast<int8_t*>(smem + c.buf);
    const uint32_t* s_sdesc = reinterpret_cast<const uint32_t*>(smem + c.sdesc);
    const PhiloxKey key = philox_schedule(c.key0, c.key1);
    const uint32_t S = (uint32_t)IndexRule(c.Lmax).S, kM = (uint32_t)(2 * c.Lmax - 255) * kInv255;
    const uint32_t cols = (uint32_t)c.P / (8 * U);
    BitSums sums;
    sums.clear();
    run_levels(
        c, reinterpret_cast<const uint32_t*>(smem + c.items), reinterpret_cast<const int32_t*>(smem + c.loff),
        (int)cols, [&](uint32_t g) { return word_offsets(g, cols); },
        [&](uint32_t item, uint32_t g, const UnitOffsets& off) {
            bits_unit<DC, DC - 1, U>(buf, s_sdesc, item, off, g, c.t, c.rho, key, smem, S, kM, c.thr, sums);
        });
    return ChainChange{sums.dE(c.Lmax), sums.dM(), sums.flips()};
}
template <int DC>
__device__ __forceinline__ ChainChange sweep_form(const ChainSweep& c, int form, bool wide) {
    if (wide) return sweep_chain<DC, 1, true>(c);
    switch (form) {
        case kFormBits: return sweep_chain_bits<DC, 8>(c);
        case kFormNibbles: return sweep_chain_bits<DC, 4>(c);
        case kFormBytes4: return sweep_chain<DC, 4, false>(c);
        case kFormBytes2: return sweep_chain<DC, 2, false>(c);
        default: return sweep_chain<DC, 1, false>(c);
    }
}

// A chain between its interleaved +-1 bytes in global memory and its form in shared memory.
__device__ void load_chain(const BatchInstance& I, int8_t* buf, const int8_t* src, int tid0, int nthr) {
    if (I.form == kFormBits)
        load_bits<8>(reinterpret_cast<uint32_t*>(buf), src, I.N, I.P >> 6, tid0, nthr);
    else if (I.form == kFormNibbles)
        load_bits<4>(reinterpret_cast<uint32_t*>(buf), src, I.N, I.P >> 5, tid0, nthr);
    else if ((I.P & 15) == 0)
        load_split16(buf, src, I.N, I.P, I.P >> 4, chunk_ginv(I.P >> 4), tid0, nthr);
    else
        load_split(buf, src, I.N, I.P, I.P >> 3, chunk_ginv(I.P >> 3), tid0, nthr);
}
__device__ void store_chain(const BatchInstance& I, int8_t* dst, const int8_t* buf, int tid0, int nthr) {
    if (I.form == kFormBits)
        store_bits<8>(dst, reinterpret_cast<const uint32_t*>(buf), I.N, I.P >> 6, tid0, nthr);
    else if (I.form == kFormNibbles)
        store_bits<4>(dst, reinterpret_cast<const uint32_t*>(buf), I.N, I.P >> 5, tid0, nthr);
    else if ((I.P & 15) == 0)
        store_split16(dst, buf, I.N, I.P, I.P >> 4, chunk_ginv(I.P >> 4), tid0, nthr);
    else
        store_split(dst, buf, I.N, I.P, I.P >> 3, chunk_ginv(I.P >> 3), tid0, nthr);
}

__device__ void run_problem(const BatchInstance& I, unsigned char* smem, BatchShared& sh, cg::cluster_group& cluster,
                            int rank, int K) {
    const int tid = threadIdx.x, nt = blockDim.x;
    const BatchLayout L(I, K, nt);
    uint32_t* s_sdesc = reinterpret_cast<uint32_t*>(smem + L.sdesc);
    uint32_t* s_items = reinterpret_cast<uint32_t*>(smem + L.items);
    int32_t* s_loff = reinterpret_cast<int32_t*>(smem + L.loff);
    int32_t* s_rung = reinterpret_cast<int32_t*>(smem + L.rung);
    int32_t* s_seq = reinterpret_cast<int32_t*>(smem + L.seq);  // sweeps of this run a chain has finished
    long long* s_E = reinterpret_cast<long long*>(smem + L.E);
    long long* s_M = reinterpret_cast<long long*>(smem + L.M);
    uint32_t* s_thr = reinterpret_cast<uint32_t*>(smem + L.thr);
    unsigned char* s_chains = smem + L.chains;
    // [pass mod 4][rung]: (E, M) of the chain on that rung; every CTA's own copy, or one in global memory
    unsigned long long* mail =
        I.mail_smem ? reinterpret_cast<unsigned long long*>(smem + L.mail) : reinterpret_cast<unsigned long long*>(I.mail);

    const int N = I.N, P = I.P, R = I.R;
    const CtaShare share(I, rank, K);
    const int c_begin = share.begin, c_count = share.count;
    const bool in_place = share.in_place;
    const IndexRule index(I.Lmax);
    const int gsize = I.group_threads, ngroups = L.ngroups;
    const int grp = tid / gsize, gtid = tid - grp * gsize;

    // ---- the problem's schedule and descriptors; this CTA's chains
    {
        const int4* src = reinterpret_cast<const int4*>(I.form >= kFormNibbles ? I.wdesc : I.sdesc);
        int4* dst = reinterpret_cast<int4*>(s_sdesc);
        for (int x = tid; x < N * L.DW / 4; x += nt) dst[x] = src[x];
        const uint32_t* g_items = I.form == I.form_t ? I.titems : I.items;
        const int32_t* g_loff = I.form == I.form_t ? I.tlevel_off : I.level_off;
        for (int x = tid; x < 2 * N; x += nt) s_items[x] = g_items[x];
        for (int x = tid; x <= I.n_levels; x += nt) s_loff[x] = g_loff[x];
        for (int x = tid; x < c_count; x += nt) {
            s_rung[x] = I.rung_of_slot[c_begin + x];
            s_seq[x] = 0;
            s_E[x] = I.E[c_begin + x];
            s_M[x] = I.M[c_begin + x];
        }
        if (I.mail_smem || rank == 0)
            for (int x = tid; x < kClusterMailPasses * R * 2; x += nt) mail[x] = 0ull;
        if (I.thr_resident) {  // every rung's row, so a chain never reloads one after a swap
            const int nL = 2 * I.Lmax + 1;
            for (int x = tid; x < R * nL; x += nt) {
                const int r = x / nL, l = x - r * nL;
#pragma unroll
                for (int c = 0; c < 3; ++c) s_thr[(size_t)r * L.thr_words + c * index.S + l] = I.thr[3 * x + c];
            }
        }
        if (in_place)
            for (int lc = 0; lc < c_count; ++lc)
                load_chain(I, reinterpret_cast<int8_t*>(s_chains + (size_t)lc * L.chain_stride),
                           I.spins + (size_t)(c_begin + lc) * I.slot_stride, tid, nt);
        if (tid == 0) sh.next = (unsigned)ngroups;
    }
    __syncthreads();
    if (K > 1) cluster_barrier();  // every mailbox is clear before anyone publishes

    const int bar = 1 + grp;
    uint32_t* thr_g = s_thr + (size_t)grp * L.thr_words;
    int* red_g = reinterpret_cast<int*>(smem + L.red) + (size_t)grp * (gsize / 32) * 3;
    int* ctl_g = reinterpret_cast<int*>(smem + L.ctl) + 4 * grp;
    const int lane = tid & 31, gwarp = gtid >> 5;
    const bool one_warp = gsize == 32, lead = gwarp == 0;
    const int sps = I.sweeps_per_swap;
    const bool keep = share.keep;
    const uint32_t qmod0 = (uint32_t)(I.q0 % kTagPeriod);
    uint32_t phase = grp < 16 ? sh.phase[grp] : 0u;
    bool stored = false;  // lead: a bulk store of the last task's chain (ctl_g) is in flight
    TaskCursor at(grp);   // lead; a group that keeps its chain steps the sweep alone

    auto next_task = [&] {  // lead
        if (keep) {
            ++at.s;
        } else {
            unsigned next = 0;
            if (lane == 0) next = atomicAdd(&sh.next, 1u);
            at.move_to(__shfl_sync(0xFFFFFFFFu, next, 0), c_count);
        }
    };

    for (;;) {
        // ---- the task, its chain's last sweep and that sweep's swap decision
        int s = 0, lc = grp, rung = 0, stop = 0;
        int publish = -1;  // lead: the pass that follows this sweep
        if (grp >= ngroups || c_count == 0 || (keep && grp >= c_count)) break;
        if (lead) {
            s = at.s;
            lc = at.lc;
            stop = s > I.n_sweeps;
            if (!keep) {
                if (stored) {
                    // the chain is back in global memory before its next task may load it
                    if (lane == 0) {
                        bulk_stores_done();
                        fence_async();
                        __threadfence_block();
                        *(volatile int*)&s_seq[ctl_g[1]] = ctl_g[0] + 1;
                    }
                    stored = false;
                }
                if (!stop && s > 0) {
                    volatile int* seq = s_seq + lc;
                    stop = !wait_for(sh, [&] { return *seq >= s; });
                    __threadfence_block();
                }
            }
            int passes = 0, since_pass = 1;  // s = passes * sps + since_pass
            if (sps > 0) {
                passes = s / sps;
                since_pass = s - passes * sps;
                if (since_pass + 1 == sps) publish = passes;
            }
            if (!stop) {
                rung = s_rung[lc];
                if (passes > 0 && since_pass == 0) {
                    // the pass after sweep s - 1
                    const int pass = passes - 1;
                    const long long q = I.q0 + pass;
                    const int rl = (rung & 1) == (int)(q & 1) ? rung : rung - 1;
                    const bool lower = rl == rung;
                    const int partner = lower ? rung + 1 : rl;
                    if (rl >= 0 && rl + 1 < R) {
                        const unsigned long long tag = mbox_tag(qmod0, pass);
                        const unsigned long long* mb =
                            mail + ((size_t)(pass & (kClusterMailPasses - 1)) * R + partner) * 2;
                        unsigned long long wa = 0, wb = 0;
                        const double ca = I.coef[rl], cc = I.coef[(R - 1) + rl];  // (not after the wait)
                        stop = !wait_for(sh, [&] {
                            if (I.mail_smem) {
                                wa = ld_cluster_local_u64(mb);
                                wb = ld_cluster_local_u64(mb + 1);
                            } else {
                                wa = ld_relaxed_u64(mb);
                                wb = ld_relaxed_u64(mb + 1);
                            }
                            return (wa & 0xFFFFFFull) == tag && (wb & 0xFFFFFFull) == tag;
                        });
                        const long long E = s_E[lc], M = s_M[lc];
                        const long long pE = (long long)wa >> 24, pM = (long long)(int32_t)(uint32_t)(wb >> 32);
                        const bool acc = swap_accept_fast(lower ? E : pE, lower ? pE : E, lower ? M : pM,
                                                          lower ? pM : M, ca, cc, (uint32_t)q, (uint32_t)rl,
                                                          philox_schedule(I.key0, I.key1), false);
                        if (!stop) {
                            if (lower && lane < (acc ? 2 : 1)) atomicAdd(I.swap_stats + 2 * rl + lane, 1ull);
                            if (acc) rung = partner;
                        }
                        __syncwarp();
                        if (lane == 0) s_rung[lc] = rung;
                    }
                }
            }
        }
        if (!one_warp) {
            if (lead && lane == 0) {
                ctl_g[0] = s;
                ctl_g[1] = lc;
                ctl_g[2] = rung;
                ctl_g[3] = stop;
            }
            group_sync(bar, gsize);
            s = ctl_g[0];
            lc = ctl_g[1];
            rung = ctl_g[2];
            stop = ctl_g[3];
        } else {
            __syncwarp();
        }
        if (stop) break;
        if (s == I.n_sweeps) {  // only the last pass's decision was left
            if (lead) next_task();
            if (!one_warp) group_sync(bar, gsize);  // everyone has read the group's control words
            continue;
        }

        // ---- the chain, and its rung's thresholds
        const int rho = c_begin + lc;
        int8_t* g_chain = I.spins + (size_t)rho * I.slot_stride;
        int8_t* buf = reinterpret_cast<int8_t*>(s_chains + (size_t)(in_place ? lc : grp) * L.chain_stride);
        const bool bulk_in = !in_place && s > 0;
        if (bulk_in) {
                // the chain in its shared-memory form, as an earlier sweep's bulk store left it
            if (lead && lane == 0) {
                fence_async();
                bulk_load(buf, g_chain, (uint32_t)L.chain_stride, &sh.mbar[grp]);
            }
        } else if (!in_place) {
            load_chain(I, buf, g_chain, gtid, gsize);
        }
        const uint32_t thr_c = (uint32_t)L.thr + 4u * (uint32_t)L.thr_words * (uint32_t)(I.thr_resident ? rung : grp);
        if (!I.thr_resident)
            for (int l = gtid; l <= 2 * I.Lmax; l += gsize)
#pragma unroll
                for (int c = 0; c < 3; ++c) thr_g[c * index.S + l] = I.thr[(size_t)rung * I.nL3 + 3 * l + c];
        if (bulk_in) {
            // (the copy completes by itself; the limit only bounds the wait)
            unsigned long long start = 0;
            while (!mbar_try_wait(&sh.mbar[grp], phase)) {
                if (start == 0) start = globaltimer_ns();
                if ((long long)(globaltimer_ns() - start) > sh.limit_ns) {
                    atomicCAS(sh.status, 0, PT_ETIMEDOUT);
                    *(volatile int*)&sh.abort = 1;
                    break;
                }
            }
            phase ^= 1u;
        }
        group_sync(bar, gsize);

        // ---- sweep s
        const ChainSweep job = {(uint32_t)L.sdesc, (uint32_t)L.items, (uint32_t)L.loff, thr_c,
                                (uint32_t)(L.chains + (size_t)(in_place ? lc : grp) * L.chain_stride),
                                I.key0, I.key1, (uint32_t)(I.t0 + s), (uint32_t)rho, I.n_levels, I.Lmax, P, gsize,
                                gtid, bar};
        const ChainChange ch =
            I.dc == 4 ? sweep_form<4>(job, I.form, index.wide) : sweep_form<8>(job, I.form, index.wide);

        // ---- the chain back (a bulk store takes it in its shared-memory form; the last sweep's
        // is converted again), and the sweep's statistics and publication
        const bool last = s + 1 == I.n_sweeps;
        if (!in_place) {
            if (!last) {
                fence_async();  // this thread's flips, for the copy the lead starts
            } else {
                store_chain(I, g_chain, buf, gtid, gsize);
            }
        }
        int dE = __reduce_add_sync(0xFFFFFFFFu, ch.dE);
        int dM = __reduce_add_sync(0xFFFFFFFFu, ch.dM);
        int nf = __reduce_add_sync(0xFFFFFFFFu, ch.flips);
        if (!one_warp) {
            if (lane == 0) {
                red_g[gwarp * 3 + 0] = dE;
                red_g[gwarp * 3 + 1] = dM;
                red_g[gwarp * 3 + 2] = nf;
            }
            group_sync(bar, gsize);
        } else {
            __syncwarp();
        }
        if (lead) {
            if (!in_place && !last) {
                if (lane == 0) bulk_store(g_chain, buf, (uint32_t)L.chain_stride);
                stored = true;
                if (one_warp && lane == 0) {
                    ctl_g[0] = s;
                    ctl_g[1] = lc;
                }
            }
            if (!one_warp) {
                dE = dM = nf = 0;
                for (int w = 0; w < gsize / 32; ++w) {
                    dE += red_g[w * 3 + 0];
                    dM += red_g[w * 3 + 1];
                    nf += red_g[w * 3 + 2];
                }
            }
            const long long E = s_E[lc] + dE, M = s_M[lc] + dM;
            __syncwarp();
            if (lane == 0) {
                s_E[lc] = E;
                s_M[lc] = M;
            }
            if (publish >= 0 && rung + 1 != I.withhold) {
                const int pass = publish;
                const unsigned long long tag = mbox_tag(qmod0, pass);
                const unsigned long long wa = ((unsigned long long)E << 24) | tag;
                const unsigned long long wb = ((unsigned long long)(uint32_t)(int32_t)M << 32) | tag;
                unsigned long long* slot = mail + ((size_t)(pass & (kClusterMailPasses - 1)) * R + rung) * 2;
                if (I.mail_smem) {
                    if (lane < K) st_cluster_u64x2(slot, (unsigned)lane, wa, wb);
                } else if (lane < 2) {
                    st_relaxed_u64(slot + lane, lane == 0 ? wa : wb);
                }
            }
            if (lane < kAccCount) {
                unsigned long long v = 1ull;
                if (lane == kAccE) v = (unsigned long long)E;
                if (lane == kAccE2) v = (unsigned long long)(E * E);
                if (lane == kAccM) v = (unsigned long long)M;
                if (lane == kAccM2) v = (unsigned long long)(M * M);
                if (lane == kAccFlip) v = (unsigned long long)(long long)nf;
                atomicAdd(I.acc + (size_t)rung * kAccCount + lane, v);
            }
            __syncwarp();
            next_task();  // before the chain is marked (TaskCursor)
            if (!keep && !stored && lane == 0) {  // (a chain being stored is marked when it has arrived)
                __threadfence_block();
                *(volatile int*)&s_seq[lc] = s + 1;
            }
        }
    }
    __syncthreads();
    if (gtid == 0 && grp < ngroups && grp < 16) sh.phase[grp] = phase;

    // ---- write the problem back
    for (int x = tid; x < c_count; x += nt) {
        I.E[c_begin + x] = s_E[x];
        I.M[c_begin + x] = s_M[x];
        I.rung_of_slot[c_begin + x] = s_rung[x];
        I.slot_of_rung[s_rung[x]] = c_begin + x;
    }
    if (in_place)
        for (int lc = 0; lc < c_count; ++lc)
            store_chain(I, I.spins + (size_t)(c_begin + lc) * I.slot_stride,
                        reinterpret_cast<const int8_t*>(s_chains + (size_t)lc * L.chain_stride), tid, nt);
    __syncthreads();
}

__global__ void __launch_bounds__(512, 1) batch_kernel(BatchParams bp) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ BatchShared sh;
    if (threadIdx.x < 16) {
        mbar_init(&sh.mbar[threadIdx.x]);
        sh.phase[threadIdx.x] = 0u;
    }
    if (threadIdx.x == 0) {
        sh.abort = 0;
        sh.limit_ns = bp.timeout_ns;
        sh.status = bp.status;
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async();
    __syncthreads();
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int K = (int)cluster.num_blocks();
    if (bp.single) {
        // one problem on this one cluster; the host keeps its counters
        run_problem(bp.one, smem, sh, cluster, rank, K);
        if (K > 1) cluster.sync();  // peers are done reading this CTA's published (E, M)
        return;
    }
    for (;;) {
        if (rank == 0 && threadIdx.x == 0) sh.job = atomicAdd(bp.next_job, 1);
        cluster.sync();
        const int job = *cluster.map_shared_rank(&sh.job, 0);
        cluster.sync();  // every CTA has read the job before rank 0 may reuse or release sh.job
        if (job >= bp.count) break;
        const BatchInstance I = bp.inst[bp.order[job]];
        run_problem(I, smem, sh, cluster, rank, K);
        cluster.sync();  // peers are done reading this CTA's published (E, M)
        if (rank == 0 && threadIdx.x == 0) {
            // a finished problem's counters advance on the device, so the same launch can be
            // replayed (a CUDA graph) without uploading the problem records again
            BatchInstance* W = bp.inst + bp.order[job];
            W->t0 = I.t0 + I.n_sweeps;
            if (I.sweeps_per_swap > 0) W->q0 = I.q0 + I.n_sweeps / I.sweeps_per_swap;
            if (bp.done) {
                // every CTA of the cluster wrote its chains back before the barrier above;
                // the fence makes those writes visible before the flag, to the host's copies
                __threadfence_system();
                atomicExch(bp.done + bp.order[job], bp.done_token);
            }
        }
    }
}

// Initial spins and (E, M) of every chain of every problem: block b handles chain map[b].
__global__ void batch_init_kernel(const BatchInstance* inst, const int2* map) {
    __shared__ long long red[2][32];
    const int2 m = map[blockIdx.x];
    const BatchInstance& I = inst[m.x];
    const int rho = m.y;
    const PhiloxKey key = philox_schedule(I.key0, I.key1);
    int8_t* sp = I.spins + (size_t)rho * I.slot_stride;
    const int P4 = (I.P + 3) >> 2;
    for (int x = threadIdx.x; x < I.N * P4; x += blockDim.x) {
        const int i = x / P4, g4 = x - i * P4;
        const uint4 u = philox(make_uint4(0u, (uint32_t)i, (uint32_t)rho, (kTagInit << 28) | (uint32_t)g4), key);
        const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int k = 4 * g4 + b;
            if (k < I.P) sp[(size_t)i * I.P + k] = (w[b] >> 31) ? (int8_t)-1 : (int8_t)1;
        }
    }
    if (threadIdx.x == 0) {
        I.rung_of_slot[rho] = rho;
        I.slot_of_rung[rho] = rho;
    }
    __syncthreads();
    // E from the site descriptors: each edge once (neighbour row > own row), h once. The
    // couplings come back out of the multipliers, h out of the constant word (see SiteDesc).
    const int DW = I.dc == 4 ? 8 : 12, NS = I.dc - 1;
    const int zero = IndexRule(I.Lmax).zero();
    long long e = 0, mm = 0;
    for (int x = threadIdx.x; x < I.N * I.P; x += blockDim.x) {
        const int i = x / I.P, k = x - i * I.P;
        const uint32_t* d = I.sdesc + (size_t)i * DW;
        const uint32_t row = I.dc == 4 ? d[7] : d[3];
        const int si = sp[x];
        int f = 0, sumJ = 0;
        for (int sl = 0; sl < NS; ++sl) {
            const int J = I.dc == 4 ? -(int)(d[4 + sl] * 127u)
                                    : (int)(int8_t)((d[1 + (sl >> 2)] >> (8 * (sl & 3))) & 0xFFu);
            const uint32_t off = I.dc == 4 ? d[1 + sl] : d[4 + sl];
            sumJ += J;
            if (off > row) f += J * (int)sp[off + k];
        }
        const uint32_t c = (d[0] - kInv127 * (uint32_t)sumJ * 0x01010101u) & 0xFFu;  // h + sum J + zero
        f += (int)c - sumJ - zero;
        e += (long long)si * f;
        mm += (long long)si * sp[(size_t)i * I.P + ((k + 1 == I.P) ? 0 : k + 1)];
    }
    for (int o = 16; o > 0; o >>= 1) {
        e += __shfl_xor_sync(0xFFFFFFFFu, e, o);
        mm += __shfl_xor_sync(0xFFFFFFFFu, mm, o);
    }
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = e;
        red[1][threadIdx.x >> 5] = mm;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        long long se = 0, sm = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            se += red[0][w];
            sm += red[1][w];
        }
        I.E[rho] = se;
        I.M[rho] = sm;
    }
}

cudaError_t launch_batch(const BatchParams& bp, int cluster, int n_clusters, int threads, size_t smem,
                         cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cluster * n_clusters);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cluster;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    BatchParams p = bp;
    return cudaLaunchKernelEx(&cfg, batch_kernel, p);
}

cudaError_t batch_max_clusters(int cluster, int threads, size_t smem, int* n_clusters) {
    // the limit is a per-function attribute shared by every batch, so it is raised once to
    // the device's opt-in maximum (less this kernel's static shared memory)
    int dev = 0, max_smem = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem - 1024);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(batch_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cluster);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cluster;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaOccupancyMaxActiveClusters(n_clusters, (void*)batch_kernel, &cfg);
}

size_t batch_smem_cap() {
    int dev = 0, max_smem = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return 0;
    return (size_t)max_smem - 1024;  // room for the kernel's static shared memory
}

cudaError_t launch_batch_single(const BatchInstance& I, int cluster, int threads, size_t smem, int* status,
                                long long timeout_ns, cudaStream_t s) {
    BatchParams bp;
    bp.inst = nullptr;
    bp.order = nullptr;
    bp.count = 1;
    bp.next_job = nullptr;
    bp.status = status;
    bp.timeout_ns = timeout_ns;
    bp.single = 1;
    bp.one = I;
    return launch_batch(bp, cluster, 1, threads, smem, s);
}

cudaError_t launch_batch_init(const BatchInstance* inst, const int2* map, int n_chains, cudaStream_t s) {
    batch_init_kernel<<<n_chains, 256, 0, s>>>(inst, map);
    return cudaGetLastError();
}

}  // namespace ptq

// ===================================================================================== host
using namespace ptq;

struct pt_batch {
    int count;
    cudaStream_t stream;
    bool own_stream;
    int cluster, threads, n_clusters;
    size_t smem;
    std::vector<void*> allocs;
    int64_t device_bytes, launches, h2d_bytes;
    BatchInstance* d_inst;
    int32_t* d_order;
    int* d_counter;
    int* d_status;
    long long timeout_ns;
    int8_t* d_staging;
    std::vector<BatchInstance> h_inst;
    std::vector<long long> sweep_limit;
    unsigned char* arena;    // constants [0, const_bytes), then every request's state
    size_t const_bytes, arena_bytes, smem_cap;
    int2* d_map;             // (request, chain) of every chain, for the initial-state kernel
    int n_map;
    int widen;               // group widening of the chosen layout (choose_groups)
    int tuned;               // layouts timed by the autotuner (0 = layout given)
    cudaGraphExec_t exec;    // the captured run (memset of the work counter + persistent launch)
    int graph_failed;        // capture was not possible; runs launch directly
    unsigned char* h_obs;    // pinned staging for pt_batch_read_observables: the device record,
    size_t h_obs_bytes;      // then one request's (E, M, permutation, statistics) block; the
                             // status word follows at h_obs + h_obs_bytes
    int err;
    char msg[256];
};

static thread_local char g_batch_create_msg[256] = "";

// Layouts chosen by the autotuner, per batch shape (every request's sizes, level count and
// sweeps), for the process: a create of a batch of the same shapes reuses the choice and
// times nothing. The layout never changes a result, so reuse is always safe.
struct BatchLayoutChoice {
    int cluster, widen;
};
static std::mutex g_layout_mutex;
static std::map<std::vector<long long>, BatchLayoutChoice> g_layout_cache;

static std::vector<long long> batch_shape_key(const std::vector<BatchInstance>& insts, int threads) {
    std::vector<long long> key;
    key.reserve(insts.size() * 9 + 1);
    key.push_back(threads);
    for (const BatchInstance& I : insts) {
        key.push_back(I.N);
        key.push_back(I.P);
        key.push_back(I.R);
        key.push_back(I.dc);
        key.push_back(I.n_levels);
        key.push_back(I.form_t);  // the forms a chain can take: Lmax decides
        key.push_back(IndexRule(I.Lmax).wide ? 1 : 0);
        key.push_back(I.n_sweeps);
        key.push_back(I.sweeps_per_swap);
    }
    return key;
}

static int bfail(pt_batch* b, int code, const char* fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(b ? b->msg : g_batch_create_msg, 256, fmt, ap);
    va_end(ap);
    if (b && (code == PT_ECUDA || code == PT_ETIMEDOUT)) b->err = code;
    return code;
}

static void free_batch(pt_batch* b) {
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->h_obs) cudaFreeHost(b->h_obs);
    for (void* p : b->allocs) cudaFree(p);
    if (b->own_stream && b->stream) cudaStreamDestroy(b->stream);
    delete b;
}

template <typename T>
static cudaError_t balloc(pt_batch* b, T** ptr, size_t bytes) {
    void* p = nullptr;
    cudaError_t e = cudaMalloc(&p, std::max<size_t>(bytes, 16));
    if (e != cudaSuccess) return e;
    b->allocs.push_back(p);
    b->device_bytes += (int64_t)std::max<size_t>(bytes, 16);
    *ptr = (T*)p;
    return cudaSuccess;
}

// Instructions of a unit, by class of neighbour slots and form (measured whole, per unit-warp).
static const int kFormInstr[2][kFormCount] = {{118, 200, 352, 384, 704}, {134, 228, 400, 448, 816}};

// The form with the least work for a chain that a warp sweeps, and the level schedule balanced
// for it. A wider unit costs less per copy (one descriptor, one address and one load per
// neighbour for more copies), and bit words are a quarter or an eighth of the bytes, so that
// more chains are resident and every warp gets a chain of its own; but a level gives fewer
// units to spread over a warp's lanes. So: the least warp rounds x instructions of a unit,
// times what fewer or wider groups cost when 16 one-warp groups' chains do not fit (measured:
// 1.8 cycles an instruction with 16 one-warp groups, 2.2 with groups of four or eight warps).
static void choose_form(Prepared& pr, const std::vector<std::vector<int>>& adj, int per_round) {
    const int P = pr.P;
    double best = 0.0;
    pr.form = -1;
    int best_round = 1;
    for (int form = 0; form < kFormCount; ++form) {
        const int copies = form_unit_copies(form);
        if (P % (2 * copies)) continue;
        if (form >= kFormNibbles && pr.Lmax > kWordBitsLmax) continue;
        if (form > kFormBytes1 && form < kFormNibbles && IndexRule(pr.Lmax).wide) continue;
        const int cols = P / (2 * copies), per = std::max(1, 32 / cols);
        // balanced levels fill whole rounds, but for the last of about every third level
        const double rounds = std::max(1.0, cols / 32.0) *
                              std::max<double>(pr.n_levels, 2.0 * pr.N / per + 0.35 * pr.n_levels);
        const size_t chain = (size_t)pr.N * form_row_bytes(form, P);
        const size_t fixed = (size_t)pr.N * (pr.dc == 4 ? 40 : 56) + 16384;
        const size_t fit = fixed < 230000 ? (230000 - fixed) / std::max<size_t>(chain, 16) : 0;
        const double spread = fit >= 16 ? 1.0 : (fit >= 10 ? 1.05 : (fit >= 2 ? 1.25 : 1.4));
        const double cost = rounds * kFormInstr[pr.dc == 4 ? 0 : 1][form] * spread;
        if (pr.form < 0 || cost < best) {
            best = cost;
            pr.form = form;
            best_round = per;
        }
    }
    if (pr.form == kFormBytes1 && best_round == per_round) {
        pr.titems = pr.items;
        pr.tlevel_off = pr.level_off;
    } else {
        level_schedule(pr.N, adj, pr.titems, pr.tlevel_off, best_round, (int)(form_row_bytes(pr.form, P) / 4));
    }
}

// Cycles a CTA takes for one sweep of its C chains in a form, by this model: a level of average
// size takes rounds of units on the group; a round takes a warp's latency, 5.5 cycles an
// instruction, or the issue of all the warps at work on a scheduler, 1.65 each; plus 150 cycles
// a level for its loop and barrier, and 4000 a chain and sweep for the task, its statistics
// and the swap decision. (Against 24 measured runs, N = 64 to 512 on clusters of 1 to 8, it is
// off by at most 20 %, and names the faster of the two forms but for near ties.)
static double sweep_cycles(const BatchInstance& I, int C) {
    const int instr = kFormInstr[I.dc == 4 ? 0 : 1][I.form];
    const int cols = I.P / (2 * form_unit_copies(I.form)), g = I.group_threads;
    const double items = 2.0 * I.N / std::max(1, I.n_levels);
    const double per = g >= cols ? g / cols : (double)g / cols;  // items a round
    const double full = std::floor(items / per), rest = std::ceil((items - full * per) * cols / 32.0);
    const int groups = std::min(C, I.n_groups);
    auto round = [&](double warps) { return instr * std::max(5.5, 1.65 * groups * warps / 4.0); };
    const double level = full * round(std::min(g / 32.0, std::ceil(per * cols / 32.0))) + (rest > 0.0 ? round(rest) : 0.0) + 150.0;
    return (I.n_levels * level + 4000.0) * std::max(1.0, (double)C / I.n_groups);
}

double ptq::request_cycles(const BatchInstance& I, int cluster) {
    return (double)I.n_sweeps * sweep_cycles(I, (I.R + cluster - 1) / cluster);
}

int ptq::prepare_request(const pt_request& r, Prepared& pr, char* why, size_t why_len, int per_round) {
    const pt_instance* inst = &r.inst;
    const int N = inst->n, nE = inst->n_edges, P = r.P, R = r.R;
    if (N < 1 || N > 65535 || nE < 0 || !inst->h || (nE > 0 && (!inst->ei || !inst->ej || !inst->J))) {
        snprintf(why, why_len, "bad instance arrays");
        return PT_EINVAL;
    }
    if (P < 8 || P % 8 || P > 4096) {
        snprintf(why, why_len, "batched problems need P %% 8 == 0 and 8 <= P <= 4096");
        return PT_EINVAL;
    }
    if (R < 1 || R > 1024 || !r.ladder) {
        snprintf(why, why_len, "batched problems need 1 <= R <= 1024 rungs");
        return PT_EINVAL;
    }
    if (r.n_sweeps < 0 || r.n_sweeps > (1ll << 30) || r.sweeps_per_swap < 0) {
        snprintf(why, why_len, "n_sweeps must be in [0, 2^30] and sweeps_per_swap >= 0");
        return PT_EINVAL;
    }
    for (int q = 0; q < R; ++q)
        if (!(r.ladder[q].T > 0.0) || !(r.ladder[q].gamma > 0.0) || !std::isfinite(r.ladder[q].T) ||
            !std::isfinite(r.ladder[q].gamma)) {
            snprintf(why, why_len, "rung %d: T and gamma must be finite and > 0", q);
            return PT_EINVAL;
        }
    std::vector<std::vector<int>> adj(N), adjJ(N);
    long long eb = 0;
    for (int b = 0; b < nE; ++b) {
        const int u = inst->ei[b], v = inst->ej[b], J = inst->J[b];
        if (u < 0 || u >= N || v < 0 || v >= N || u == v || J == 0 || J < -127 || J > 127) {
            snprintf(why, why_len, "edge %d invalid", b);
            return PT_EINVAL;
        }
        adj[u].push_back(v);
        adjJ[u].push_back(J);
        adj[v].push_back(u);
        adjJ[v].push_back(J);
        eb += abs(J);
    }
    int dmax = 0, Lmax = 0;
    for (int i = 0; i < N; ++i) {
        std::vector<int> sorted = adj[i];
        std::sort(sorted.begin(), sorted.end());
        if (std::adjacent_find(sorted.begin(), sorted.end()) != sorted.end()) {
            snprintf(why, why_len, "duplicate edge at site %d", i);
            return PT_EINVAL;
        }
        dmax = std::max(dmax, (int)adj[i].size());
        if (inst->h[i] < -127 || inst->h[i] > 127) {
            snprintf(why, why_len, "site %d: h must be in [-127,127]", i);
            return PT_EINVAL;
        }
        int l = abs(inst->h[i]);
        for (int J : adjJ[i]) l += abs(J);
        if (l > 127) {
            snprintf(why, why_len, "site %d: |h| + sum |J| > 127", i);
            return PT_EINVAL;
        }
        Lmax = std::max(Lmax, l);
        eb += abs(inst->h[i]);
    }
    if (dmax + 1 > 8) {
        snprintf(why, why_len, "batched problems need degree <= 7");
        return PT_EINVAL;
    }
    eb *= P;
    const long long mb = (long long)N * P;
    if (eb >= (1ll << 39) || mb >= (1ll << 31)) {
        snprintf(why, why_len, "energy or Trotter sum too large");
        return PT_EINVAL;
    }
    const long long big = std::max(std::max(eb, mb), 1ll);
    pr.sweep_limit = std::min<long long>(big > 3037000499ll ? 0 : 9223372036854775807ll / (big * big), 0xFFFFFFFFll);
    pr.N = N;
    pr.P = P;
    pr.R = R;
    pr.Lmax = Lmax;
    pr.dc = (dmax + 1 <= 4) ? 4 : 8;
    pr.slot_stride = (int)(((size_t)N * P + 15) & ~(size_t)15);
    build_tables(R, P, Lmax, r.ladder, pr.thr, pr.coef);
    if (pr.coef.size() < 2) pr.coef.assign(2, 0.0);
    level_schedule(N, adj, pr.items, pr.level_off, per_round, P / 4);  // rows of P bytes (int8 packed)
    pr.n_levels = (int)pr.level_off.size() - 1;
    choose_form(pr, adj, per_round);
    build_site_desc(N, P, pr.dc, Lmax, adj, adjJ, inst->h, pr.sdesc);
    if (pr.form >= kFormNibbles)
        build_site_desc(N, (int)form_row_bytes(pr.form, P), pr.dc, Lmax, adj, adjJ, inst->h, pr.wdesc, true);
    return PT_OK;
}

// Offsets of one request's data inside a block of its own (constants, then state).
size_t ptq::request_block_layout(Prepared& p, size_t mailbox_entries) {
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t o = off;
        off += (bytes + 255) & ~(size_t)255;
        return o;
    };
    p.off_sdesc = take(p.sdesc.size() * 4);
    p.off_wdesc = take(p.wdesc.size() * 4);
    p.off_items = take(p.items.size() * 4);
    p.off_loff = take(p.level_off.size() * 4);
    p.off_titems = take(p.titems.size() * 4);
    p.off_tloff = take(p.tlevel_off.size() * 4);
    p.off_thr = take(p.thr.size() * 4);
    p.off_coef = take(p.coef.size() * 8);
    p.off_spins = take((size_t)p.R * p.slot_stride);
    p.off_E = take((size_t)p.R * 8);
    p.off_M = take((size_t)p.R * 8);
    p.off_rung = take((size_t)p.R * 4);
    p.off_slot = take((size_t)p.R * 4);
    p.off_acc = take((size_t)p.R * kAccCount * 8);
    p.off_sw = take((size_t)p.R * 16);
    p.off_mbox = take(mailbox_entries * sizeof(Mailbox));
    p.off_inst = take(sizeof(BatchInstance));
    p.off_map = take((size_t)p.R * sizeof(int2));
    p.off_status = take(16);
    return off;
}

void ptq::fill_instance(BatchInstance& I, const Prepared& p, unsigned char* base, const pt_request& r) {
    memset(&I, 0, sizeof(I));
    I.N = p.N;
    I.P = p.P;
    I.R = p.R;
    I.Lmax = p.Lmax;
    I.nL3 = (2 * p.Lmax + 1) * 3;
    I.n_levels = p.n_levels;
    I.dc = p.dc;
    I.form = I.form_t = p.form;
    I.slot_stride = p.slot_stride;
    I.key0 = (uint32_t)(r.seed & 0xFFFFFFFFu);
    I.key1 = (uint32_t)(r.seed >> 32);
    I.n_sweeps = (int)r.n_sweeps;
    I.sweeps_per_swap = r.sweeps_per_swap;
    I.sdesc = (const uint32_t*)(base + p.off_sdesc);
    I.wdesc = (const uint32_t*)(base + p.off_wdesc);
    I.items = (const uint32_t*)(base + p.off_items);
    I.level_off = (const int32_t*)(base + p.off_loff);
    I.titems = (const uint32_t*)(base + p.off_titems);
    I.tlevel_off = (const int32_t*)(base + p.off_tloff);
    I.thr = (const uint32_t*)(base + p.off_thr);
    I.coef = (const double*)(base + p.off_coef);
    I.spins = (int8_t*)(base + p.off_spins);
    I.E = (long long*)(base + p.off_E);
    I.M = (long long*)(base + p.off_M);
    I.rung_of_slot = (int32_t*)(base + p.off_rung);
    I.slot_of_rung = (int32_t*)(base + p.off_slot);
    I.acc = (unsigned long long*)(base + p.off_acc);
    I.swap_stats = (unsigned long long*)(base + p.off_sw);
    I.mail = (Mailbox*)(base + p.off_mbox);
}

// Every rung's threshold row in shared memory when the rows take at most 48 KB and the chains still
// fit; resident chains come first.
static int rows_resident(const BatchInstance& I) {
    return (size_t)I.R * up16((size_t)IndexRule(I.Lmax).row_words() * 4) <= 49152 ? 1 : 0;
}

static void groups_of_form(BatchInstance& I, int cluster, int threads, size_t smem_cap, int widen) {
    // threads per chain: about one 4-copy unit per thread in an average level, at least two
    // warps, and no more groups than a CTA has chains; chains stay resident when they fit.
    // widen > 0 doubles the group that many times (fewer chains at once, shorter levels);
    // widen < 0 halves it (more chains at once, each with more rounds per level), as long as
    // the CTA's chain buffers still fit.
    const long long units = 2ll * I.N * (I.P / 8);
    const long long avg = (units + I.n_levels - 1) / I.n_levels;
    const int C = (I.R + cluster - 1) / cluster;
    // widths are powers of two that divide the CTA, so every thread is in a group
    auto up_ok = [&](int x) {
        const int y = 2 * x;
        return y <= threads && threads % y == 0;
    };
    int g = 64;
    while (up_ok(g) && g < avg) g <<= 1;
    while (up_ok(g) && threads / g > C) g <<= 1;
    for (int w = 0; w < widen && up_ok(g); ++w) g <<= 1;
    for (int w = 0; w < -widen && g > 32; ++w) g >>= 1;  // down to one warp per chain
    while (up_ok(g) && threads / g > C) g <<= 1;         // still no more groups than chains
    while (g > 32 && up_ok(g) && threads / g > 15) g <<= 1;  // named barriers 1..15 (0: the CTA's)
    const int thr_ok = rows_resident(I);
    for (bool ok = false; !ok;) {
        // resident chains come first, then threshold rows, then the swap mailboxes; with chains
        // streamed through one buffer a group, a few groups less than the CTA's warps could
        // form are better than wider ones (at least five eighths of the warps at work)
        I.group_threads = g;
        const int most = threads / g, least = std::max(1, (5 * most + 7) / 8);
        for (int n = most; n >= least && !ok; --n) {
            I.n_groups = n;
            for (int k = n == most ? 0 : 4; k < 8 && !ok; ++k) {
                I.resident = k < 4 ? 1 : 0;
                I.thr_resident = (k & 2) ? 0 : thr_ok;
                I.mail_smem = (k & 1) ? 0 : 1;
                ok = batch_smem_bytes(I, cluster, threads) <= smem_cap;
            }
        }
        if (ok || !up_ok(g)) break;
        g <<= 1;
        while (up_ok(g) && threads / g > 15) g <<= 1;
    }
}

bool ptq::resident_groups(BatchInstance& I, int cluster, int threads, size_t smem_cap, int group_threads, int least) {
    BatchInstance T = I;
    T.group_threads = group_threads;
    T.resident = 1;
    for (int n = threads / group_threads; n >= std::max(1, least); --n) {
        T.n_groups = n;
        for (int k = 0; k < 4; ++k) {
            T.thr_resident = (k & 2) ? 0 : rows_resident(I);
            T.mail_smem = (k & 1) ? 0 : 1;
            if (batch_smem_bytes(T, cluster, threads) <= smem_cap) {
                I = T;
                return true;
            }
        }
    }
    return false;
}

void ptq::choose_groups(BatchInstance& I, int cluster, int threads, size_t smem_cap, int widen) {
    // the form for one-warp groups, or four-copy units where a CTA has few chains and wide
    // groups sweep them
    const int C = (I.R + cluster - 1) / cluster;
    I.form = I.form_t;
    groups_of_form(I, cluster, threads, smem_cap, widen);
    if (I.form_t == kFormBytes1) return;
    BatchInstance F = I;
    F.form = kFormBytes1;
    groups_of_form(F, cluster, threads, smem_cap, widen);
    const bool fits_t = batch_smem_bytes(I, cluster, threads) <= smem_cap;
    const bool fits_f = batch_smem_bytes(F, cluster, threads) <= smem_cap;
    if (fits_f && (!fits_t || sweep_cycles(F, C) < sweep_cycles(I, C))) I = F;
}

// Groups per request, the CTA's shared memory and the persistent grid for one layout.
static int plan_layout(pt_batch* b, int cluster, int widen, char* why, size_t why_len) {
    size_t smem = 0;
    for (int k = 0; k < b->count; ++k) {
        BatchInstance& I = b->h_inst[k];
        choose_groups(I, cluster, b->threads, b->smem_cap, widen);
        const size_t need = batch_smem_bytes(I, cluster, b->threads);
        if (need > b->smem_cap) {
            snprintf(why, why_len, "request %d needs %zu bytes of shared memory per CTA (device: %zu)", k, need,
                     b->smem_cap);
            return PT_EINVAL;
        }
        smem = std::max(smem, need);
    }
    int ncl = 0;
    const cudaError_t e = batch_max_clusters(cluster, b->threads, smem, &ncl);
    if (e != cudaSuccess || ncl < 1) {
        cudaGetLastError();
        snprintf(why, why_len, "no cluster of %d CTAs with %zu bytes of shared memory fits (%s)", cluster, smem,
                 cudaGetErrorString(e));
        return PT_EINVAL;
    }
    b->cluster = cluster;
    b->widen = widen;
    b->smem = smem;
    b->n_clusters = std::min(ncl, b->count);
    return PT_OK;
}

// Every request back to its initial state: zero statistics, counters at 0, initial spins
// and (E, M) from the Philox init stream. Synchronous.
static cudaError_t reset_state(pt_batch* b) {
    for (BatchInstance& I : b->h_inst) I.t0 = I.q0 = 0;
    cudaStream_t s = b->stream;
    cudaError_t e;
    if ((e = cudaMemsetAsync(b->arena + b->const_bytes, 0, b->arena_bytes - b->const_bytes, s)) != cudaSuccess ||
        (e = cudaMemcpyAsync(b->d_inst, b->h_inst.data(), sizeof(BatchInstance) * b->count, cudaMemcpyHostToDevice,
                             s)) != cudaSuccess ||
        (e = cudaMemsetAsync(b->d_status, 0, 16, s)) != cudaSuccess ||
        (e = launch_batch_init(b->d_inst, b->d_map, b->n_map, s)) != cudaSuccess)
        return e;
    b->launches += 1;
    b->h2d_bytes += (int64_t)(sizeof(BatchInstance) * b->count);
    return cudaStreamSynchronize(s);
}

// One run of every request: reset the work counter, then the persistent launch.
static cudaError_t enqueue_run(pt_batch* b) {
    cudaError_t e = cudaMemsetAsync(b->d_counter, 0, sizeof(int), b->stream);
    if (e != cudaSuccess) return e;
    BatchParams bp;
    bp.inst = b->d_inst;
    bp.order = b->d_order;
    bp.count = b->count;
    bp.next_job = b->d_counter;
    bp.status = b->d_status;
    bp.timeout_ns = b->timeout_ns;
    return launch_batch(bp, b->cluster, b->n_clusters, b->threads, b->smem, b->stream);
}

// Layout autotuner: times a short run (1 % of every request's sweeps, at least two) for
// each cluster size and group width that fits and keeps the fastest. The layout changes
// which CTA sweeps which chain and when, never the arithmetic or the random counters, so
// the choice cannot change any result; the state is reset afterwards.
static int autotune(pt_batch* b) {
    static const int kClusters[] = {1, 2, 4, 8};
    std::vector<int> full(b->count), withhold(b->count);
    for (int k = 0; k < b->count; ++k) {
        full[k] = b->h_inst[k].n_sweeps;
        withhold[k] = b->h_inst[k].withhold;
        b->h_inst[k].withhold = 0;
        b->h_inst[k].n_sweeps = std::min(full[k], std::max(2, full[k] / 100));
    }
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaError_t e = cudaEventCreate(&e0);
    if (e == cudaSuccess) e = cudaEventCreate(&e1);
    float best_ms = 0.f;
    int best_c = 0, best_w = 0, timed = 0;
    char why[200];
    std::vector<int> shape, seen;
    // wider groups, then wider clusters, are tried while they are not clearly losing
    bool wider = true;
    for (int ci = 0; ci < 4 && e == cudaSuccess && wider; ++ci) {
        seen.clear();
        float cluster_ms = 0.f;
        for (int w = -4; w < 2 && e == cudaSuccess; ++w) {
            if (plan_layout(b, kClusters[ci], w, why, sizeof(why)) != PT_OK) continue;
            shape.clear();
            for (const BatchInstance& I : b->h_inst) shape.push_back(I.group_threads);
            if (shape == seen) continue;  // the groups of the width before
            seen = shape;
            for (int rep = 0; rep < (timed == 0 ? 2 : 1) && e == cudaSuccess; ++rep) {  // first: one warm-up
                for (BatchInstance& I : b->h_inst) I.t0 = I.q0 = 0;
                if ((e = cudaMemcpyAsync(b->d_inst, b->h_inst.data(), sizeof(BatchInstance) * b->count,
                                         cudaMemcpyHostToDevice, b->stream)) != cudaSuccess ||
                    (e = cudaEventRecord(e0, b->stream)) != cudaSuccess || (e = enqueue_run(b)) != cudaSuccess ||
                    (e = cudaEventRecord(e1, b->stream)) != cudaSuccess || (e = cudaEventSynchronize(e1)) != cudaSuccess)
                    break;
                b->launches += 1;
            }
            float ms = 0.f;
            if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
            if (e != cudaSuccess) break;
            if (timed == 0 || ms < best_ms) {
                best_ms = ms;
                best_c = kClusters[ci];
                best_w = w;
            }
            ++timed;
            if (cluster_ms > 0.f && ms > 1.25f * cluster_ms) break;
            cluster_ms = cluster_ms > 0.f ? std::min(cluster_ms, ms) : ms;
        }
        wider = cluster_ms <= 0.f || cluster_ms <= 1.5f * best_ms;
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    for (int k = 0; k < b->count; ++k) {
        b->h_inst[k].n_sweeps = full[k];
        b->h_inst[k].withhold = withhold[k];
    }
    if (e != cudaSuccess) return bfail(b, PT_ECUDA, "autotuner: %s", cudaGetErrorString(e));
    int st = 0;
    if ((e = cudaMemcpy(&st, b->d_status, sizeof(int), cudaMemcpyDeviceToHost)) != cudaSuccess || st)
        return bfail(b, PT_ECUDA, "autotuner: device status %d (%s)", st, cudaGetErrorString(e));
    if (timed == 0) return bfail(b, PT_EINVAL, "no batched layout fits: %s", why);
    b->tuned = timed;
    const int rc = plan_layout(b, best_c, best_w, why, sizeof(why));
    if (rc) return bfail(b, rc, "%s", why);
    if ((e = reset_state(b)) != cudaSuccess) return bfail(b, PT_ECUDA, "autotuner reset: %s", cudaGetErrorString(e));
    return PT_OK;
}

extern "C" int pt_batch_create(const pt_request* reqs, int32_t count, const pt_options* opt, void* cuda_stream,
                               pt_batch** out) {
    if (!reqs || !out || count < 1) return bfail(nullptr, PT_EINVAL, "need at least one request");
    int dev_count = 0;
    if (cudaGetDeviceCount(&dev_count) != cudaSuccess || dev_count < 1) return bfail(nullptr, PT_ENODEV, "no CUDA device");
    std::vector<Prepared> pr(count);
    char why[200];
    {
        // Requests are prepared independently (checks, tables, level schedule, descriptors),
        // on up to 16 host threads; the first failing request in index order is reported.
        // Levels are balanced for one-warp chain groups (the default and the usual autotuned width).
        std::vector<int> rcs(count, PT_OK);
        std::vector<std::string> whys(count);
        auto work = [&](int first, int step) {
            char w[200];
            for (int k = first; k < count; k += step) {
                rcs[k] = prepare_request(reqs[k], pr[k], w, sizeof(w),
                                         reqs[k].P >= 8 ? std::max(1, 32 / (reqs[k].P / 8)) : 0);
                if (rcs[k]) whys[k] = w;
            }
        };
        const unsigned hw = std::max(1u, std::thread::hardware_concurrency());
        const int n_threads = (int)std::min<unsigned>(std::min(hw, 16u), (unsigned)((count + 7) / 8));
        if (n_threads <= 1) {
            work(0, 1);
        } else {
            std::vector<std::thread> pool;
            pool.reserve(n_threads - 1);
            for (int t = 1; t < n_threads; ++t) pool.emplace_back(work, t, n_threads);
            work(0, n_threads);
            for (std::thread& th : pool) th.join();
        }
        for (int k = 0; k < count; ++k)
            if (rcs[k]) return bfail(nullptr, rcs[k], "request %d: %s", k, whys[k].c_str());
    }
    if (opt && (opt->cluster_size < 0 || opt->cluster_size > 16))
        return bfail(nullptr, PT_EINVAL, "cluster_size must be 0 (autotune) or 1..16");
    pt_batch* b = new pt_batch();
    b->count = count;
    b->stream = (cudaStream_t)cuda_stream;
    b->own_stream = false;
    b->device_bytes = b->launches = b->h2d_bytes = 0;
    b->arena = nullptr;
    b->d_map = nullptr;
    b->exec = nullptr;
    b->graph_failed = 0;
    b->h_obs = nullptr;
    b->h_obs_bytes = 0;
    b->tuned = 0;
    b->widen = 0;
    b->timeout_ns = (opt && opt->wait_timeout_ms > 0 ? opt->wait_timeout_ms : 5000) * 1000000ll;
    b->err = 0;
    b->msg[0] = 0;
    if (!b->stream) {
        if (cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking) != cudaSuccess) {
            delete b;
            return bfail(nullptr, PT_ECUDA, "cudaStreamCreate failed");
        }
        b->own_stream = true;
    }
    int dev = 0, max_smem = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    b->smem_cap = (size_t)max_smem - 1024;  // room for the kernel's static shared memory
    b->threads = 512;

    // device layout of every request in one arena: constants first, then state
    b->h_inst.resize(count);
    b->sweep_limit.resize(count);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t o = off;
        off += (bytes + 255) & ~(size_t)255;
        return o;
    };
    size_t max_state = 0;
    for (int k = 0; k < count; ++k) {
        Prepared& p = pr[k];
        p.off_sdesc = take(p.sdesc.size() * 4);
        p.off_wdesc = take(p.wdesc.size() * 4);
        p.off_items = take(p.items.size() * 4);
        p.off_loff = take(p.level_off.size() * 4);
        p.off_titems = take(p.titems.size() * 4);
        p.off_tloff = take(p.tlevel_off.size() * 4);
        p.off_thr = take(p.thr.size() * 4);
        p.off_coef = take(p.coef.size() * 8);
    }
    const size_t const_bytes = off;
    for (int k = 0; k < count; ++k) {
        Prepared& p = pr[k];
        p.off_spins = take((size_t)p.R * p.slot_stride);
        p.off_E = take((size_t)p.R * 8);
        p.off_M = take((size_t)p.R * 8);
        p.off_rung = take((size_t)p.R * 4);
        p.off_slot = take((size_t)p.R * 4);
        p.off_acc = take((size_t)p.R * kAccCount * 8);
        p.off_sw = take((size_t)p.R * 16);
        p.off_mbox = take((size_t)kClusterMailPasses * p.R * sizeof(Mailbox));
        max_state = std::max(max_state, (size_t)p.R * p.N * p.P);
        BatchInstance& I = b->h_inst[k];
        memset(&I, 0, sizeof(I));
        I.N = p.N;
        I.P = p.P;
        I.R = p.R;
        I.Lmax = p.Lmax;
        I.nL3 = (2 * p.Lmax + 1) * 3;
        I.n_levels = p.n_levels;
        I.dc = p.dc;
        I.form = I.form_t = p.form;
        I.withhold = opt && opt->test_withhold_rung > 0 ? opt->test_withhold_rung : 0;
        I.slot_stride = p.slot_stride;
        I.key0 = (uint32_t)(reqs[k].seed & 0xFFFFFFFFu);
        I.key1 = (uint32_t)(reqs[k].seed >> 32);
        I.n_sweeps = (int)reqs[k].n_sweeps;
        I.sweeps_per_swap = reqs[k].sweeps_per_swap;
        b->sweep_limit[k] = p.sweep_limit;
    }
    b->const_bytes = const_bytes;
    b->arena_bytes = off;
    const int fixed_cluster = (opt && opt->cluster_size > 0) ? opt->cluster_size : 0;
    {
        // the given layout, or (autotuning) the smallest cluster, which needs the most
        // shared memory per CTA: a request that fits nowhere is rejected before allocating
        const int rc = plan_layout(b, fixed_cluster ? fixed_cluster : 1, kGroupWidenDefault, why, sizeof(why));
        if (rc != PT_OK &&
            (fixed_cluster || plan_layout(b, 8, kGroupWidenDefault, why, sizeof(why)) != PT_OK)) {
            free_batch(b);
            return bfail(nullptr, PT_EINVAL, "%s", why);
        }
    }

    unsigned char* arena = nullptr;
    cudaError_t e;
    if ((e = balloc(b, &arena, off)) != cudaSuccess || (e = balloc(b, &b->d_inst, sizeof(BatchInstance) * count)) ||
        (e = balloc(b, &b->d_order, sizeof(int32_t) * count)) || (e = balloc(b, &b->d_counter, 16)) ||
        (e = balloc(b, &b->d_status, 16)) || (e = balloc(b, &b->d_staging, max_state))) {
        free_batch(b);
        return bfail(nullptr, e == cudaErrorMemoryAllocation ? PT_ENOMEM : PT_ECUDA, "cudaMalloc: %s",
                     cudaGetErrorString(e));
    }
    b->arena = arena;
    {
        size_t most = 0;
        for (int k = 0; k < count; ++k) most = std::max(most, pr[k].off_sw + (size_t)pr[k].R * 16 - pr[k].off_E);
        b->h_obs_bytes = (sizeof(BatchInstance) + most + 15) & ~(size_t)15;
        if ((e = cudaMallocHost(&b->h_obs, b->h_obs_bytes + 16)) != cudaSuccess) {  // + the status word
            b->h_obs = nullptr;
            free_batch(b);
            return bfail(nullptr, PT_ENOMEM, "cudaMallocHost: %s", cudaGetErrorString(e));
        }
    }
    std::vector<unsigned char> host_const(const_bytes, 0);
    std::vector<int2> map;
    for (int k = 0; k < count; ++k) {
        Prepared& p = pr[k];
        memcpy(&host_const[p.off_sdesc], p.sdesc.data(), p.sdesc.size() * 4);
        if (!p.wdesc.empty()) memcpy(&host_const[p.off_wdesc], p.wdesc.data(), p.wdesc.size() * 4);
        memcpy(&host_const[p.off_items], p.items.data(), p.items.size() * 4);
        memcpy(&host_const[p.off_loff], p.level_off.data(), p.level_off.size() * 4);
        memcpy(&host_const[p.off_titems], p.titems.data(), p.titems.size() * 4);
        memcpy(&host_const[p.off_tloff], p.tlevel_off.data(), p.tlevel_off.size() * 4);
        memcpy(&host_const[p.off_thr], p.thr.data(), p.thr.size() * 4);
        memcpy(&host_const[p.off_coef], p.coef.data(), p.coef.size() * 8);
        BatchInstance& I = b->h_inst[k];
        I.sdesc = (const uint32_t*)(arena + p.off_sdesc);
        I.wdesc = (const uint32_t*)(arena + p.off_wdesc);
        I.items = (const uint32_t*)(arena + p.off_items);
        I.level_off = (const int32_t*)(arena + p.off_loff);
        I.titems = (const uint32_t*)(arena + p.off_titems);
        I.tlevel_off = (const int32_t*)(arena + p.off_tloff);
        I.thr = (const uint32_t*)(arena + p.off_thr);
        I.coef = (const double*)(arena + p.off_coef);
        I.spins = (int8_t*)(arena + p.off_spins);
        I.E = (long long*)(arena + p.off_E);
        I.M = (long long*)(arena + p.off_M);
        I.rung_of_slot = (int32_t*)(arena + p.off_rung);
        I.slot_of_rung = (int32_t*)(arena + p.off_slot);
        I.acc = (unsigned long long*)(arena + p.off_acc);
        I.swap_stats = (unsigned long long*)(arena + p.off_sw);
        I.mail = (Mailbox*)(arena + p.off_mbox);
        for (int rho = 0; rho < p.R; ++rho) map.push_back(make_int2(k, rho));
    }
    // requests with the most work first, so the last ones to finish are small
    std::vector<int32_t> order(count);
    for (int k = 0; k < count; ++k) order[k] = k;
    std::stable_sort(order.begin(), order.end(), [&](int a, int c) {
        const double wa = (double)pr[a].N * pr[a].P * pr[a].R * (double)reqs[a].n_sweeps;
        const double wc = (double)pr[c].N * pr[c].P * pr[c].R * (double)reqs[c].n_sweeps;
        return wa > wc;
    });
    cudaStream_t s = b->stream;
    b->n_map = (int)map.size();
    if ((e = balloc(b, &b->d_map, map.size() * sizeof(int2))) != cudaSuccess ||
        (e = cudaMemcpyAsync(arena, host_const.data(), const_bytes, cudaMemcpyHostToDevice, s)) != cudaSuccess ||
        (e = cudaMemcpyAsync(b->d_order, order.data(), sizeof(int32_t) * count, cudaMemcpyHostToDevice, s)) !=
            cudaSuccess ||
        (e = cudaMemcpyAsync(b->d_map, map.data(), map.size() * sizeof(int2), cudaMemcpyHostToDevice, s)) !=
            cudaSuccess ||
        (e = reset_state(b)) != cudaSuccess) {
        cudaStreamSynchronize(s);
        free_batch(b);
        return bfail(nullptr, PT_ECUDA, "batch setup: %s", cudaGetErrorString(e));
    }
    b->h2d_bytes += (int64_t)(const_bytes + sizeof(int32_t) * count + map.size() * sizeof(int2));
    if (!fixed_cluster) {
        const std::vector<long long> key = batch_shape_key(b->h_inst, b->threads);
        BatchLayoutChoice cached{0, 0};
        {
            std::lock_guard<std::mutex> lock(g_layout_mutex);
            auto it = g_layout_cache.find(key);
            if (it != g_layout_cache.end()) cached = it->second;
        }
        if (cached.cluster > 0 && plan_layout(b, cached.cluster, cached.widen, why, sizeof(why)) == PT_OK) {
            // the device records carry the layout too (groups, what is resident): the launch's
            // shared memory is sized for this one
            if ((e = cudaMemcpyAsync(b->d_inst, b->h_inst.data(), sizeof(BatchInstance) * count,
                                     cudaMemcpyHostToDevice, s)) != cudaSuccess ||
                (e = cudaStreamSynchronize(s)) != cudaSuccess) {
                free_batch(b);
                return bfail(nullptr, PT_ECUDA, "batch setup: %s", cudaGetErrorString(e));
            }
            b->h2d_bytes += (int64_t)(sizeof(BatchInstance) * count);
            *out = b;
            return PT_OK;
        }
        const int rc = autotune(b);
        if (rc == PT_OK) {
            std::lock_guard<std::mutex> lock(g_layout_mutex);
            g_layout_cache[key] = BatchLayoutChoice{b->cluster, b->widen};
        }
        if (rc != PT_OK) {
            snprintf(g_batch_create_msg, sizeof(g_batch_create_msg), "%s", b->msg);
            free_batch(b);
            return rc;
        }
    }
    *out = b;
    return PT_OK;
}

static int bguard(pt_batch* b) {
    if (!b) return PT_EINVAL;
    return b->err;
}

static int bcheck(pt_batch* b) {
    // the status word through the pinned staging once it exists (a copy into pageable memory
    // is staged by the driver and costs more than the synchronisation itself)
    int local = 0;
    int* st = b->h_obs ? reinterpret_cast<int*>(b->h_obs + b->h_obs_bytes) : &local;
    *st = 0;
    cudaError_t e = cudaMemcpyAsync(st, b->d_status, sizeof(int), cudaMemcpyDeviceToHost, b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return bfail(b, PT_ECUDA, "CUDA error: %s", cudaGetErrorString(e));
    if (*st == PT_ETIMEDOUT) return bfail(b, PT_ETIMEDOUT, "a wait inside the batched kernel timed out");
    if (*st) return bfail(b, PT_ECUDA, "device status %d", *st);
    return PT_OK;
}

extern "C" int pt_batch_run(pt_batch* b) {
    int g = bguard(b);
    if (g) return g;
    for (int k = 0; k < b->count; ++k) {
        const BatchInstance& I = b->h_inst[k];
        const long long passes = I.sweeps_per_swap > 0 ? I.n_sweeps / I.sweeps_per_swap : 0;
        if (I.t0 + I.n_sweeps > b->sweep_limit[k] || I.q0 + passes > 0xFFFFFFFFll)
            return bfail(b, PT_EOVERFLOW, "request %d: sweep or pass counter would overflow", k);
    }
    cudaError_t e = cudaSuccess;
    if (!b->exec && !b->graph_failed) {
        // the first run is captured into a CUDA graph and every run replays it (the problem
        // records on the device carry the counters forward). A stream that is already
        // capturing gets the plain launch, recorded into the caller's own graph.
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(b->stream, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone) {
            cudaGetLastError();
        } else if (cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
            cudaGraph_t graph = nullptr;
            const cudaError_t le = enqueue_run(b);
            const cudaError_t ce = cudaStreamEndCapture(b->stream, &graph);
            if (le == cudaSuccess && ce == cudaSuccess && graph &&
                cudaGraphInstantiate(&b->exec, graph, 0) != cudaSuccess)
                b->exec = nullptr;
            if (graph) cudaGraphDestroy(graph);
            if (!b->exec) {
                b->graph_failed = 1;
                cudaGetLastError();
            }
        } else {
            b->graph_failed = 1;
            cudaGetLastError();
        }
    }
    if (b->exec)
        e = cudaGraphLaunch(b->exec, b->stream);
    else
        e = enqueue_run(b);
    if (e != cudaSuccess) return bfail(b, PT_ECUDA, "batch launch: %s", cudaGetErrorString(e));
    b->launches += 1;
    for (int k = 0; k < b->count; ++k) {
        BatchInstance& I = b->h_inst[k];
        I.t0 += I.n_sweeps;
        if (I.sweeps_per_swap > 0) I.q0 += I.n_sweeps / I.sweeps_per_swap;
    }
    return PT_OK;
}

extern "C" int pt_batch_sync(pt_batch* b) {
    int g = bguard(b);
    if (g) return g;
    return bcheck(b);
}

extern "C" int pt_batch_read_state(pt_batch* b, int32_t index, int8_t* out, size_t bytes) {
    int g = bguard(b);
    if (g) return g;
    if (index < 0 || index >= b->count) return bfail(b, PT_EINVAL, "index out of range");
    const BatchInstance& I = b->h_inst[index];
    const size_t need = (size_t)I.R * I.N * I.P;
    if (!out || bytes < need) return bfail(b, PT_EINVAL, "state buffer needs %zu bytes", need);
    DevProblem p;
    memset(&p, 0, sizeof(p));
    p.spins = I.spins;
    p.slot_of_rung = I.slot_of_rung;
    p.N = I.N;
    p.P = I.P;
    p.R = I.R;
    p.slot_stride = I.slot_stride;
    cudaError_t e;
    if ((e = launch_gather_state(p, b->d_staging, b->stream)) != cudaSuccess ||
        (e = cudaMemcpyAsync(out, b->d_staging, need, cudaMemcpyDeviceToHost, b->stream)) != cudaSuccess)
        return bfail(b, PT_ECUDA, "%s", cudaGetErrorString(e));
    b->launches += 1;
    return bcheck(b);
}

extern "C" int pt_batch_read_observables(pt_batch* b, int32_t index, pt_observables* o) {
    int g = bguard(b);
    if (g) return g;
    if (index < 0 || index >= b->count || !o) return bfail(b, PT_EINVAL, "bad index or null observables");
    const BatchInstance& I = b->h_inst[index];
    const int R = I.R;
    // the device record (its counters also count replays of a caller's graph), then the
    // request's state block from E to the swap counts (contiguous in the arena), in two copies
    // into pinned staging
    const unsigned char* blk = reinterpret_cast<const unsigned char*>(I.E);
    const size_t blk_bytes =
        (size_t)(reinterpret_cast<const unsigned char*>(I.swap_stats) - blk) + (size_t)R * 16;
    unsigned char* h_blk = b->h_obs + sizeof(BatchInstance);
    cudaStream_t s = b->stream;
    cudaError_t e;
    if ((e = cudaMemcpyAsync(b->h_obs, b->d_inst + index, sizeof(BatchInstance), cudaMemcpyDeviceToHost, s)) !=
            cudaSuccess ||
        (e = cudaMemcpyAsync(h_blk, blk, blk_bytes, cudaMemcpyDeviceToHost, s)) != cudaSuccess)
        return bfail(b, PT_ECUDA, "%s", cudaGetErrorString(e));
    int rc = bcheck(b);
    if (rc) return rc;
    BatchInstance dev_rec;
    memcpy(&dev_rec, b->h_obs, sizeof(BatchInstance));
    auto at = [&](const void* dev) { return h_blk + (reinterpret_cast<const unsigned char*>(dev) - blk); };
    const long long* E = reinterpret_cast<const long long*>(at(I.E));
    const long long* M = reinterpret_cast<const long long*>(at(I.M));
    const int32_t* slot_of = reinterpret_cast<const int32_t*>(at(I.slot_of_rung));
    const unsigned long long* acc = reinterpret_cast<const unsigned long long*>(at(I.acc));
    const unsigned long long* sw = reinterpret_cast<const unsigned long long*>(at(I.swap_stats));
    o->t = dev_rec.t0;
    o->q = dev_rec.q0;
    for (int r = 0; r < R; ++r) {
        const int slot = slot_of[r];
        if (o->E) o->E[r] = E[slot];
        if (o->M) o->M[r] = M[slot];
        const unsigned long long* a = &acc[(size_t)r * kAccCount];
        if (o->n_meas) o->n_meas[r] = (int64_t)a[kAccN];
        if (o->sum_E) o->sum_E[r] = (int64_t)a[kAccE];
        if (o->sum_E2) o->sum_E2[r] = (int64_t)a[kAccE2];
        if (o->sum_M) o->sum_M[r] = (int64_t)a[kAccM];
        if (o->sum_M2) o->sum_M2[r] = (int64_t)a[kAccM2];
        if (o->flip_acc) o->flip_acc[r] = (int64_t)a[kAccFlip];
        if (o->replica_at) o->replica_at[r] = slot;
    }
    for (int r = 0; r + 1 < R; ++r) {
        if (o->swap_att) o->swap_att[r] = (int64_t)sw[2 * r];
        if (o->swap_acc) o->swap_acc[r] = (int64_t)sw[2 * r + 1];
    }
    return PT_OK;
}

extern "C" int pt_batch_get_info(const pt_batch* b, pt_batch_info* o) {
    if (!b || !o) return PT_EINVAL;
    o->count = b->count;
    o->cluster = b->cluster;
    o->n_clusters = b->n_clusters;
    o->threads_per_block = b->threads;
    o->smem_bytes = (int64_t)b->smem;
    o->device_bytes = b->device_bytes;
    o->kernel_launches = b->launches;
    o->h2d_bytes = b->h2d_bytes;
    o->tuned_layouts = b->tuned;
    o->group_widen = b->widen;
    o->graph = b->exec ? 1 : 0;
    o->reserved = 0;
    return PT_OK;
}

extern "C" int pt_batch_destroy(pt_batch* b) {
    if (!b) return PT_OK;
    cudaStreamSynchronize(b->stream);
    free_batch(b);
    return PT_OK;
}

extern "C" const char* pt_batch_last_error(const pt_batch* b) { return b ? b->msg : g_batch_create_msg; }
