// pt_kernels.cu -- sm_103a kernels of the PT-QMC hot path.
//
// Sweep (Sec. 2 Metropolis sweeps; Sec. 5 "two groups of independent regions", swept one
// after the other with a barrier between them): one CTA owns one chain (replica) for the
// whole launch, with its spins, the instance and the chain's current Metropolis table in
// shared memory. The sequential order (sites in index order, even copies then odd copies)
// is replayed exactly by a static level schedule computed on the host: update (i, p)
// (site i, copy parity p, all P/2 copies of that parity) must follow (i, 0) when p = 1
// and (j, p) for every neighbour j < i; updates in one level touch disjoint spins, so
// running a level in parallel and putting a CTA barrier between levels reproduces the
// sequential result bit for bit. Random numbers are a pure function of the counter
// (Philox4x32-10), so the thread layout does not change any result.
//
// Swap (Sec. 2: neighbouring chains, disjoint pairs): inside a cooperative launch each
// chain publishes (E, M) for pass q in a per-(pass, rung) mailbox and waits, with a time
// limit, only for its pair partner; both partners evaluate the same decision.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "pt.h"
#include "pt_device.cuh"
#include "pt_internal.h"

namespace ptq {

namespace cg = cooperative_groups;

// ------------------------------------------------------------------------- smem layouts

// Threshold rows (of row_words entries) and per-rung statistics in shared memory (when they fit).
__host__ __device__ inline size_t thr_bytes(const DevProblem& p, int row_words) {
    return up16((size_t)(p.tables_in_smem ? p.R : 1) * row_words * 4);
}
__host__ __device__ inline size_t acc_bytes(const DevProblem& p) {
    return p.acc_in_smem ? (size_t)p.R * kAccCount * 8 : 0;
}

// Byte-wise path (any even P, any degree up to 32).
struct GenericLayout {
    size_t spins, nbr, h, items, loff, thr, acc, red, ctl, total;
    __host__ __device__ explicit GenericLayout(const DevProblem& p) {
        const int N = p.N, P = p.P;
        size_t o = 0;
        spins = o; o += up16((size_t)N * P);
        nbr = o;   o += up16((size_t)N * p.dmax * 4);
        h = o;     o += up16((size_t)N);
        items = o; o += up16((size_t)2 * N * 4);
        loff = o;  o += up16((size_t)(p.n_levels + 1) * 4);
        thr = o;   o += thr_bytes(p, p.nL3);
        acc = o;   o += acc_bytes(p);
        red = o;   o += 32 * 3 * 8;
        ctl = o;   o += 16;
        total = o;
    }
};

// Path 1's word-wise kernel (any even P, any degree up to 32): rows whose parity halves are
// padded to whole words, and descriptors built in shared memory from the neighbour table.
// With pre and cswap as FastLayout has them, for the one-copy-a-thread kernels.
struct RowsLayout {
    size_t spins, desc, items, loff, thr, acc, red, ctl, cmb, rbuf, total;
    __host__ __device__ explicit RowsLayout(const DevProblem& p, bool pre = false, bool cswap = false) {
        const size_t N = p.N, G = ((size_t)p.P / 2 + 3) / 4;
        size_t o = 0;
        spins = o; o += up16(N * 8 * G);
        desc = o;  o += (p.records ? 2 * N : N) * rows_desc_words(p.slots) * 4;
        items = o; o += up16(2 * N * 4);
        loff = o;  o += up16((size_t)(p.n_levels + 1) * 4);
        thr = o;   o += thr_bytes(p, IndexRule(p.Lmax).row_words());
        acc = o;   o += acc_bytes(p);
        red = o;   o += 16;  // the sweep's three sums
        ctl = o;   o += 32;
        cmb = o;   o += cswap ? (size_t)kClusterMailPasses * p.R * 16 : 0;
        rbuf = o;  o += pre ? 2 * (2 * N) * G * 16 : 0;
        total = o;
    }
};

size_t copy_smem_bytes(const DevProblem& p, bool cluster) { return RowsLayout(p, true, cluster).total; }

// Packed path (P % 8 == 0, degree <= 7): spins, per-site descriptors, the schedule, level
// offsets, the threshold row(s), statistics, reduction scratch, control words and, when
// the random words are produced ahead, two buffers of one sweep's words each.
// With bits, the chain is P/8 bytes per site and two 256-entry tables spread parity bits
// into +1/-1 bytes.
// With cswap (path 9), each CTA also holds the swap mailboxes of the cluster's chains: four
// passes of R (E, M) words each (see eos_decide_cluster).
struct FastLayout {
    size_t spins, lut, desc, items, loff, thr, acc, red, ctl, cmb, rbuf, total;
    __host__ __device__ FastLayout(const DevProblem& p, int dc, bool pre, bool bits = false, bool cswap = false) {
        const int N = p.N, P = p.P;
        const size_t row = bits ? (size_t)P / (p.nibble ? 4 : 8) : (size_t)P;
        size_t o = 0;
        spins = o; o += up16((size_t)N * row);
        lut = o;   o += bits && !p.nibble ? 2048 : 0;
        desc = o;  o += p.records && !bits ? (size_t)2 * N * record_words(dc) * 4 : (size_t)N * (dc == 4 ? 32 : 48);
        items = o; o += up16((size_t)2 * N * 4);
        loff = o;  o += up16((size_t)(p.n_levels + 1) * 4);
        thr = o;   o += thr_bytes(p, IndexRule(p.Lmax).row_words());
        acc = o;   o += acc_bytes(p);
        red = o;   o += 16;  // the sweep's three sums
        ctl = o;   o += 32;
        cmb = o;   o += cswap ? (size_t)kClusterMailPasses * p.R * 16 : 0;
        rbuf = o;
        if (pre) o += (size_t)2 * (p.n_chunks > 1 ? p.chunk_items : 2 * N) * (P / 8) * 16;
        total = o;
    }
};

size_t split_smem_bytes(const DevProblem& p, int dclass, bool pre);

int rows_slots(const DevProblem& p, int max_degree, size_t max_smem) {
    if (p.P < 2) return 0;
    DevProblem q = p;
    q.slots = std::max(4, (max_degree + 3) / 4 * 4);
    q.tables_in_smem = q.acc_in_smem = 0;
    q.n_levels = std::max(p.n_levels, 1);
    return RowsLayout(q).total <= max_smem ? q.slots : 0;
}

size_t sweep_smem_bytes(const DevProblem& p, int path, int dclass, bool cluster_pre) {
    if (path == kPathGeneric) return p.slots > 0 ? RowsLayout(p).total : GenericLayout(p).total;
    if (path == kPathCluster) return FastLayout(p, dclass, cluster_pre, false, true).total;
    if (path == kPathPeer) return FastLayout(p, dclass, true, false).total;
    if (path == kPathSplit || path == kPathSplitInline) return split_smem_bytes(p, dclass, path == kPathSplit);
    return FastLayout(p, dclass, path == kPathPacked, path == kPathBits).total;
}


// ------------------------------------------------------------------------- end of a sweep
// The other rung of `rung`'s pair in pass q, or -1.
__device__ __forceinline__ int pair_rung(int rung, long long q, int R) {
    const int other = (rung & 1) == (int)(q & 1) ? rung + 1 : rung - 1;
    return other >= 0 && other < R ? other : -1;
}

// A chain's side of the swap pass that follows a sweep: rl is the lower rung of its pair,
// partner the other rung; active = 0 when no pass follows or the chain has no partner.
struct SwapSide {
    int active, rl, partner, pass;
    long long q;
    unsigned long long tag;
};

// Thread 0 of a chain's CTA, after the sweep's changes are reduced: update E and M, add the
// statistics of the rung the chain sits on (to `acc`, shared or global) and, when a swap
// pass follows this sweep, publish (E, M) in the pass's mailbox. Does not wait.
// pass >= 0: a swap pass with this index (within the launch) follows the sweep.
// write = false: a CTA that shares the chain with the one that publishes (split kernel).
__device__ SwapSide eos_publish(const DevProblem& p, int rung, long long& E, long long& M, long long dE,
                                long long dM, int pass, long long q0, uint32_t qmod0, bool write = true) {
    E += dE;
    M += dM;
    SwapSide w;
    w.active = w.pass = 0;
    if (pass >= 0) {
        const int R = p.R;
        w.pass = pass;
        w.q = q0 + w.pass;
        w.tag = mbox_tag(qmod0, w.pass);
        Mailbox* mb = p.mbox + (size_t)w.pass * R;
        if (write && rung != p.withhold_rung) {
            st_relaxed_u64(&mb[rung].a, ((unsigned long long)E << 24) | w.tag);
            st_relaxed_u64(&mb[rung].b, ((unsigned long long)(uint32_t)(int32_t)M << 32) | w.tag);
        }
        if ((rung & 1) == (int)(w.q & 1)) {
            w.rl = rung;
            w.partner = rung + 1;
        } else {
            w.rl = rung - 1;
            w.partner = rung - 1;
        }
        w.active = (w.rl >= 0 && w.rl + 1 < R) ? 1 : 0;
    }
    return w;
}

static_assert(kAccN == 0 && kAccE == 1 && kAccE2 == 2 && kAccM == 3 && kAccM2 == 4 && kAccFlip == 5 && kAccCount == 6,
              "eos_stats pairs the counters in this order");

// Thread 0: the statistics of the rung the chain sat on during the sweep (to `acc`, shared or
// global), from the updated E and M.
__device__ __forceinline__ void eos_stats(const DevProblem& p, unsigned long long* acc, int rung, long long E,
                                          long long M, long long nflip) {
    unsigned long long* a = acc + (size_t)rung * kAccCount;
    if (p.acc_in_smem) {
        // the rung's six counters (48 bytes, 16-byte aligned) in three paired loads and stores
        ulonglong2* a2 = reinterpret_cast<ulonglong2*>(a);
        ulonglong2 v0 = a2[0], v1 = a2[1], v2 = a2[2];
        v0.x += 1ull;                                // kAccN
        v0.y += (unsigned long long)E;               // kAccE
        v1.x += (unsigned long long)(E * E);         // kAccE2
        v1.y += (unsigned long long)M;               // kAccM
        v2.x += (unsigned long long)(M * M);         // kAccM2
        v2.y += (unsigned long long)nflip;           // kAccFlip
        a2[0] = v0;
        a2[1] = v1;
        a2[2] = v2;
    } else {
        atomicAdd(a + kAccN, 1ull);
        atomicAdd(a + kAccE, (unsigned long long)E);
        atomicAdd(a + kAccE2, (unsigned long long)(E * E));
        atomicAdd(a + kAccM, (unsigned long long)M);
        atomicAdd(a + kAccM2, (unsigned long long)(M * M));
        atomicAdd(a + kAccFlip, (unsigned long long)nflip);
    }
}

// One thread, or a warp whose lanes all follow E and M (count in one of them): wait for the
// partner's mailbox (bounded by timeout_ns) and take the decision both chains of the pair take. Returns the chain's rung for the next sweep; sets *abort when
// the partner's mailbox never arrived within the time limit. read(partner, wa, wb) loads the
// partner's two tagged words. The pass's coefficients and random word do not depend on the
// partner and are fetched before the wait, as is nothing but the loads and the comparison
// after it; the clock is read only once the first polls have failed. count = false: the
// pair's attempt and acceptance are counted by another CTA of the chain (split kernel).
template <typename Read>
__device__ __forceinline__ int eos_decide_from(const DevProblem& p, const SwapSide& w, int rung, long long E,
                                               long long M, long long timeout_ns, const PhiloxKey& key, int* abort,
                                               bool count, Read read) {
    *abort = 0;
    if (!w.active) return rung;
    const int R = p.R, rl = w.rl;
    const bool lower = (rung == rl);
    const double ca = p.coef[rl], cc = p.coef[(R - 1) + rl];
    const uint32_t word = swap_word((uint32_t)w.q, (uint32_t)rl, key);
    unsigned long long wa, wb, start = 0;
    // the first polls spin (the partner usually publishes within a round trip); later ones back
    // off with __nanosleep, doubling up to 256 ns, so that a CTA waiting on a slow partner
    // leaves its issue slots and the L2 to the CTAs sharing its SM
    unsigned int nap = 0;
    for (int polls = 0;; ++polls) {
        read(w.partner, wa, wb);
        if ((wa & 0xFFFFFFull) == w.tag && (wb & 0xFFFFFFull) == w.tag) break;
        if (polls >= 32) {
            if (polls == 32) start = globaltimer_ns();
            if ((long long)(globaltimer_ns() - start) > timeout_ns) {
                atomicCAS(p.status, 0, PT_ETIMEDOUT);
                *abort = 1;
                return rung;
            }
            nap = nap ? min(2u * nap, 256u) : 16u;
            __nanosleep(nap);
        }
    }
    const long long pE = (long long)wa >> 24, pM = (long long)(int32_t)(uint32_t)(wb >> 32);
    const bool acc_swap =
        swap_accept_fast_by(lower ? E : pE, lower ? pE : E, lower ? M : pM, lower ? pM : M, ca, cc,
                            [&] { return word; }, p.exact_swaps != 0);
    if (lower && count) {
        atomicAdd(p.swap_stats + 2 * rl, 1ull);
        if (acc_swap) atomicAdd(p.swap_stats + 2 * rl + 1, 1ull);
    }
    return acc_swap ? w.partner : rung;
}
__device__ __forceinline__ int eos_decide(const DevProblem& p, const SwapSide& w, int rung, long long E, long long M,
                                          long long timeout_ns, const PhiloxKey& key, int* abort, bool count = true) {
    const Mailbox* mb = p.mbox + (size_t)w.pass * p.R;
    return eos_decide_from(p, w, rung, E, M, timeout_ns, key, abort, count,
                           [&](int partner, unsigned long long& wa, unsigned long long& wb) {
                               wa = ld_relaxed_u64(&mb[partner].a);
                               wb = ld_relaxed_u64(&mb[partner].b);
                           });
}

// Path 9 (one cluster holds every chain): the same decision with the partner's (E, M) read
// from this CTA's own copy of the cluster mailboxes. Every chain that publishes for a pass
// writes its two tagged words into every CTA of the cluster, at [pass mod 4][rung], so the
// wait polls local shared memory. Four slots suffice: the chain that would overwrite the
// slot a waiting chain reads (the holder of that rung three passes later) must first finish
// the pass two later, in which it waits for the reader's own publication again.
__device__ __forceinline__ int eos_decide_cluster(const DevProblem& p, const unsigned long long* s_cmb,
                                                  const SwapSide& w, int rung, long long E, long long M,
                                                  long long timeout_ns, const PhiloxKey& key, int* abort,
                                                  bool count = true) {
    const unsigned long long* mb = s_cmb + (size_t)(w.pass & (kClusterMailPasses - 1)) * p.R * 2;
    return eos_decide_from(p, w, rung, E, M, timeout_ns, key, abort, count,
                           [&](int partner, unsigned long long& wa, unsigned long long& wb) {
                               wa = ld_cluster_local_u64(mb + 2 * partner);
                               wb = ld_cluster_local_u64(mb + 2 * partner + 1);
                           });
}

// Both steps at once (the byte-wise kernel).
__device__ int end_of_sweep(const DevProblem& p, unsigned long long* acc, int rung, long long& E, long long& M,
                            long long dE, long long dM, long long nflip, int s, long long q0, int sweeps_per_swap,
                            long long timeout_ns, const PhiloxKey& key, int* abort) {
    const int pass = (sweeps_per_swap > 0 && (s + 1) % sweeps_per_swap == 0) ? (s + 1) / sweeps_per_swap - 1 : -1;
    const SwapSide w = eos_publish(p, rung, E, M, dE, dM, pass, q0, (uint32_t)(q0 % kTagPeriod));
    eos_stats(p, acc, rung, E, M, nflip);
    return eos_decide(p, w, rung, E, M, timeout_ns, key, abort);
}

// Programmatic dependent launch (LaunchPlan::overlap). A kernel first does what no earlier kernel
// of the context writes (tables, schedule, records, random words); after wait_for_earlier_kernels
// everything before it in the stream is complete and visible. allow_next_kernel lets the next
// one's blocks start as soon as all of this kernel's have got there. Both do nothing in a launch
// without the attribute.
__device__ __forceinline__ void wait_for_earlier_kernels() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void allow_next_kernel() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Shared-memory threshold rows: every rung's row when they fit, else the current one. The
// byte-wise kernels keep the public layout ...
__device__ __forceinline__ void load_thr(const DevProblem& p, uint32_t* s_thr, int rung, int tid, int nt) {
    if (p.tables_in_smem) {
        for (int x = tid; x < p.R * p.nL3; x += nt) s_thr[x] = p.thr[x];
    } else {
        for (int x = tid; x < p.nL3; x += nt) s_thr[x] = p.thr[(size_t)rung * p.nL3 + x];
    }
}
__device__ __forceinline__ const uint32_t* thr_row(const DevProblem& p, const uint32_t* s_thr, int rung) {
    return p.tables_in_smem ? s_thr + (size_t)rung * p.nL3 : s_thr;
}
// ... and the packed ones rearrange it into columns (see IndexRule).
__device__ __forceinline__ void load_thr_columns(const DevProblem& p, uint32_t* s_thr, int rung, int tid, int nt) {
    const IndexRule rule(p.Lmax);
    const uint32_t* src = p.tables_in_smem ? p.thr : p.thr + (size_t)rung * p.nL3;
    const int rows = p.tables_in_smem ? p.R : 1, nL = 2 * p.Lmax + 1;
    for (int x = tid; x < rows * nL; x += nt) {
        const int r = x / nL, l = x - r * nL;
        uint32_t* dst = s_thr + (size_t)r * rule.row_words() + l;
#pragma unroll
        for (int c = 0; c < 3; ++c) dst[c * rule.S] = src[3 * x + c];
    }
}

// Per-launch statistics gathered in shared memory are added to the global rows once.
__device__ __forceinline__ void flush_acc(const DevProblem& p, const unsigned long long* s_acc, int tid, int nt) {
    if (!p.acc_in_smem) return;
    for (int x = tid; x < p.R * kAccCount; x += nt)
        if (s_acc[x]) atomicAdd(p.acc + x, s_acc[x]);
}

// ------------------------------------------------------------------------- generic sweep
// One CTA per chain (slot); byte-wise spins, Philox inline in each 4-copy unit. Used for P = 1
// and where the word-wise kernel's layout does not fit; other shapes
// that the packed kernels refuse run word-wise (sweep_rows_kernel, sweep_copy_kernel).
template <int DCLASS>
__global__ void __launch_bounds__(512, 1)
sweep_kernel(DevProblem p, long long t0, long long q0, int n_sweeps, int sweeps_per_swap,
             long long timeout_ns, int n_consumer) {
    extern __shared__ __align__(16) unsigned char smem[];
    wait_for_earlier_kernels();
    allow_next_kernel();
    const int N = p.N, P = p.P;
    const int tid = threadIdx.x, nt = blockDim.x;
    const int slot = blockIdx.x;
    const GenericLayout L(p);
    int8_t* sp = reinterpret_cast<int8_t*>(smem + L.spins);
    uint32_t* s_nbr = reinterpret_cast<uint32_t*>(smem + L.nbr);
    int8_t* s_h = reinterpret_cast<int8_t*>(smem + L.h);
    uint32_t* s_items = reinterpret_cast<uint32_t*>(smem + L.items);
    int32_t* s_loff = reinterpret_cast<int32_t*>(smem + L.loff);
    uint32_t* s_thr = reinterpret_cast<uint32_t*>(smem + L.thr);
    long long* s_red = reinterpret_cast<long long*>(smem + L.red);
    int* s_ctl = reinterpret_cast<int*>(smem + L.ctl);
    unsigned long long* s_acc = reinterpret_cast<unsigned long long*>(smem + L.acc);
    (void)n_consumer;

    {
        const int4* src = reinterpret_cast<const int4*>(p.spins + (size_t)slot * p.slot_stride);
        int4* dst = reinterpret_cast<int4*>(sp);
        const int n16 = (int)(up16((size_t)N * P) / 16);
        for (int x = tid; x < n16; x += nt) dst[x] = src[x];
        for (int x = tid; x < N * DCLASS; x += nt) s_nbr[x] = p.nbr[x];
        for (int x = tid; x < N; x += nt) s_h[x] = p.h[x];
        for (int x = tid; x < 2 * N; x += nt) s_items[x] = p.items[x];
        for (int x = tid; x <= p.n_levels; x += nt) s_loff[x] = p.level_off[x];
    }
    int rung = p.rung_of_slot[slot];
    load_thr(p, s_thr, rung, tid, nt);
    if (p.acc_in_smem)
        for (int x = tid; x < p.R * kAccCount; x += nt) s_acc[x] = 0ull;
    long long E = p.E[slot], M = p.M[slot];  // meaningful in thread 0 only
    __syncthreads();
    const uint32_t* thr = thr_row(p, s_thr, rung);

    const PhiloxKey key = philox_schedule(p.key0, p.key1);
    const int G = (((P + 1) >> 1) + 3) >> 2;  // 4-copy groups per parity (P = 1: one even copy)
    int lg = 0;
    while ((1 << lg) < G) ++lg;
    const int gmask = (1 << lg) - 1;
    const int Lmax = p.Lmax;
    const int lane = tid & 31, warp = tid >> 5, nwarps = (nt + 31) >> 5;

    for (int s = 0; s < n_sweeps; ++s) {
        const uint32_t t = (uint32_t)(t0 + s);
        int dE = 0, dM = 0, nf = 0;
        for (int lev = 0; lev < p.n_levels; ++lev) {
            const int base = s_loff[lev];
            const int units = (s_loff[lev + 1] - base) << lg;
            for (int u = tid; u < units; u += nt) {
                const int g = u & gmask;
                if (g >= G) continue;
                const uint32_t it = s_items[base + (u >> lg)];
                const int i = (int)(it >> 1), par = (int)(it & 1u);
                const uint4 r4 = philox(make_uint4(t, (uint32_t)i, (uint32_t)slot,
                                                   ((uint32_t)par << 24) | (uint32_t)g), key);
                const uint32_t rw[4] = {r4.x, r4.y, r4.z, r4.w};
                uint32_t nb[DCLASS];
#pragma unroll
                for (int d = 0; d < DCLASS; ++d) nb[d] = s_nbr[i * DCLASS + d];
                const int hi = s_h[i];
                int8_t* row = sp + (size_t)i * P;
                const int n_par = (P + 1 - par) >> 1;  // copies of this parity
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    const int hh = 4 * g + w;
                    if (hh < n_par) {
                        const int k = par + 2 * hh;
                        const int sk = row[k];
                        int f = hi;
#pragma unroll
                        for (int d = 0; d < DCLASS; ++d) {
                            const int j = (int)(nb[d] >> 8);
                            const int J = (int)(int8_t)(nb[d] & 0xFFu);
                            f += J * (int)sp[(size_t)j * P + k];
                        }
                        const int Lf = sk * f;
                        const int km1 = (k == 0) ? P - 1 : k - 1;
                        const int kp1 = (k + 1 == P) ? 0 : k + 1;
                        // a classical chain's lone copy (P = 1) has no Trotter neighbours
                        const int m = P == 1 ? 0 : sk * ((int)row[km1] + (int)row[kp1]);
                        const uint32_t th = thr[(Lf + Lmax) * 3 + (m >> 1) + 1];
                        if (th == 0xFFFFFFFFu || rw[w] < th) {
                            row[k] = (int8_t)(-sk);
                            dE -= 2 * Lf;
                            dM -= 2 * m;
                            nf += 1;
                        }
                    }
                }
            }
            __syncthreads();
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            dE += __shfl_xor_sync(0xFFFFFFFFu, dE, o);
            dM += __shfl_xor_sync(0xFFFFFFFFu, dM, o);
            nf += __shfl_xor_sync(0xFFFFFFFFu, nf, o);
        }
        if (lane == 0) {
            s_red[warp * 3 + 0] = dE;
            s_red[warp * 3 + 1] = dM;
            s_red[warp * 3 + 2] = nf;
        }
        __syncthreads();
        if (tid == 0) {
            long long sE = 0, sM = 0, sF = 0;
            for (int w = 0; w < nwarps; ++w) {
                sE += s_red[w * 3 + 0];
                sM += s_red[w * 3 + 1];
                sF += s_red[w * 3 + 2];
            }
            int abort_flag = 0;
            s_ctl[0] = end_of_sweep(p, p.acc_in_smem ? s_acc : p.acc, rung, E, M, sE, sM, sF, s, q0,
                                    sweeps_per_swap, timeout_ns, key, &abort_flag);
            s_ctl[1] = abort_flag;
        }
        __syncthreads();
        if (s_ctl[1]) return;  // a partner never arrived; status holds PT_ETIMEDOUT
        const int nr = s_ctl[0];
        if (nr != rung) {
            rung = nr;
            if (!p.tables_in_smem) load_thr(p, s_thr, rung, tid, nt);
            thr = thr_row(p, s_thr, rung);
        }
        __syncthreads();
    }
    flush_acc(p, s_acc, tid, nt);

    {
        int4* dst = reinterpret_cast<int4*>(p.spins + (size_t)slot * p.slot_stride);
        const int4* src = reinterpret_cast<const int4*>(sp);
        const int n16 = (int)(up16((size_t)N * P) / 16);
        for (int x = tid; x < n16; x += nt) dst[x] = src[x];
    }
    if (tid == 0) {
        p.E[slot] = E;
        p.M[slot] = M;
        p.rung_of_slot[slot] = rung;
        p.slot_of_rung[rung] = slot;
    }
}

// ------------------------------------------------------------------------- classical sweep
// Path 10 (P = 1, classical tempering): the R chains packed C to a CTA (C a power of two),
// chain fastest in shared memory (site i of chain c at byte i C + c), on one cluster of
// K = ceil(R / C) CTAs. A level's updates are (site, chain) pairs, chain fastest, and every
// thread keeps one chain (blockDim is a multiple of C), so a warp reads one site's neighbour
// list for up to 32 chains and their bytes side by side, and the thread's threshold row is
// its chain's. After a sweep thread c of the CTA ends chain c's sweep: statistics, then the
// swap publication into every CTA of the cluster and the partner's wait in its own shared
// memory, as path 9 does (eos_decide_cluster). The update, its counter and its table entry
// are the byte-wise kernel's for P = 1.
struct ClassicalLayout {
    size_t spins, nbr, h, items, loff, thr, acc, cmb, E, M, rung, sums, ctl, total;
    __host__ __device__ ClassicalLayout(const DevProblem& p, int C) {
        size_t o = 0;
        spins = o; o += up16((size_t)p.N * C);
        nbr = o;   o += up16((size_t)p.N * p.dmax * 4);
        h = o;     o += up16((size_t)p.N);
        items = o; o += up16((size_t)2 * p.N * 4);
        loff = o;  o += up16((size_t)(p.n_levels + 1) * 4);
        thr = o;   o += up16((size_t)p.R * p.nL3 * 4);  // every rung's row
        acc = o;   o += (size_t)p.R * kAccCount * 8;      // this launch's statistics, by rung
        cmb = o;   o += (size_t)kClusterMailPasses * p.R * 16;
        E = o;     o += up16((size_t)C * 8);
        M = o;     o += up16((size_t)C * 8);
        rung = o;  o += up16((size_t)C * 4);
        sums = o;  o += up16((size_t)C * 8);               // per chain: dE and flips of the sweep
        ctl = o;   o += 16;
        total = o;
    }
};

size_t classical_smem_bytes(const DevProblem& p, int chains) { return ClassicalLayout(p, chains).total; }

template <int DCLASS>
__global__ void __launch_bounds__(512, 1)
    sweep_classical_kernel(DevProblem p, long long t0, long long q0, int n_sweeps, int sweeps_per_swap,
                           long long timeout_ns, int C) {
    extern __shared__ __align__(16) unsigned char smem[];
    wait_for_earlier_kernels();
    allow_next_kernel();
    cg::cluster_group cluster = cg::this_cluster();
    const int K = (p.R + C - 1) / C;
    if (cluster.num_blocks() != (unsigned)K || gridDim.x != (unsigned)K || p.P != 1 || C < 1 || (C & (C - 1)) ||
        (blockDim.x % (unsigned)C) || (blockDim.x & 31u)) {
        if (threadIdx.x == 0) atomicCAS(p.status, 0, PT_ECUDA);
        return;  // every CTA returns here, before any cluster barrier
    }
    const int N = p.N, R = p.R;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
    const int rank = (int)cluster.block_rank();
    const int c0 = rank * C, nc = min(C, R - c0);  // this CTA's chains: slots c0 .. c0 + nc - 1
    const ClassicalLayout L(p, C);
    int8_t* sp = reinterpret_cast<int8_t*>(smem + L.spins);
    uint32_t* s_nbr = reinterpret_cast<uint32_t*>(smem + L.nbr);
    int8_t* s_h = reinterpret_cast<int8_t*>(smem + L.h);
    uint32_t* s_items = reinterpret_cast<uint32_t*>(smem + L.items);
    int32_t* s_loff = reinterpret_cast<int32_t*>(smem + L.loff);
    uint32_t* s_thr = reinterpret_cast<uint32_t*>(smem + L.thr);
    unsigned long long* s_acc = reinterpret_cast<unsigned long long*>(smem + L.acc);
    unsigned long long* s_cmb = reinterpret_cast<unsigned long long*>(smem + L.cmb);
    long long* s_E = reinterpret_cast<long long*>(smem + L.E);
    long long* s_M = reinterpret_cast<long long*>(smem + L.M);
    int* s_rung = reinterpret_cast<int*>(smem + L.rung);
    int* s_sums = reinterpret_cast<int*>(smem + L.sums);  // [c][0] = dE, [c][1] = flips
    int* s_ctl = reinterpret_cast<int*>(smem + L.ctl);

    for (int x = tid; x < N * C; x += nt) {
        const int i = x / C, c = x - i * C;
        sp[x] = c < nc ? p.spins[(size_t)(c0 + c) * p.slot_stride + i] : (int8_t)1;
    }
    for (int x = tid; x < N * DCLASS; x += nt) s_nbr[x] = p.nbr[x];
    for (int x = tid; x < N; x += nt) s_h[x] = p.h[x];
    for (int x = tid; x < 2 * N; x += nt) s_items[x] = p.items[x];
    for (int x = tid; x <= p.n_levels; x += nt) s_loff[x] = p.level_off[x];
    for (int x = tid; x < R * p.nL3; x += nt) s_thr[x] = p.thr[x];
    for (int x = tid; x < R * kAccCount; x += nt) s_acc[x] = 0ull;
    for (int x = tid; x < kClusterMailPasses * R * 2; x += nt) s_cmb[x] = 0ull;
    for (int c = tid; c < C; c += nt) {
        s_E[c] = c < nc ? p.E[c0 + c] : 0;
        s_M[c] = c < nc ? p.M[c0 + c] : 0;
        s_rung[c] = c < nc ? p.rung_of_slot[c0 + c] : 0;
        s_sums[2 * c] = s_sums[2 * c + 1] = 0;
    }
    if (tid == 0) s_ctl[0] = 0;
    __syncthreads();
    cluster_barrier();  // every CTA's mailboxes are clear before anyone publishes

    const PhiloxKey key = philox_schedule(p.key0, p.key1);
    const int Lmax = p.Lmax;
    const int my_c = tid & (C - 1);  // this thread's chain, the same in every level
    int lgC = 0;
    while ((1 << lgC) < C) ++lgC;
    const bool live = my_c < nc;
    const uint32_t my_slot = (uint32_t)(c0 + my_c);
    const uint32_t* thr = s_thr + (size_t)s_rung[my_c] * p.nL3 + 1;  // m = 0 column
    const uint32_t qmod0 = (uint32_t)(q0 % kTagPeriod);
    int since_pass = 0, next_pass = 0;  // thread c < nc: chain c's swap schedule

    for (int s = 0; s < n_sweeps; ++s) {
        const uint32_t t = (uint32_t)(t0 + s);
        int dE = 0, nf = 0;
        for (int lev = 0; lev < p.n_levels; ++lev) {
            const int base = s_loff[lev];
            const int units = (s_loff[lev + 1] - base) << lgC;
            if (live)
                for (int u = tid; u < units; u += nt) {
                    const int i = (int)(s_items[base + (u >> lgC)] >> 1);
                    const uint32_t r = philox(make_uint4(t, (uint32_t)i, my_slot, 0u), key).x;
                    int f = s_h[i];
#pragma unroll
                    for (int d = 0; d < DCLASS; ++d) {
                        const uint32_t nb = s_nbr[i * DCLASS + d];
                        f += (int)(int8_t)(nb & 0xFFu) * (int)sp[(size_t)(nb >> 8) * C + my_c];
                    }
                    int8_t* own = sp + (size_t)i * C + my_c;
                    const int sk = *own;
                    const int Lf = sk * f;
                    const uint32_t th = thr[(Lf + Lmax) * 3];
                    if (th == 0xFFFFFFFFu || r < th) {
                        *own = (int8_t)(-sk);
                        dE -= 2 * Lf;
                        nf += 1;
                    }
                }
            __syncthreads();
        }
        // the sweep's changes of each chain: lanes of a warp that share a chain are C apart
        for (int o = 16; o >= C; o >>= 1) {
            dE += __shfl_xor_sync(0xFFFFFFFFu, dE, o);
            nf += __shfl_xor_sync(0xFFFFFFFFu, nf, o);
        }
        if (live && lane < C && (dE | nf)) {
            atomicAdd(s_sums + 2 * my_c, dE);
            atomicAdd(s_sums + 2 * my_c + 1, nf);
        }
        __syncthreads();
        // chain tid's end of sweep, in two phases: every chain of the CTA publishes before
        // any of them waits, so partners on one CTA never wait on a thread that has not
        // published yet (spreading the copies over the CTA's threads, behind one more
        // barrier, measured slower)
        SwapSide side;
        long long E = 0, M = 0;
        int rung = 0;
        if (tid < nc) {
            const int c = tid;
            E = s_E[c];
            M = s_M[c];
            rung = s_rung[c];
            const int sE = s_sums[2 * c], sF = s_sums[2 * c + 1];
            s_sums[2 * c] = s_sums[2 * c + 1] = 0;
            int pass = -1;
            if (sweeps_per_swap > 0 && ++since_pass == sweeps_per_swap) {
                since_pass = 0;
                pass = next_pass++;
            }
            side = eos_publish(p, rung, E, M, sE, 0, pass, q0, qmod0, false);
            eos_stats(p, s_acc, rung, E, M, sF);
            if (side.active && rung != p.withhold_rung) {
                const int idx = ((side.pass & (kClusterMailPasses - 1)) * R + rung) * 2;
                const unsigned long long wa = ((unsigned long long)E << 24) | side.tag;
                const unsigned long long wb = ((unsigned long long)(uint32_t)(int32_t)M << 32) | side.tag;
                for (int r = 0; r < K; ++r) st_cluster_u64x2(s_cmb + idx, (unsigned)r, wa, wb);
            }
        }
        __syncthreads();
        if (tid < nc) {
            const int c = tid;
            int abort_flag = 0;
            s_rung[c] = eos_decide_cluster(p, s_cmb, side, rung, E, M, timeout_ns, key, &abort_flag);
            s_E[c] = E;
            s_M[c] = M;
            if (abort_flag) s_ctl[0] = 1;  // a partner never arrived
        }
        __syncthreads();
        if (s_ctl[0]) break;  // to the cluster barrier that every CTA passes before leaving
        thr = s_thr + (size_t)s_rung[my_c] * p.nL3 + 1;
    }
    __syncthreads();
    // no CTA leaves while another may still write its mailboxes (every wait is bounded)
    cluster_barrier();
    if (s_ctl[0]) return;  // status holds PT_ETIMEDOUT
    for (int x = tid; x < R * kAccCount; x += nt)
        if (s_acc[x]) atomicAdd(p.acc + x, s_acc[x]);
    for (int x = tid; x < N * nc; x += nt) {
        const int c = x / N, i = x - c * N;
        p.spins[(size_t)(c0 + c) * p.slot_stride + i] = sp[(size_t)i * C + c];
    }
    for (int c = tid; c < nc; c += nt) {
        const int rung = s_rung[c];
        p.E[c0 + c] = s_E[c];
        p.M[c0 + c] = s_M[c];
        p.rung_of_slot[c0 + c] = rung;
        p.slot_of_rung[rung] = c0 + c;
    }
}

// ------------------------------------------------------------------------- packed sweep
// Random words of one sweep for the producer warps: word w of philox((t, i, slot,
// p<<24 | g)) goes with copy 8g + p + 2w of site i (the same counter the update would use).
__device__ __forceinline__ void produce_words(uint4* buf, uint32_t t, const uint32_t* s_items, int n_items, int G,
                                              int ptid, int np, uint32_t slot, const PhiloxKey& key) {
    if (ptid < 0 || np <= 0) return;  // producer threads only
    auto make = [&](int q, int g) {
        const uint32_t it = s_items[q];
        // stored as min(u, 2^32 - 2): then u < thr alone is the acceptance rule, the
        // "accept always" entry 0xFFFFFFFF included
        const uint4 r = philox(make_uint4(t, it >> 1, slot, ((it & 1u) << 24) | (uint32_t)g), key);
        buf[q * G + g] = make_uint4(min(r.x, 0xFFFFFFFEu), min(r.y, 0xFFFFFFFEu), min(r.z, 0xFFFFFFFEu),
                                    min(r.w, 0xFFFFFFFEu));
    };
    if (np >= G) {  // a thread keeps one column
        const int step = np / G, q0 = ptid / G, g = ptid - q0 * G;
        if (q0 < step)
            for (int q = q0; q < n_items; q += step) make(q, g);
    } else {
        for (int q = 0; q < n_items; ++q)
            for (int g = ptid; g < G; g += np) make(q, g);
    }
}

// One CTA per chain with the chain, the unit descriptors and the threshold row in shared
// memory. PRE: the last (blockDim - n_consumer) threads are producer warps that write the
// random words of sweep s+1 into one shared buffer while the consumer warps run the levels
// of sweep s out of the other; consumers synchronise levels on named barrier 1 and both
// groups meet once per sweep.
// PEER (path 8): the CTA is rank 0 of a cluster of two, and rank 1 (peer_producer below)
// writes the random words into this CTA's buffers through distributed shared memory; every
// thread here sweeps, and the two CTAs meet at a cluster barrier once per sweep.
// CSWAP (path 9): the CTAs of all R chains form one cluster (slot = rank) and the swap
// mailboxes live in every CTA's shared memory (eos_decide_cluster); the CTAs meet at a
// cluster barrier only after the mailboxes are cleared and before they leave.
// DC = 0: path 1's word-wise kernel (RowsLayout, rows_unit_eval) on the same loop.
// COPY (with DC = 0 and PRE): one copy a thread.
// PIECES (with PEER): a sweep's random words come in p.n_chunks pieces (pt_internal.h).
// NIB > 0: the nibble form of the bit-packed chain with NIB neighbour slots in use.
// REC: records in place of descriptors (DevProblem::records, with a thread for every column). The
// instances without records hold the loop over descriptors alone: beside the one over records it
// took 15 to 20 % longer (path 2, N=2048, P=32, R=48: 17.1 us per sweep against 14.8). Those with
// records keep both, and the run-time choice, although only one runs: the loop over records by
// itself is compiled to 1 to 5 % slower code (path 9, N=16, P=32, R=16: 2.31 -> 2.40 us per sweep).
template <int DC, bool PRE, bool WIDE, bool BITS = false, bool SPEC = true, bool PEER = false, bool CSWAP = false,
          int NIB = 0, bool COPY = false, bool PIECES = false, bool REC = false>
__device__ __forceinline__ void sweep_packed_body(const DevProblem& p, int slot, long long t0, long long q0,
                                                  int n_sweeps, int sweeps_per_swap, long long timeout_ns,
                                                  int n_consumer, unsigned char* smem) {
    const int N = p.N, P = p.P;
    const int tid = threadIdx.x, nt = blockDim.x;
    constexpr bool ROWS = DC == 0;
    struct PackedLayout : FastLayout {
        __device__ explicit PackedLayout(const DevProblem& q) : FastLayout(q, DC, PRE, BITS, CSWAP) {}
    };
    struct WordsLayout : RowsLayout {
        __device__ explicit WordsLayout(const DevProblem& q) : RowsLayout(q, PRE, CSWAP) {}
    };
    const std::conditional_t<ROWS, WordsLayout, PackedLayout> L(p);
    int8_t* sp = reinterpret_cast<int8_t*>(smem + L.spins);
    uint32_t* s_desc = reinterpret_cast<uint32_t*>(smem + L.desc);
    uint32_t* s_items = reinterpret_cast<uint32_t*>(smem + L.items);
    int32_t* s_loff = reinterpret_cast<int32_t*>(smem + L.loff);
    uint32_t* s_thr = reinterpret_cast<uint32_t*>(smem + L.thr);
    long long* s_red = reinterpret_cast<long long*>(smem + L.red);
    int* s_ctl = reinterpret_cast<int*>(smem + L.ctl);
    unsigned long long* s_acc = reinterpret_cast<unsigned long long*>(smem + L.acc);
    uint4* rbuf = reinterpret_cast<uint4*>(smem + L.rbuf);
    unsigned long long* s_cmb = reinterpret_cast<unsigned long long*>(smem + L.cmb);
    uint8_t* bp = nullptr;
    uint32_t* s_lut = nullptr;
    if constexpr (!ROWS) {
        bp = reinterpret_cast<uint8_t*>(smem + L.spins);
        s_lut = reinterpret_cast<uint32_t*>(smem + L.lut);
    }
    const int NC = PRE ? n_consumer : nt;
    const bool consumer = tid < NC;
    // columns of a parity of a row: words of 4 copies, or nibble words of 16
    const int G = NIB ? P >> 5 : ((P >> 1) + 3) >> 2;
    const uint32_t half = 4u * (uint32_t)G;
    const int desc_words = ROWS ? rows_desc_words(p.slots) : SiteDesc<ROWS ? 4 : DC>::DW;
    static_assert(!REC || (!BITS && (COPY || !ROWS)), "kernels that have records");
    const bool rec = REC && p.records;

    // what no earlier kernel writes
    if constexpr (ROWS) {
        const int RB = 2 * (int)half;
        // descriptors from the neighbour table (entries with J = 0 are padding), or (COPY) records:
        // descriptors in schedule order with the parity worked in
        const uint32_t zero = (uint32_t)IndexRule(p.Lmax).zero();
        for (int x = tid; x < (rec ? 2 * N : N); x += nt) {
            const uint32_t item = rec ? p.items[x] : 2u * (uint32_t)x;
            const uint32_t i = item >> 1, shift = (item & 1u) * half, row = i * (uint32_t)RB;
            uint32_t* d = s_desc + (size_t)x * desc_words;
            uint32_t sumJ = 0u, n = 0u;
            for (int k = 0; k < p.dmax; ++k) {
                const uint32_t e = p.nbr[(size_t)i * p.dmax + k];
                const uint32_t J = (uint32_t)(int)(int8_t)(e & 0xFFu);
                if (J == 0u) continue;
                d[4 + 2 * n] = (e >> 8) * (uint32_t)RB + shift;
                d[5 + 2 * n] = COPY ? J : J * (0u - kInv127);
                sumJ += J;
                ++n;
            }
            for (; n == 0u || (n & 3u); ++n) {  // at least the four slots every unit reads
                d[4 + 2 * n] = row + shift;
                d[5 + 2 * n] = 0u;
            }
            d[0] = COPY ? (uint32_t)(int)p.h[i]
                        : ((uint32_t)(int)p.h[i] + sumJ + zero + kInv127 * sumJ) * 0x01010101u;
            d[1] = row + shift;
            d[2] = n;
            d[3] = row + half - shift;
        }
    } else if constexpr (BITS && NIB == 0) {
        for (int x = tid; x < 512; x += nt) {
            const uint32_t par = (uint32_t)x >> 8, byte = (uint32_t)x & 0xFFu;
            uint32_t v = 0;
#pragma unroll
            for (int w = 0; w < 4; ++w) v |= (((byte >> (par + 2 * w)) & 1u) ? 0xFFu : 0x01u) << (8 * w);
            s_lut[x] = v;
        }
    }
    {
        if constexpr (!ROWS) {
            if (rec) {
                for (int x = tid; x < 2 * N; x += nt) {
                    const uint32_t item = p.items[x];
                    make_record<DC>(s_desc + (size_t)x * UnitRecord<DC>::kWords, p.desc + (item >> 1) * desc_words,
                                    item, half);
                }
            } else {
                const int4* dsrc = reinterpret_cast<const int4*>(p.desc);
                int4* ddst = reinterpret_cast<int4*>(s_desc);
                for (int x = tid; x < N * desc_words / 4; x += nt) ddst[x] = dsrc[x];
            }
        }
        for (int x = tid; x < 2 * N; x += nt) s_items[x] = p.items[x];
        for (int x = tid; x <= p.n_levels; x += nt) s_loff[x] = p.level_off[x];
    }
    if (p.tables_in_smem) load_thr_columns(p, s_thr, 0, tid, nt);
    if (p.acc_in_smem)
        for (int x = tid; x < p.R * kAccCount; x += nt) s_acc[x] = 0ull;
    if (tid == 0) {
        s_ctl[5] = 0;  // a swap wait gave up
        int* s_sum = reinterpret_cast<int*>(s_red);
        s_sum[0] = s_sum[1] = s_sum[2] = 0;  // the sweep's dE, dM and flips
    }
    if (CSWAP)
        for (int x = tid; x < kClusterMailPasses * p.R * 2; x += nt) s_cmb[x] = 0ull;
    const int n_items = 2 * N;
    if (PRE && !PEER) {
        __syncthreads();
        if (!consumer)
            produce_words(rbuf, (uint32_t)t0, s_items, n_items, G, tid - NC, nt - NC, (uint32_t)slot,
                          philox_schedule(p.key0, p.key1));
    }
    wait_for_earlier_kernels();
    allow_next_kernel();

    // the chain, its energies and its rung
    if constexpr (ROWS) {
        const int8_t* src = p.spins + (size_t)slot * p.slot_stride;
        const int RB = 2 * (int)half, n_par = P >> 1;
        for (int x = tid; x < N * RB; x += nt) {
            const int i = x / RB, c = x - i * RB;
            const int par = c >= (int)half, h = c - par * (int)half;
            sp[x] = h < n_par ? src[(size_t)i * P + 2 * h + par] : (int8_t)1;
        }
    } else if constexpr (NIB > 0) {
        load_bits<4>(reinterpret_cast<uint32_t*>(sp), p.spins + (size_t)slot * p.slot_stride, N, G, tid, nt);
    } else if constexpr (BITS) {
        // int8 chain in global memory -> one bit per copy in shared memory
        const uint2* src = reinterpret_cast<const uint2*>(p.spins + (size_t)slot * p.slot_stride);
        for (int x = tid; x < N * (P / 8); x += nt) {
            const uint2 v = src[x];
            uint32_t b = 0;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                b |= ((v.x >> (8 * k + 7)) & 1u) << k;
                b |= ((v.y >> (8 * k + 7)) & 1u) << (k + 4);
            }
            bp[x] = (uint8_t)b;
        }
    } else {
        // interleaved int8 chain in global memory -> parity-split rows in shared memory
        load_split(sp, p.spins + (size_t)slot * p.slot_stride, N, P, P >> 3, chunk_ginv(P >> 3), tid, nt);
    }
    int rung = p.rung_of_slot[slot];
    if (!p.tables_in_smem) load_thr_columns(p, s_thr, rung, tid, nt);
    long long E = p.E[slot], M = p.M[slot];  // meaningful in the threads that end the sweeps
    __syncthreads();
    if (CSWAP) cluster_barrier();  // every CTA's mailboxes are clear before anyone publishes

    const PhiloxKey key = philox_schedule(p.key0, p.key1);
    const int cols = COPY ? P >> 1 : G;  // units of an item
    const UnitRule<WIDE> rule(p.Lmax);
    // byte offset in shared memory at which the current rung's threshold row is looked up
    const int S = IndexRule(p.Lmax).S;
    const uint32_t thr0 =
        COPY ? (uint32_t)L.thr + 4u * (uint32_t)(p.Lmax + S) : thr_base<WIDE>((uint32_t)L.thr, p.Lmax);
    const uint32_t thr_step = p.tables_in_smem ? 12u * (uint32_t)S : 0u;
    uint32_t thr_c = thr0 + thr_step * (uint32_t)rung;
    const int lane = tid & 31;
    if (PEER) {
        // the barrier entered at the start of the kernel, then: the peer CTA has written the first
        // sweep's words (its arrival releases them); this CTA's arrival orders nothing of its own,
        // so it is relaxed
        cluster_wait_acquire();
        cluster_arrive_relaxed();
        cluster_wait_acquire();
    }

    // Level 0 of the next sweep can be evaluated while the swap decision is still pending:
    // its inputs are the spins after this sweep and the next sweep's random words; only its
    // threshold row depends on the decision, and both candidate rows are in shared memory.
    // Up to two level-0 units per consumer thread are held in registers.
    // Warp 0 takes no level-0 unit, so that thread 0 can poll the partner's mailbox at once.
    const int units0 = (s_loff[1] - s_loff[0]) * cols;
    const bool spec_ok = SPEC && !BITS && p.tables_in_smem && NC > 32 && units0 <= 2 * (NC - 32);
    bool spec_done = false;  // level 0 of sweep s was applied at the end of sweep s - 1
    int spec_q[2], spec_g[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int u = (tid - 32) + k * (NC - 32);
        const bool ok = spec_ok && consumer && tid >= 32 && u < units0;
        spec_q[k] = ok ? s_loff[0] + u / cols : -1;
        spec_g[k] = ok ? u % cols : 0;
    }
    // With a thread for every column, a thread keeps its column g and walks the items q_lane,
    // q_lane + q_step, ... of a level
    const bool g_fixed = NC >= cols;
    const int q_step = NC / cols, q_lane = tid / cols, g_own = tid - q_lane * cols;
    const bool lane_ok = consumer && q_lane < q_step;
    // words of one of the two buffers; PIECES: pieces used so far
    const size_t buf_words = (size_t)(PIECES ? p.chunk_items : n_items) * G;
    int chunk = 0;
    FlipSums sums;
    sums.clear();
    BitSums nib_sums = {0, 0, 0};
    CopySums copy_sums = {0, 0, 0};
    // A unit of item q and column g up to its index and random words, its flips against the
    // threshold row at thr, and the commit.
    using Column = std::conditional_t<COPY, UnitOffsets, RowsColumn>;
    using Eval = std::conditional_t<COPY, CopyEval, UnitEval<1>>;
    auto column = [&](int g) -> Column {
        if constexpr (COPY)
            return copy_offsets((uint32_t)g, half, (uint32_t)P >> 1);
        else if constexpr (ROWS)
            return rows_column((uint32_t)g, (uint32_t)G, (uint32_t)P >> 1);
        else
            return RowsColumn{row_offsets<1>((uint32_t)g, half), 0u, 0u};
    };
    const Column col_own = column(g_own);  // this thread's fixed one
    using Record = std::conditional_t<COPY, RowsTerms, LoadedRecord<ROWS ? 4 : DC>>;
    auto load_rec = [&](int q) -> Record {
        if constexpr (COPY)
            return load_rows_site(s_desc + q * desc_words);
        else
            return load_record<ROWS ? 4 : DC>(s_desc + q * UnitRecord<ROWS ? 4 : DC>::kWords);
    };
    auto eval_rec = [&](const Record& r, int q, int g, const Column& c, const uint4* rb, uint32_t t) -> Eval {
        if constexpr (COPY)
            // word h % 4 of call h / 4: the words of an item's copies are consecutive
            return copy_record_eval(sp, r, (uint32_t)g, c.edge[0] - half, c.edge[1],
                                    reinterpret_cast<const uint32_t*>(rb + q * G)[g]);
        else
            return record_eval<ROWS ? 4 : DC, PRE, WIDE>(sp, r, 4u * (uint32_t)g, c.o.edge[0] - half, c.o.edge[1],
                                                         rb + q * G + g, t, (uint32_t)slot, rule, key);
    };
    auto eval_desc = [&](int q, int g, const Column& c, const uint4* rb, uint32_t t) -> Eval {
        const uint32_t item = s_items[q];
        const uint32_t* desc = s_desc + (item >> 1) * (uint32_t)desc_words;
        if constexpr (COPY) {
            return copy_eval(sp, desc, item & 1u, c, reinterpret_cast<const uint32_t*>(rb + q * G)[g]);
        } else {
            UnitEval<1> e;
            unit_words<1, PRE>(e.u, item, rb + q * G + g, t, (uint32_t)slot, (uint32_t)g, key);
            if constexpr (ROWS)
                rows_eval_site<WIDE>(e, sp, load_rows_site(desc), item & 1u, c, rule);
            else
                unit_eval_site<DC, 1, WIDE>(e, sp, load_site<DC>(desc), item & 1u, c.o, rule);
            return e;
        }
    };
    auto flips = [&](const Eval& e, const Column& c, uint32_t thr) -> uint32_t {
        if constexpr (COPY) {
            return copy_flips(e, smem, (int)thr, S);
        } else {
            uint32_t F[1];
            unit_flips<1, PRE, WIDE>(e, smem, rule, thr, F);
            return ROWS ? F[0] & c.live : F[0];
        }
    };
    auto commit = [&](const Eval& e, uint32_t F) {
        if constexpr (COPY)
            copy_commit(e, F != 0u, copy_sums);
        else
            unit_commit<1>(e, &F, sums);
    };
    const bool ender = CSWAP ? tid < 32 : tid == 0;  // follows E and M and ends the sweeps
    SwapSide side;  // ender
    side.active = 0;
    const uint32_t qmod0 = (uint32_t)(q0 % kTagPeriod);
    int since_pass = 0, next_pass = 0;
    int sweep_flips = 0;  // ender

    for (int s = 0; s < n_sweeps; ++s) {
        const uint32_t t = (uint32_t)(t0 + s);
        if (consumer && !s_ctl[5]) {
            const uint4* rb = rbuf + (size_t)((PIECES ? chunk : s) & 1) * buf_words;
            if (!spec_done) {
                sums.clear();
                copy_sums = CopySums{0, 0, 0};
            }
            if constexpr (NIB > 0) {
                const IndexRule index(p.Lmax);
                nib_sums.clear();
                auto unit = [&](int q, uint32_t g, const UnitOffsets& off) {
                    bits_unit<DC, NIB, 4>(sp, s_desc, s_items[q], off, g, t, (uint32_t)slot, key, smem,
                                          (uint32_t)index.S, (uint32_t)(2 * p.Lmax - 255) * kInv255, thr_c, nib_sums);
                };
                const UnitOffsets off = word_offsets((uint32_t)g_own, (uint32_t)G);
                for (int lev = 0; lev < p.n_levels; ++lev) {
                    const int base = s_loff[lev], end = s_loff[lev + 1];
                    if (g_fixed) {
                        if (lane_ok)
                            for (int q = base + q_lane; q < end; q += q_step) unit(q, (uint32_t)g_own, off);
                    } else {
                        for (int u = tid; u < (end - base) * cols; u += NC) {
                            const int q = u / cols;
                            unit(base + q, (uint32_t)(u - q * cols), word_offsets((uint32_t)(u - q * cols), (uint32_t)G));
                        }
                    }
                    __syncthreads();
                }
            } else {
                for (int piece = 0; piece < (PIECES ? p.n_chunks : 1); ++piece) {
                    if (PIECES && piece > 0) {  // the next piece's words; this one's are no longer needed
                        cluster_arrive_relaxed();
                        cluster_wait_acquire();
                        ++chunk;
                        rb = rbuf + (size_t)(chunk & 1) * buf_words - (size_t)s_loff[p.chunk_level[piece]] * G;
                    }
                    const int lev0 = piece > 0 ? p.chunk_level[piece] : spec_done ? 1 : 0;
                    const int lev_end = PIECES ? p.chunk_level[piece + 1] : p.n_levels;
                    if (rec && g_fixed) {
                        // this thread's column never changes: its row offsets are loop invariants. Each
                        // level's first record is loaded before the barrier that ends the level before.
                        int end = s_loff[min(lev0 + 1, lev_end)], q = s_loff[lev0] + q_lane;
                        bool have = lane_ok && q < end;
                        Record r = {};
                        if (have) r = load_rec(q);
                        for (int lev = lev0; lev < lev_end; ++lev) {
                            const int end2 = s_loff[min(lev + 2, lev_end)];
                            if (have) {
                                Eval e = eval_rec(r, q, g_own, col_own, rb, t);
                                commit(e, flips(e, col_own, thr_c));
                                for (q += q_step; q < end; q += q_step) {
                                    e = eval_rec(load_rec(q), q, g_own, col_own, rb, t);
                                    commit(e, flips(e, col_own, thr_c));
                                }
                            }
                            q = end + q_lane;
                            end = end2;
                            have = lane_ok && q < end;
                            if (have) r = load_rec(q);
                            if (PRE) named_barrier(1, NC); else __syncthreads();
                        }
                    } else {
                        for (int lev = lev0; lev < lev_end; ++lev) {
                            const int base = s_loff[lev];
                            auto unit = [&](int q, int g, const Column& c) {
                                if constexpr (BITS) {
                                    packed_unit_bits<DC, WIDE>(bp, s_desc, s_items[q], g, G, s_lut, t, (uint32_t)slot,
                                                               key, smem, rule, thr_c, sums);
                                } else {
                                    const Eval e = rec ? eval_rec(load_rec(q), q, g, c, rb, t) : eval_desc(q, g, c, rb, t);
                                    commit(e, flips(e, c, thr_c));
                                }
                            };
                            if (g_fixed) {
                                if (lane_ok) {
                                    const int end = s_loff[lev + 1];
                                    for (int q = base + q_lane; q < end; q += q_step) unit(q, g_own, col_own);
                                }
                            } else {
                                const int units = (s_loff[lev + 1] - base) * cols;
                                for (int u = tid; u < units; u += NC) {
                                    const int q = u / cols, g = u - q * cols;
                                    unit(base + q, g, column(g));
                                }
                            }
                            if (PRE) named_barrier(1, NC); else __syncthreads();
                        }
                    }
                }
            }
            // a chain's per-sweep changes fit in 32 bits: each warp adds its sums to three
            // shared counters, which thread 0 reads and clears
            int dE = sums.dE(rule), dM = sums.dM(rule), dF = sums.flips();
            if (COPY) {
                dE = -2 * copy_sums.L;
                dM = -2 * copy_sums.M;
                dF = copy_sums.n;
            }
            if (NIB > 0) {
                dE = nib_sums.dE(p.Lmax);
                dM = nib_sums.dM();
                dF = nib_sums.flips();
            }
            dE = __reduce_add_sync(0xFFFFFFFFu, dE);
            dM = __reduce_add_sync(0xFFFFFFFFu, dM);
            dF = __reduce_add_sync(0xFFFFFFFFu, dF);
            int* s_sum = reinterpret_cast<int*>(s_red);
            if (lane == 0) {
                atomicAdd(s_sum + 0, dE);
                atomicAdd(s_sum + 1, dM);
                atomicAdd(s_sum + 2, dF);
            }
        } else if (PRE && !consumer && s + 1 < n_sweeps) {
            // producer warps only: a consumer whose swap wait gave up skips to the barrier below
            produce_words(rbuf + (size_t)((s + 1) & 1) * n_items * G, t + 1u, s_items, n_items, G, tid - NC, nt - NC,
                          (uint32_t)slot, key);
        }
        ++chunk;
        // a swap pass follows every sweeps_per_swap-th sweep (counted, not divided)
        int pass = -1;
        if (sweeps_per_swap > 0 && ++since_pass == sweeps_per_swap) {
            since_pass = 0;
            pass = next_pass++;
        }
        // the sweep's sums and the next sweep's random words are complete, and every consumer has
        // finished sweep s; a wait that gave up in the previous sweep ends the launch here, for
        // every thread
        if constexpr (PEER) {
            // The peer CTA learns at the cluster barrier that this CTA leaves, and leaves too.
            // Otherwise the arrival is relaxed: a release would first wait for earlier global
            // stores to reach L2, on the way to the swap decision. The words this CTA read are in
            // registers by now, so the peer may overwrite their buffer.
            named_barrier(1, NC);
            if (s_ctl[5]) {
                if (tid == 0) cg::this_cluster().map_shared_rank(s_ctl, 1)[6] = 1;
                cluster_arrive_release();
            } else {
                cluster_arrive_relaxed();
            }
        } else {
            __syncthreads();
        }
        // Thread 0 ends the sweep. On path 9 all of warp 0 does, every lane with the same E and M, so
        // that lane r writes the publication into CTA r (one store instruction; thread 0 alone took
        // 17 cycles a copy: 2.42 -> 2.32 us per sweep on N=16, P=32, R=16; through global mailboxes
        // a warp's polls measured 0.1 us slower than one thread's).
        if (ender && !s_ctl[5]) {
            int* s_sum = reinterpret_cast<int*>(s_red);
            const int sE = s_sum[0], sM = s_sum[1];
            sweep_flips = s_sum[2];
            if (CSWAP) __syncwarp();
            if (lane == 0) s_sum[0] = s_sum[1] = s_sum[2] = 0;
            side = eos_publish(p, rung, E, M, sE, sM, pass, q0, qmod0, !CSWAP && lane == 0);
            if (CSWAP && side.active && rung != p.withhold_rung && lane < p.R) {
                const int idx = ((side.pass & (kClusterMailPasses - 1)) * p.R + rung) * 2;
                const unsigned long long wa = ((unsigned long long)E << 24) | side.tag;
                const unsigned long long wb = ((unsigned long long)(uint32_t)(int32_t)M << 32) | side.tag;
                st_cluster_u64x2(s_cmb + idx, (unsigned)lane, wa, wb);
            }
        }
        if constexpr (PEER) cluster_wait_acquire();
        if (s_ctl[5]) {  // status holds PT_ETIMEDOUT
            if (CSWAP) break;  // to the cluster barrier that every CTA passes before leaving
            return;
        }
        if (!consumer) continue;

        // level 0 of sweep s + 1 under both candidate rungs
        const bool spec = spec_ok && s + 1 < n_sweeps;
        const int prung = pass >= 0 ? pair_rung(rung, q0 + pass, p.R) : -1;
        Eval ev[2];
        uint32_t Fa[2] = {0u, 0u}, Fb[2] = {0u, 0u};
        bool valid[2] = {false, false};
        if (spec) {
            const uint4* rb1 = rbuf + (size_t)((PIECES ? chunk : s + 1) & 1) * buf_words;
            const uint32_t thr_b = prung >= 0 ? thr0 + thr_step * (uint32_t)prung : thr_c;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                valid[k] = spec_q[k] >= 0;
                if (valid[k]) {
                    const int q = spec_q[k], g = spec_g[k];
                    const Column c = column(g);
                    ev[k] = rec ? eval_rec(load_rec(q), q, g, c, rb1, t + 1u) : eval_desc(q, g, c, rb1, t + 1u);
                    Fa[k] = flips(ev[k], c, thr_c);
                    Fb[k] = prung >= 0 ? flips(ev[k], c, thr_b) : Fa[k];
                }
            }
        }
        if (ender) {
            // the statistics of sweep s (rung unchanged until the decision below), while
            // the partner's mailbox may still be on its way
            if (lane == 0) eos_stats(p, p.acc_in_smem ? s_acc : p.acc, rung, E, M, sweep_flips);
            if (prung >= 0) {
                int abort_flag = 0;
                const int next =
                    CSWAP ? eos_decide_cluster(p, s_cmb, side, rung, E, M, timeout_ns, key, &abort_flag, lane == 0)
                          : eos_decide(p, side, rung, E, M, timeout_ns, key, &abort_flag, lane == 0);
                if (CSWAP) __syncwarp();
                if (lane == 0) {
                    s_ctl[2 * (s & 1)] = next;
                    if (abort_flag) s_ctl[5] = 1;  // a partner never arrived
                }
            }
        }
        bool moved = false;
        if (prung >= 0) {  // nobody waits for a decision that is not to be taken
            if (PRE) named_barrier(1, NC); else __syncthreads();
            if (s_ctl[5]) continue;  // skip to the next barrier with the producers, then leave
            const int nr = s_ctl[2 * (s & 1)];
            moved = nr != rung;
            if (moved) {
                rung = nr;
                if (!p.tables_in_smem) load_thr_columns(p, s_thr, rung, tid, NC);
                thr_c = thr0 + thr_step * (uint32_t)rung;
            }
        }
        spec_done = spec;
        if (spec) {
            sums.clear();
            copy_sums = CopySums{0, 0, 0};
#pragma unroll
            for (int k = 0; k < 2; ++k)
                if (valid[k]) commit(ev[k], moved ? Fb[k] : Fa[k]);
        }
        // the next sweep's reads of shared memory (level 1, or a reloaded threshold row) follow
        if (PRE) named_barrier(1, NC); else __syncthreads();
    }
    __syncthreads();
    // no CTA of a path-9 cluster leaves while another may still write its mailboxes (every
    // wait is bounded, so every CTA gets here)
    if (CSWAP) cluster_barrier();
    if (s_ctl[5]) return;  // the last sweep's wait gave up
    flush_acc(p, s_acc, tid, nt);

    if constexpr (NIB > 0) {
        store_bits<4>(p.spins + (size_t)slot * p.slot_stride, reinterpret_cast<const uint32_t*>(sp), N, G, tid, nt);
    } else if constexpr (BITS) {
        uint2* dst = reinterpret_cast<uint2*>(p.spins + (size_t)slot * p.slot_stride);
        for (int x = tid; x < N * (P / 8); x += nt) {
            const uint32_t b = bp[x];
            uint2 v = make_uint2(0u, 0u);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                v.x |= (((b >> k) & 1u) ? 0xFFu : 0x01u) << (8 * k);
                v.y |= (((b >> (k + 4)) & 1u) ? 0xFFu : 0x01u) << (8 * k);
            }
            dst[x] = v;
        }
    } else if constexpr (ROWS) {
        int8_t* dst = p.spins + (size_t)slot * p.slot_stride;
        for (int x = tid; x < N * P; x += nt) {
            const int i = x / P, k = x - i * P;
            dst[x] = sp[(size_t)i * 2 * half + (k & 1 ? half : 0u) + (k >> 1)];
        }
    } else {
        store_split(p.spins + (size_t)slot * p.slot_stride, sp, N, P, P >> 3, chunk_ginv(P >> 3), tid, nt);
    }
    if (tid == 0) {
        p.E[slot] = E;
        p.M[slot] = M;
        p.rung_of_slot[slot] = rung;
        p.slot_of_rung[rung] = slot;
    }
}

// Path 8, rank 1 of each cluster: the random words of every sweep of chain `slot`, written
// one sweep (or piece of a sweep, where two whole sweeps' words do not fit: DevProblem::n_chunks)
// ahead into rank 0's double buffer through distributed shared memory (the words
// are a function of the chain, the sweep and the update, never of the rung, so they need no
// swap decision). It passes the same cluster barriers as rank 0 (one entered at the start of the
// kernel, which shows that both CTAs run, one before the first sweep, one per sweep or piece) and
// leaves after the one at which rank 0 reports that it leaves.
template <int DC, bool PIECES>
__device__ void peer_producer(const DevProblem& p, int slot, long long t0, int n_sweeps, unsigned char* smem) {
    cg::cluster_group cluster = cg::this_cluster();
    const int tid = threadIdx.x, nt = blockDim.x;
    const FastLayout L(p, DC, true, false);
    uint32_t* s_items = reinterpret_cast<uint32_t*>(smem + L.items);
    int* s_ctl = reinterpret_cast<int*>(smem + L.ctl);
    uint4* peer_rbuf = cluster.map_shared_rank(reinterpret_cast<uint4*>(smem + L.rbuf), 0);
    const int n_items = 2 * p.N, G = p.P >> 3;
    int32_t* s_loff = reinterpret_cast<int32_t*>(smem + L.loff);
    for (int x = tid; x < n_items; x += nt) s_items[x] = p.items[x];
    for (int x = tid; x <= p.n_levels; x += nt) s_loff[x] = p.level_off[x];
    if (tid == 0) s_ctl[6] = 0;
    const PhiloxKey key = philox_schedule(p.key0, p.key1);
    __syncthreads();
    cluster_wait_acquire();  // rank 0 has started: its shared memory may be written
    const int pieces = PIECES ? p.n_chunks : 1;
    const size_t buf_words = (size_t)(PIECES ? p.chunk_items : n_items) * G;
    // piece k of the launch (piece k % pieces of sweep t0 + k / pieces), into buffer k & 1
    auto produce = [&](int sweep, int piece, int buffer) {
        const int first = PIECES ? s_loff[p.chunk_level[piece]] : 0;
        const int end = PIECES ? s_loff[p.chunk_level[piece + 1]] : n_items;
        produce_words(peer_rbuf + (size_t)buffer * buf_words, (uint32_t)(t0 + sweep), s_items + first, end - first, G,
                      tid, nt, (uint32_t)slot, key);
    };
    produce(0, 0, 0);
    wait_for_earlier_kernels();  // no CTA may end before the kernels before this one
    allow_next_kernel();
    cluster_barrier();  // release: the words are visible to rank 0 after its wait
    int buffer = 0;
    for (int s = 0; s < n_sweeps; ++s)
        for (int piece = 0; piece < pieces; ++piece) {
            buffer ^= 1;
            const bool wrap = piece + 1 == pieces;
            if (!wrap || s + 1 < n_sweeps) produce(wrap ? s + 1 : s, wrap ? 0 : piece + 1, buffer);
            cluster_barrier();
            if (s_ctl[6]) return;  // rank 0's swap wait gave up; it leaves after this barrier too
        }
}

// Path 8: R clusters of two CTAs; rank 0 sweeps chain (cluster index) with every thread,
// rank 1 produces its random words. The cluster shape is compiled in, and checked on entry
// (both CTAs return before any barrier or remote access if it is not 2).
// MAXT = 1024: the lean instance, without the held level-0 units (as sweep_packed_kernel).
template <int DC, bool PIECES, bool REC, int MAXT = 512>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(MAXT, 1)
    sweep_peer_kernel(DevProblem p, long long t0, long long q0, int n_sweeps, int sweeps_per_swap,
                      long long timeout_ns, int n_consumer) {
    extern __shared__ __align__(16) unsigned char smem[];
    cg::cluster_group cluster = cg::this_cluster();
    if (cluster.num_blocks() != 2) {
        if (threadIdx.x == 0) atomicCAS(p.status, 0, PT_ECUDA);
        return;
    }
    const int slot = (int)(blockIdx.x >> 1);
    // no CTA touches the other's shared memory before its wait on this barrier shows that the other
    // has started; arriving first and waiting only then leaves the set-up in between
    cluster_arrive_relaxed();
    if (cluster.block_rank() == 0) {
        if (IndexRule(p.Lmax).wide)
            sweep_packed_body<DC, true, true, false, (MAXT <= 512), true, false, 0, false, PIECES, REC>(
                p, slot, t0, q0, n_sweeps, sweeps_per_swap, timeout_ns, blockDim.x, smem);
        else
            sweep_packed_body<DC, true, false, false, (MAXT <= 512), true, false, 0, false, PIECES, REC>(
                p, slot, t0, q0, n_sweeps, sweeps_per_swap, timeout_ns, blockDim.x, smem);
    } else
        peer_producer<DC, PIECES>(p, slot, t0, n_sweeps, smem);
}

template <int DC, bool PRE, int MAXT, bool BITS = false, bool REC = false>
__global__ void __launch_bounds__(MAXT, 1)
sweep_packed_kernel(DevProblem p, long long t0, long long q0, int n_sweeps, int sweeps_per_swap,
                    long long timeout_ns, int n_consumer) {
    extern __shared__ __align__(16) unsigned char smem[];
    // the held level-0 units do not fit the 64 registers of a 1024-thread block
    if (IndexRule(p.Lmax).wide)
        sweep_packed_body<DC, PRE, true, BITS, (MAXT <= 512), false, false, 0, false, false, REC>(
            p, blockIdx.x, t0, q0, n_sweeps, sweeps_per_swap, timeout_ns, n_consumer, smem);
    else
        sweep_packed_body<DC, PRE, false, BITS, (MAXT <= 512), false, false, 0, false, false, REC>(
            p, blockIdx.x, t0, q0, n_sweeps, sweeps_per_swap, timeout_ns, n_consumer, smem);
}

// Path 4's nibble form (P % 32 == 0, Lmax <= kWordBitsLmax).
template <int DC, int NIB>
__global__ void __launch_bounds__(512, 1)
    sweep_nibble_kernel(DevProblem p, long long t0, long long q0, int n_sweeps, int sweeps_per_swap,
                        long long timeout_ns, int n_consumer) {
    extern __shared__ __align__(16) unsigned char smem[];
    sweep_packed_body<DC, false, false, true, false, false, false, NIB>(p, blockIdx.x, t0, q0, n_sweeps,
                                                                        sweeps_per_swap, timeout_ns, n_consumer, smem);
}

// One copy a thread (DevProblem::slots > 0): a CTA per chain, or (path 9) all of them in one
// cluster, checked on entry as sweep_cluster_kernel does.
template <bool REC>
__global__ void __launch_bounds__(512, 1)
    sweep_copy_kernel(DevProblem p, long long t0, long long q0, int n_sweeps, int sweeps_per_swap,
                      long long timeout_ns, int n_consumer) {
    extern __shared__ __align__(16) unsigned char smem[];
    sweep_packed_body<0, true, false, false, true, false, false, 0, true, false, REC>(
        p, blockIdx.x, t0, q0, n_sweeps, sweeps_per_swap, timeout_ns, n_consumer, smem);
}
template <bool REC>
__global__ void __launch_bounds__(512, 1)
    sweep_copy_cluster_kernel(DevProblem p, long long t0, long long q0, int n_sweeps, int sweeps_per_swap,
                              long long timeout_ns, int n_consumer) {
    extern __shared__ __align__(16) unsigned char smem[];
    cg::cluster_group cluster = cg::this_cluster();
    if (cluster.num_blocks() != (unsigned)p.R || gridDim.x != (unsigned)p.R) {
        if (threadIdx.x == 0) atomicCAS(p.status, 0, PT_ECUDA);
        return;
    }
    sweep_packed_body<0, true, false, false, true, false, true, 0, true, false, REC>(
        p, (int)cluster.block_rank(), t0, q0, n_sweeps, sweeps_per_swap, timeout_ns, n_consumer, smem);
}

// Path 1's word-wise kernel: any even P and any degree up to 32 whose descriptors fit.
__global__ void __launch_bounds__(512, 1)
    sweep_rows_kernel(DevProblem p, long long t0, long long q0, int n_sweeps, int sweeps_per_swap,
                      long long timeout_ns, int n_consumer) {
    extern __shared__ __align__(16) unsigned char smem[];
    if (IndexRule(p.Lmax).wide)
        sweep_packed_body<0, false, true>(p, blockIdx.x, t0, q0, n_sweeps, sweeps_per_swap, timeout_ns, n_consumer,
                                          smem);
    else
        sweep_packed_body<0, false, false>(p, blockIdx.x, t0, q0, n_sweeps, sweeps_per_swap, timeout_ns, n_consumer,
                                           smem);
}

// Path 9: one cluster of R CTAs, CTA r sweeping chain r as paths 2 (PRE = false) and 3 do,
// with the swap mailboxes in shared memory. The cluster shape is set at launch and checked
// on entry: if the cluster is not the whole grid, every CTA returns before any cluster
// barrier or remote access.
template <int DC, bool PRE, bool REC>
__global__ void __launch_bounds__(384, 1)
    sweep_cluster_kernel(DevProblem p, long long t0, long long q0, int n_sweeps, int sweeps_per_swap,
                         long long timeout_ns, int n_consumer) {
    extern __shared__ __align__(16) unsigned char smem[];
    cg::cluster_group cluster = cg::this_cluster();
    if (cluster.num_blocks() != (unsigned)p.R || gridDim.x != (unsigned)p.R) {
        if (threadIdx.x == 0) atomicCAS(p.status, 0, PT_ECUDA);
        return;
    }
    if (IndexRule(p.Lmax).wide)
        sweep_packed_body<DC, PRE, true, false, true, false, true, 0, false, false, REC>(
            p, (int)cluster.block_rank(), t0, q0, n_sweeps, sweeps_per_swap, timeout_ns, n_consumer, smem);
    else
        sweep_packed_body<DC, PRE, false, false, true, false, true, 0, false, false, REC>(
            p, (int)cluster.block_rank(), t0, q0, n_sweeps, sweeps_per_swap, timeout_ns, n_consumer, smem);
}

// Several problems in one cooperative launch (all chains resident at once): block b sweeps
// chain map[b].y of problem map[b].x with the random words computed inline. Swap passes use
// each problem's own mailboxes, so problems never wait for one another.
__global__ void __launch_bounds__(512, 1) sweep_packed_multi_kernel(const MultiProblem* probs, const int2* map) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int2 m = map[blockIdx.x];
    const MultiProblem mp = probs[m.x];
    const bool wide = IndexRule(mp.p.Lmax).wide;
    if (mp.dc == 4 && !wide)
        sweep_packed_body<4, false, false>(mp.p, m.y, mp.t0, mp.q0, mp.n_sweeps, mp.sweeps_per_swap, mp.timeout_ns,
                                           blockDim.x, smem);
    else if (mp.dc == 4)
        sweep_packed_body<4, false, true>(mp.p, m.y, mp.t0, mp.q0, mp.n_sweeps, mp.sweeps_per_swap, mp.timeout_ns,
                                          blockDim.x, smem);
    else if (!wide)
        sweep_packed_body<8, false, false>(mp.p, m.y, mp.t0, mp.q0, mp.n_sweeps, mp.sweeps_per_swap, mp.timeout_ns,
                                           blockDim.x, smem);
    else
        sweep_packed_body<8, false, true>(mp.p, m.y, mp.t0, mp.q0, mp.n_sweeps, mp.sweeps_per_swap, mp.timeout_ns,
                                          blockDim.x, smem);
}

size_t multi_smem_bytes(const DevProblem& p, int dc) { return FastLayout(p, dc, false).total; }

cudaError_t multi_prepare(int threads, size_t smem, int* blocks_per_sm) {
    int dev = 0, max_smem = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(sweep_packed_multi_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, sweep_packed_multi_kernel, threads, smem);
}

cudaError_t launch_multi(const MultiProblem* probs, const int2* map, int n_blocks, int threads, size_t smem,
                         cudaStream_t s) {
    void* args[] = {(void*)&probs, (void*)&map};
    return cudaLaunchCooperativeKernel((const void*)sweep_packed_multi_kernel, dim3(n_blocks), dim3(threads), args,
                                       smem, s);
}

// ------------------------------------------------------------------------- split sweep
// One chain on a cluster of two CTAs (P % 16 == 0), for ladders short enough that a CTA per
// chain would leave SMs idle. CTA h owns copies [h P/2, (h+1) P/2): W = P/16 four-copy words
// per parity. Updates couple a copy only to its Trotter neighbours k +- 1 (Eq. 3), so the
// only copies a CTA needs from its peer are
//   - the peer's first even word (copies h P/2 + P/2 .. +6): recomputed here every sweep,
//     with the same inputs, random words and order as the peer, so bit for bit the same;
//   - the peer's first odd word and its last odd copy as of the previous sweep, which the
//     recomputed word and the own first even word read; the peer writes them into this
//     CTA's shared memory once per sweep, into one of two buffers by sweep parity.
// Each CTA therefore runs the whole level schedule on 2W + 1 words per site, and the two meet
// once per sweep at a cluster barrier, where they also add their halves of dE, dM and the
// flip count. Both CTAs take the swap decision from the same mailbox values; the first CTA
// alone publishes, counts and writes the chain's statistics.
//
// Row layout (bytes) of site i, RB = 8W + 16 per row:
//   [0, 4W+4)         even words 0..W-1 (own), word W = the peer's first even word
//   [4W+4, 8W+4)      odd words 0..W-1 (own)
//   [8W+4, 8W+12)     the peer's first odd word, previous sweep, buffers 0 and 1
//   [8W+12, 8W+14)    the peer's last odd copy, previous sweep, buffers 0 and 1
struct SplitLayout {
    size_t spins, desc, items, loff, thr, acc, red, ctl, xch, rbuf, total;
    int W, RB, Gc;
    __host__ __device__ SplitLayout(const DevProblem& p, int dc, bool pre) {
        const int N = p.N;
        W = p.P / 16;
        RB = 8 * W + 16;
        Gc = W + 1;  // word columns of an even item; odd items use W of them
        size_t o = 0;
        spins = o; o += up16((size_t)N * RB);
        desc = o;  o += (size_t)N * (dc == 4 ? 32 : 48);
        items = o; o += up16((size_t)2 * N * 4);
        loff = o;  o += up16((size_t)(p.n_levels + 1) * 4);
        thr = o;   o += thr_bytes(p, IndexRule(p.Lmax).row_words());
        acc = o;   o += acc_bytes(p);
        red = o;   o += 16;  // the sweep's three sums
        ctl = o;   o += 32;
        xch = o;   o += 64;  // written by the peer: [sweep parity][dE, dM, flips, abort], final abort
        rbuf = o;
        if (pre) o += (size_t)2 * (2 * N) * Gc * 16;
        total = o;
    }
};

size_t split_smem_bytes(const DevProblem& p, int dclass, bool pre) { return SplitLayout(p, dclass, pre).total; }

// Global copy held at byte c of a split row of CTA h, or -1 for padding.
__device__ __forceinline__ int split_copy(int c, int W, int h, int P) {
    const int hs = 4 * W + 4;
    if (c < hs) return 8 * ((h * W + (c >> 2)) % (2 * W)) + 2 * (c & 3);
    if (c < 8 * W + 4) return 8 * (h * W + ((c - hs) >> 2)) + 2 * (c & 3) + 1;
    if (c < 8 * W + 12) return 8 * (((h + 1) * W) % (2 * W)) + 2 * (c & 3) + 1;
    if (c < 8 * W + 14) return (8 * h * W - 1 + P) % P;
    return -1;
}

// Offsets of column g's reads (see UnitOffsets) while the peer's previous-sweep copies sit
// in buffer b.
__device__ __forceinline__ UnitOffsets split_offsets(int g, int W, int b) {
    const uint32_t hs = 4u * W + 4u, w4 = 4u * (uint32_t)g;
    UnitOffsets o;
    o.own[0] = w4;
    o.own[1] = hs + w4;
    o.opp[0] = g < W ? hs + w4 : 8u * W + 4u + 4u * (uint32_t)b;
    o.opp[1] = w4;
    o.edge[0] = g >= 1 ? hs + w4 - 1u : 8u * W + 12u + (uint32_t)b;
    o.edge[1] = w4 + 4u;
    return o;
}

template <int DC, bool PRE, bool WIDE>
__device__ __forceinline__ void split_body(const DevProblem& p, long long t0, long long q0, int n_sweeps,
                                           int sweeps_per_swap, long long timeout_ns, int n_consumer,
                                           unsigned char* smem, cg::cluster_group& cluster) {
    const int h = (int)cluster.block_rank();
    const bool lead = h == 0;
    const int slot = blockIdx.x >> 1;
    const int N = p.N, P = p.P;
    const int tid = threadIdx.x, nt = blockDim.x;
    const SplitLayout L(p, DC, PRE);
    const int W = L.W, RB = L.RB, Gc = L.Gc;
    const int hs = 4 * W + 4;
    int8_t* sp = reinterpret_cast<int8_t*>(smem + L.spins);
    uint32_t* s_desc = reinterpret_cast<uint32_t*>(smem + L.desc);
    uint32_t* s_items = reinterpret_cast<uint32_t*>(smem + L.items);
    int32_t* s_loff = reinterpret_cast<int32_t*>(smem + L.loff);
    uint32_t* s_thr = reinterpret_cast<uint32_t*>(smem + L.thr);
    long long* s_red = reinterpret_cast<long long*>(smem + L.red);
    int* s_ctl = reinterpret_cast<int*>(smem + L.ctl);
    int* s_xch = reinterpret_cast<int*>(smem + L.xch);
    uint4* rbuf = reinterpret_cast<uint4*>(smem + L.rbuf);
    unsigned long long* s_acc = reinterpret_cast<unsigned long long*>(smem + L.acc);
    int8_t* peer_sp = cluster.map_shared_rank(sp, h ^ 1);
    int* peer_xch = cluster.map_shared_rank(s_xch, h ^ 1);
    const int NC = PRE ? n_consumer : nt;
    const bool consumer = tid < NC;
    const int DW = SiteDesc<DC>::DW;

    {
        const int8_t* src = p.spins + (size_t)slot * p.slot_stride;
        for (int x = tid; x < N * RB; x += nt) {
            const int i = x / RB, c = x - i * RB;
            const int k = split_copy(c, W, h, P);
            sp[x] = k >= 0 ? src[(size_t)i * P + k] : (int8_t)0;
        }
        // descriptors with the row offsets rescaled from P to RB bytes per row
        for (int x = tid; x < N * DW; x += nt) {
            const int f = x % DW;
            uint32_t v = p.desc[x];
            const bool is_row = DC == 4 ? ((f >= 1 && f <= 3) || f == 7) : (f == 3 || (f >= 4 && f <= 10));
            if (is_row) v = (v / (uint32_t)P) * (uint32_t)RB;
            s_desc[x] = v;
        }
        for (int x = tid; x < 2 * N; x += nt) s_items[x] = p.items[x];
        for (int x = tid; x <= p.n_levels; x += nt) s_loff[x] = p.level_off[x];
        for (int x = tid; x < 16; x += nt) s_xch[x] = 0;
    }
    int rung = p.rung_of_slot[slot];
    load_thr_columns(p, s_thr, rung, tid, nt);
    if (p.acc_in_smem)
        for (int x = tid; x < p.R * kAccCount; x += nt) s_acc[x] = 0ull;
    long long E = p.E[slot], M = p.M[slot];  // meaningful in thread 0 only

    const PhiloxKey key = philox_schedule(p.key0, p.key1);
    const UnitRule<WIDE> rule(p.Lmax);
    const uint32_t thr0 = thr_base<WIDE>((uint32_t)L.thr, p.Lmax);
    const uint32_t thr_step = p.tables_in_smem ? 4u * (uint32_t)IndexRule(p.Lmax).row_words() : 0u;
    uint32_t thr_c = thr0 + thr_step * (uint32_t)rung;
    const int n_items = 2 * N;
    const int lane = tid & 31;
    if (tid == 0) {
        s_ctl[4] = -1;  // partner rung of the pending swap pass
        s_ctl[5] = 0;   // this CTA's swap wait gave up
        s_ctl[6] = 0;   // either CTA's wait gave up (known at the last cluster barrier)
        int* s_sum = reinterpret_cast<int*>(s_red);
        s_sum[0] = s_sum[1] = s_sum[2] = 0;
    }
    // every CTA of the cluster is running and initialised before any shared-memory exchange
    cluster_barrier();

    // random words of sweep t for this CTA's columns (global chunk (hW + g) mod 2W)
    auto produce = [&](uint4* buf, uint32_t t) {
        const int ptid = tid - NC, np = nt - NC;
        const int pg = ptid % Gc, pstep = np / Gc;
        if (ptid / Gc >= pstep) return;
        const uint32_t gg = (uint32_t)((h * W + pg) % (2 * W));
        for (int q = ptid / Gc; q < n_items; q += pstep) {
            const uint32_t it = s_items[q];
            if ((it & 1u) && pg == W) continue;
            const uint4 r = philox(make_uint4(t, it >> 1, (uint32_t)slot, ((it & 1u) << 24) | gg), key);
            buf[q * Gc + pg] = make_uint4(min(r.x, 0xFFFFFFFEu), min(r.y, 0xFFFFFFFEu), min(r.z, 0xFFFFFFFEu),
                                          min(r.w, 0xFFFFFFFEu));
        }
    };
    if (PRE && !consumer) produce(rbuf, (uint32_t)t0);
    __syncthreads();

    // consumers: a fixed column g_own per thread, items q_lane, q_lane + q_step, ... of a level
    const int g_own = tid % Gc, q_lane = tid / Gc, q_step = NC / Gc;
    const bool lane_ok = consumer && q_lane < q_step;
    const bool ghost_col = g_own == W;  // the recomputed peer word: its flips are the peer's
    const uint32_t gg_own = (uint32_t)((h * W + g_own) % (2 * W));  // its chunk in the whole chain
    // level 0 of the next sweep during the swap wait: units v, v + (NC - 32) of the level
    // (v = tid - 32), so that warp 0 is free to poll the partner's mailbox
    const int units0 = (s_loff[1] - s_loff[0]) * Gc;
    const bool spec_ok = p.tables_in_smem && NC > 32 && units0 <= 2 * (NC - 32);
    int sq[2], sg[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int u = (tid - 32) + k * (NC - 32);
        sg[k] = u % Gc;
        sq[k] = (tid >= 32 && consumer && u < units0) ? s_loff[0] + u / Gc : -1;
    }
    bool spec_done = false;
    FlipSums lev_sums, pre_sums;  // this sweep's own units in the levels; the level-0 units applied early
    lev_sums.clear();
    pre_sums.clear();
    SwapSide side;
    side.active = 0;
    const uint32_t qmod0 = (uint32_t)(q0 % kTagPeriod);
    int since_pass = 0, next_pass = 0;  // thread 0
    long long sE = 0, sM = 0, sF = 0;   // thread 0: this CTA's half of the sweep's changes

    for (int s = 0; s < n_sweeps; ++s) {
        const uint32_t t = (uint32_t)(t0 + s);
        const int b = s & 1;
        const bool dead = (s_ctl[5] | s_ctl[6]) != 0;
        if (consumer) {
            if (!dead) {
                const uint4* rb = rbuf + (size_t)b * n_items * Gc;
                const UnitOffsets off = split_offsets(g_own, W, b);
                if (!spec_done) pre_sums.clear();
                lev_sums.clear();
                for (int lev = spec_done ? 1 : 0; lev < p.n_levels; ++lev) {
                    if (lane_ok) {
                        const int end = s_loff[lev + 1];
                        for (int q = s_loff[lev] + q_lane; q < end; q += q_step) {
                            const uint32_t it = s_items[q];
                            if (ghost_col && (it & 1u)) continue;
                            const UnitEval<1> e = unit_eval<DC, 1, PRE, WIDE>(sp, s_desc, it, off, rb + q * Gc + g_own, t,
                                                                        (uint32_t)slot, gg_own, rule, key);
                            uint32_t F[1];
                            unit_flips<1, PRE, WIDE>(e, smem, rule, thr_c, F);
                            unit_commit<1>(e, F, lev_sums);
                        }
                    }
                    named_barrier(1, NC);
                }
                if (ghost_col) lev_sums.clear();
                FlipSums m = lev_sums;
                m.add(pre_sums);
                const int dE = __reduce_add_sync(0xFFFFFFFFu, m.dE(rule));
                const int dM = __reduce_add_sync(0xFFFFFFFFu, m.dM(rule));
                const int dF = __reduce_add_sync(0xFFFFFFFFu, m.flips());
                int* s_sum = reinterpret_cast<int*>(s_red);
                if (lane == 0) {
                    atomicAdd(s_sum + 0, dE);
                    atomicAdd(s_sum + 1, dM);
                    atomicAdd(s_sum + 2, dF);
                }
                named_barrier(1, NC);
                // the peer's next sweep reads this sweep's first odd word and last odd copy
                const int bn = b ^ 1;
                for (int i = tid; i < N; i += NC) {
                    const int8_t* r = sp + (size_t)i * RB;
                    int8_t* pr = peer_sp + (size_t)i * RB;
                    *reinterpret_cast<uint32_t*>(pr + 8 * W + 4 + 4 * bn) = *reinterpret_cast<const uint32_t*>(r + hs);
                    pr[8 * W + 12 + bn] = r[hs + 4 * W - 1];
                }
            }
            if (tid == 0) {
                int* s_sum = reinterpret_cast<int*>(s_red);
                sE = s_sum[0];
                sM = s_sum[1];
                sF = s_sum[2];
                s_sum[0] = s_sum[1] = s_sum[2] = 0;
                int* x = peer_xch + 4 * b;
                x[0] = (int)sE;
                x[1] = (int)sM;
                x[2] = (int)sF;
                x[3] = s_ctl[5];
            }
        } else if (PRE && !dead && s + 1 < n_sweeps) {
            produce(rbuf + (size_t)(b ^ 1) * n_items * Gc, t + 1u);
        }
        // both halves of the sweep are done, the exchanged words and sums are visible and
        // the next sweep's random words are complete
        cluster_barrier();
        if (tid == 0) {
            const int* x = s_xch + 4 * b;
            if (x[3] || s_ctl[5]) s_ctl[6] = 1;
            if (!s_ctl[6]) {
                int pass = -1;
                if (sweeps_per_swap > 0 && ++since_pass == sweeps_per_swap) {
                    since_pass = 0;
                    pass = next_pass++;
                }
                side = eos_publish(p, rung, E, M, sE + x[0], sM + x[1], pass, q0, qmod0, lead);
                sF += x[2];
                s_ctl[4] = side.active ? side.partner : -1;
            }
        }
        __syncthreads();
        if (s_ctl[6] || !consumer) continue;

        // level 0 of sweep s + 1 under both candidate rungs
        const bool spec = spec_ok && s + 1 < n_sweeps;
        const int prung = s_ctl[4];
        UnitEval<1> ev[2];
        uint32_t Fa[2] = {0u, 0u}, Fb[2] = {0u, 0u};
        bool valid[2] = {false, false};
        if (spec) {
            const uint4* rb1 = rbuf + (size_t)(b ^ 1) * n_items * Gc;
            const uint32_t thr_b = prung >= 0 ? thr0 + thr_step * (uint32_t)prung : thr_c;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                if (sq[k] < 0) continue;
                const uint32_t it = s_items[sq[k]];
                valid[k] = !((it & 1u) && sg[k] == W);
                if (valid[k]) {
                    ev[k] = unit_eval<DC, 1, PRE, WIDE>(sp, s_desc, it, split_offsets(sg[k], W, b ^ 1),
                                                  rb1 + sq[k] * Gc + sg[k], t + 1u, (uint32_t)slot,
                                                  (uint32_t)((h * W + sg[k]) % (2 * W)), rule, key);
                    unit_flips<1, PRE, WIDE>(ev[k], smem, rule, thr_c, Fa + k);
                    if (prung >= 0)
                        unit_flips<1, PRE, WIDE>(ev[k], smem, rule, thr_b, Fb + k);
                    else
                        Fb[k] = Fa[k];
                }
            }
        }
        if (tid == 0) {
            if (lead) eos_stats(p, p.acc_in_smem ? s_acc : p.acc, rung, E, M, sF);
            int abort_flag = 0;
            s_ctl[2 * b] = eos_decide(p, side, rung, E, M, timeout_ns, key, &abort_flag, lead);
            if (abort_flag) s_ctl[5] = 1;
        }
        named_barrier(1, NC);
        if (s_ctl[5]) continue;  // the next sweep is skipped; the cluster barriers go on
        const int nr = s_ctl[2 * b];
        const bool moved = nr != rung;
        if (moved) {
            rung = nr;
            if (!p.tables_in_smem) load_thr_columns(p, s_thr, rung, tid, NC);
            thr_c = thr0 + thr_step * (uint32_t)rung;
        }
        spec_done = spec;
        if (spec) {
            pre_sums.clear();
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                if (!valid[k]) continue;
                const uint32_t F[1] = {moved ? Fb[k] : Fa[k]};
                FlipSums unit;
                unit.clear();
                unit_commit<1>(ev[k], F, unit);
                if (sg[k] != W) pre_sums.add(unit);
            }
        }
        named_barrier(1, NC);
    }
    // both CTAs agree whether a swap wait gave up before either writes anything back
    if (tid == 0) peer_xch[8] = s_ctl[5] | s_ctl[6];
    cluster_barrier();
    if (tid == 0 && (s_xch[8] || s_ctl[5] || s_ctl[6])) s_ctl[6] = 1;
    __syncthreads();
    if (s_ctl[6]) return;
    if (lead) flush_acc(p, s_acc, tid, nt);
    {
        int8_t* dst = p.spins + (size_t)slot * p.slot_stride;
        for (int x = tid; x < N * RB; x += nt) {
            const int i = x / RB, c = x - i * RB;
            if (c < 4 * W || (c >= hs && c < hs + 4 * W)) dst[(size_t)i * P + split_copy(c, W, h, P)] = sp[x];
        }
    }
    if (tid == 0 && lead) {
        p.E[slot] = E;
        p.M[slot] = M;
        p.rung_of_slot[slot] = rung;
        p.slot_of_rung[rung] = slot;
    }
}

// MAXT = 640: the lean instance. Its 96 registers a thread (98 otherwise) let one more CTA of a small
// block be resident (160 threads: 4 an SM instead of 3); with that limit on every launch the kernels
// took 5 to 20 % longer (N=200, degree 7, P=64, R=70: 6.83 -> 8.19 us per sweep).
template <int DC, bool PRE, int MAXT = 512>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(MAXT, 1)
    sweep_split_kernel(DevProblem p, long long t0, long long q0, int n_sweeps, int sweeps_per_swap,
                       long long timeout_ns, int n_consumer) {
    extern __shared__ __align__(16) unsigned char smem[];
    wait_for_earlier_kernels();
    allow_next_kernel();
    cg::cluster_group cluster = cg::this_cluster();
    // the cluster shape is compiled in; should a launch ever run without it, no CTA touches
    // a peer's shared memory or waits at a cluster barrier
    if (cluster.num_blocks() != 2) {
        if (threadIdx.x == 0) atomicCAS(p.status, 0, PT_ECUDA);
        return;
    }
    if (IndexRule(p.Lmax).wide)
        split_body<DC, PRE, true>(p, t0, q0, n_sweeps, sweeps_per_swap, timeout_ns, n_consumer, smem, cluster);
    else
        split_body<DC, PRE, false>(p, t0, q0, n_sweeps, sweeps_per_swap, timeout_ns, n_consumer, smem, cluster);
}

// ------------------------------------------------------------------------- init / energy
// Initial spins: copy k of site i of chain rho is -1 iff bit 31 of word k%4 of
// philox((0, i, rho, INIT<<28 | k/4)) is set.
__global__ void init_kernel(DevProblem p) {
    const int slot = blockIdx.x;
    const int P4 = (p.P + 3) >> 2;
    const PhiloxKey key = philox_schedule(p.key0, p.key1);
    int8_t* dst = p.spins + (size_t)slot * p.slot_stride;
    for (int x = threadIdx.x; x < p.N * P4; x += blockDim.x) {
        const int i = x / P4, g4 = x - i * P4;
        const uint4 u = philox(make_uint4(0u, (uint32_t)i, (uint32_t)slot, (kTagInit << 28) | (uint32_t)g4), key);
        const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int k = 4 * g4 + b;
            if (k < p.P) dst[(size_t)i * p.P + k] = (w[b] >> 31) ? (int8_t)-1 : (int8_t)1;
        }
    }
    if (threadIdx.x == 0) {
        p.rung_of_slot[slot] = slot;
        p.slot_of_rung[slot] = slot;
    }
}

// E = sum_k E(s^k) and M = sum_k sum_i s_i^k s_i^{k+1} of every chain from scratch.
__global__ void energy_kernel(DevProblem p) {
    __shared__ long long red[2][32];
    const int slot = blockIdx.x;
    const int8_t* sp = p.spins + (size_t)slot * p.slot_stride;
    long long e = 0, m = 0;
    for (int x = threadIdx.x; x < p.N * p.P; x += blockDim.x) {
        const int i = x / p.P, k = x - i * p.P;
        const int si = sp[x];
        int f = p.h[i];
        for (int d = 0; d < p.dmax; ++d) {
            const uint32_t e8 = p.nbr[(size_t)i * p.dmax + d];
            const int j = (int)(e8 >> 8);
            if (j > i) f += (int)(int8_t)(e8 & 0xFFu) * (int)sp[(size_t)j * p.P + k];
        }
        e += (long long)si * f;
        m += (long long)si * sp[(size_t)i * p.P + ((k + 1 == p.P) ? 0 : k + 1)];
    }
    for (int o = 16; o > 0; o >>= 1) {
        e += __shfl_xor_sync(0xFFFFFFFFu, e, o);
        m += __shfl_xor_sync(0xFFFFFFFFu, m, o);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) {
        red[0][warp] = e;
        red[1][warp] = m;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        long long se = 0, sm = 0;
        for (int w = 0; w < (int)((blockDim.x + 31) >> 5); ++w) {
            se += red[0][w];
            sm += red[1][w];
        }
        p.E[slot] = se;
        p.M[slot] = sm;
    }
}

// ------------------------------------------------------------------------- swap / copies
// One swap pass q with chains in place (state already in global memory).
__global__ void swap_kernel(DevProblem p, long long q) {
    const PhiloxKey key = philox_schedule(p.key0, p.key1);
    allow_next_kernel();  // the next sweeps' set-up waits for this kernel all the same
    // the first pair's coefficients and random word depend on no earlier kernel either
    const int rl0 = (int)(q & 1) + 2 * (int)threadIdx.x;
    double ca = 0.0, cc = 0.0;
    uint32_t word = 0u;
    auto pair_inputs = [&](int rl) {
        ca = p.coef[rl];
        cc = p.coef[(p.R - 1) + rl];
        word = swap_word((uint32_t)q, (uint32_t)rl, key);
    };
    if (rl0 + 1 < p.R) pair_inputs(rl0);
    wait_for_earlier_kernels();
    for (int rl = rl0; rl + 1 < p.R; rl += 2 * (int)blockDim.x) {
        if (rl != rl0) pair_inputs(rl);
        const int X = p.slot_of_rung[rl], Y = p.slot_of_rung[rl + 1];
        const bool acc = swap_accept_fast_by(p.E[X], p.E[Y], p.M[X], p.M[Y], ca, cc, [&] { return word; },
                                             p.exact_swaps != 0);
        p.swap_stats[2 * rl] += 1ull;
        if (acc) {
            p.swap_stats[2 * rl + 1] += 1ull;
            p.slot_of_rung[rl] = Y;
            p.slot_of_rung[rl + 1] = X;
            p.rung_of_slot[X] = rl + 1;
            p.rung_of_slot[Y] = rl;
        }
    }
}

__global__ void gather_kernel(DevProblem p, int8_t* out) {
    const int r = blockIdx.x;
    const int8_t* src = p.spins + (size_t)p.slot_of_rung[r] * p.slot_stride;
    int8_t* dst = out + (size_t)r * p.N * p.P;
    const int n = p.N * p.P;
    if ((n & 15) == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0) {
        // 16 bytes a thread: chains start on 16-byte boundaries (slot_stride), and so does
        // every rung's output row when a chain is a whole number of 16-byte words
        const uint4* s4 = reinterpret_cast<const uint4*>(src);
        uint4* d4 = reinterpret_cast<uint4*>(dst);
        for (int x = threadIdx.x; x < (n >> 4); x += blockDim.x) d4[x] = s4[x];
    } else {
        for (int x = threadIdx.x; x < n; x += blockDim.x) dst[x] = src[x];
    }
}

__global__ void scatter_kernel(DevProblem p, const int8_t* in) {
    const int r = blockIdx.x;
    int8_t* dst = p.spins + (size_t)p.slot_of_rung[r] * p.slot_stride;
    const int8_t* src = in + (size_t)r * p.N * p.P;
    for (int x = threadIdx.x; x < p.N * p.P; x += blockDim.x) dst[x] = src[x];
}

// ------------------------------------------------------------------------- launchers
// The instances of a neighbour class with (REC) and without records.
template <int DC, bool REC>
static const void* class_fn(const LaunchPlan& plan) {
    if (plan.path == kPathPeer) {
        if (plan.pieces > 1) return (const void*)sweep_peer_kernel<DC, true, REC>;
        return (const void*)sweep_peer_kernel<DC, false, REC>;
    }
    if (plan.path == kPathCluster)
        return plan.n_consumer < plan.threads ? (const void*)sweep_cluster_kernel<DC, true, REC>
                                              : (const void*)sweep_cluster_kernel<DC, false, REC>;
    const bool pre = plan.path == kPathPacked;
    // (at 64 registers the descriptors' loop alone is no faster: one instance serves both)
    if (plan.threads > 512 || plan.lean)
        return pre ? (const void*)sweep_packed_kernel<DC, true, 1024, false, true>
                   : (const void*)sweep_packed_kernel<DC, false, 1024, false, true>;
    return pre ? (const void*)sweep_packed_kernel<DC, true, 512, false, REC>
               : (const void*)sweep_packed_kernel<DC, false, 512, false, REC>;
}
static const void* sweep_fn(const LaunchPlan& plan) {
    if (plan.copy && plan.path == kPathCluster)
        return plan.records ? (const void*)sweep_copy_cluster_kernel<true>
                            : (const void*)sweep_copy_cluster_kernel<false>;
    if (plan.copy) return plan.records ? (const void*)sweep_copy_kernel<true> : (const void*)sweep_copy_kernel<false>;
    if (plan.path == kPathClassical) {
        switch (plan.dclass) {
            case 4: return (const void*)sweep_classical_kernel<4>;
            case 8: return (const void*)sweep_classical_kernel<8>;
            default: return (const void*)sweep_classical_kernel<32>;
        }
    }
    if (plan.path == kPathGeneric && plan.rows) return (const void*)sweep_rows_kernel;
    if (plan.path == kPathGeneric) {
        switch (plan.dclass) {
            case 4: return (const void*)sweep_kernel<4>;
            case 8: return (const void*)sweep_kernel<8>;
            default: return (const void*)sweep_kernel<32>;
        }
    }
    if (plan.path == kPathPeer && plan.lean && plan.pieces <= 1)  // (without records)
        return plan.dclass == 4 ? (const void*)sweep_peer_kernel<4, false, false, 1024>
                                : (const void*)sweep_peer_kernel<8, false, false, 1024>;
    if (plan.path == kPathSplit)
        return plan.dclass == 4 ? (const void*)sweep_split_kernel<4, true> : (const void*)sweep_split_kernel<8, true>;
    if (plan.path == kPathSplitInline && plan.dclass == 4 && plan.lean)
        return (const void*)sweep_split_kernel<4, false, 640>;
    if (plan.path == kPathSplitInline)
        return plan.dclass == 4 ? (const void*)sweep_split_kernel<4, false> : (const void*)sweep_split_kernel<8, false>;
    if (plan.path == kPathBits && plan.nibble) {
        if (plan.dclass == 4) return (const void*)sweep_nibble_kernel<4, 3>;
        return plan.nibble == 6 ? (const void*)sweep_nibble_kernel<8, 6> : (const void*)sweep_nibble_kernel<8, 7>;
    }
    if (plan.path == kPathBits) {
        if (plan.threads > 512 || plan.lean)
            return plan.dclass == 4 ? (const void*)sweep_packed_kernel<4, false, 1024, true>
                                    : (const void*)sweep_packed_kernel<8, false, 1024, true>;
        return plan.dclass == 4 ? (const void*)sweep_packed_kernel<4, false, 512, true>
                                : (const void*)sweep_packed_kernel<8, false, 512, true>;
    }
    if (plan.dclass == 4) return plan.records ? class_fn<4, true>(plan) : class_fn<4, false>(plan);
    return plan.records ? class_fn<8, true>(plan) : class_fn<8, false>(plan);
}

// The dynamic shared-memory limit is a per-function attribute shared by every context, so
// it is raised once to the device's opt-in maximum rather than to one context's size.
cudaError_t prepare_sweep_kernel(const LaunchPlan& plan) {
    int dev = 0, max_smem = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    if (plan.path == kPathCluster || plan.path == kPathClassical) {
        // clusters of up to 16 CTAs (above 8 is a non-portable size)
        e = cudaFuncSetAttribute(sweep_fn(plan), cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
    }
    return cudaFuncSetAttribute(sweep_fn(plan), cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
}

cudaError_t sweep_kernel_occupancy(const DevProblem& p, const LaunchPlan& plan, int* blocks_per_sm) {
    (void)p;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, sweep_fn(plan), plan.threads,
                                                         plan.smem_bytes);
}

// The split kernel's launch: R clusters of two CTAs (the cluster shape is compiled into the
// kernel); cooperative when swap passes run inside.
static cudaLaunchConfig_t split_config(const DevProblem& p, const LaunchPlan& plan, bool cooperative,
                                       cudaStream_t s, cudaLaunchAttribute* attr) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * p.R);
    cfg.blockDim = dim3(plan.threads);
    cfg.dynamicSmemBytes = plan.smem_bytes;
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cooperative ? 1 : 0;
    return cfg;
}

// Path 9's launch: one cluster of all R CTAs; path 10's: one cluster of ceil(R / C) CTAs.
static cudaLaunchConfig_t cluster_config(const DevProblem& p, const LaunchPlan& plan, cudaStream_t s,
                                         cudaLaunchAttribute* attr) {
    const int ctas = plan.path == kPathClassical ? (p.R + plan.chains_per_cta - 1) / plan.chains_per_cta : p.R;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(plan.threads);
    cfg.dynamicSmemBytes = plan.smem_bytes;
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)ctas;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

cudaError_t sweep_resident_chains(const DevProblem& p, const LaunchPlan& plan, long long* chains) {
    *chains = 0;
    if (plan.path == kPathCluster || plan.path == kPathClassical) {
        const int ctas = plan.path == kPathClassical ? (p.R + plan.chains_per_cta - 1) / plan.chains_per_cta : p.R;
        if (ctas > 16) return cudaSuccess;
        cudaLaunchAttribute attr[1];
        cudaLaunchConfig_t cfg = cluster_config(p, plan, 0, attr);
        int clusters = 0;
        cudaError_t e = cudaOccupancyMaxActiveClusters(&clusters, sweep_fn(plan), &cfg);
        if (e == cudaSuccess) *chains = (long long)clusters * p.R;
        return e;
    }
    if (plan.path == kPathSplit || plan.path == kPathSplitInline || plan.path == kPathPeer) {
        cudaLaunchAttribute attr[2];
        cudaLaunchConfig_t cfg = split_config(p, plan, false, 0, attr);
        int clusters = 0;
        cudaError_t e = cudaOccupancyMaxActiveClusters(&clusters, sweep_fn(plan), &cfg);
        if (e == cudaSuccess) *chains = clusters;
        return e;
    }
    int dev = 0, n_sm = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = sweep_kernel_occupancy(p, plan, &per_sm);
    if (e == cudaSuccess) *chains = (long long)per_sm * n_sm;
    return e;
}

// The launch attribute of LaunchPlan::overlap: 1 where it was appended (not under capture, where
// the graph would get edges of a kind its user may not expect).
static unsigned overlap_attr(bool overlap, cudaStream_t s, cudaLaunchAttribute* attr) {
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (!overlap || cudaStreamIsCapturing(s, &capture) != cudaSuccess || capture != cudaStreamCaptureStatusNone) {
        if (overlap) (void)cudaGetLastError();
        return 0;
    }
    attr->id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr->val.programmaticStreamSerializationAllowed = 1;
    return 1;
}

cudaError_t launch_sweeps(const DevProblem& p, const LaunchPlan& plan, long long t0, long long q0,
                          int n_sweeps, int sweeps_per_swap, long long timeout_ns, bool cooperative,
                          cudaStream_t s) {
    if ((plan.records != 0) != (p.records != 0)) return cudaErrorInvalidValue;  // the kernel's layout
    DevProblem pp = p;
    // the last argument: consumer threads, or (path 10) chains per CTA
    int n_consumer = plan.path == kPathClassical ? plan.chains_per_cta : plan.n_consumer;
    void* args[] = {&pp, &t0, &q0, &n_sweeps, &sweeps_per_swap, &timeout_ns, &n_consumer};
    const void* fn = sweep_fn(plan);
    if (plan.path == kPathCluster || plan.path == kPathClassical) {
        // one cluster holds every chain, so the swap passes never need a cooperative launch
        cudaLaunchAttribute attr[2];
        cudaLaunchConfig_t cfg = cluster_config(p, plan, s, attr);
        cfg.numAttrs += overlap_attr(plan.overlap, s, attr + cfg.numAttrs);
        const cudaError_t e = cudaLaunchKernelExC(&cfg, fn, args);
        if (e != cudaSuccess) (void)cudaGetLastError();
        return e;
    }
    if (plan.path == kPathSplit || plan.path == kPathSplitInline || plan.path == kPathPeer) {
        cudaLaunchAttribute attr[2];
        cudaLaunchConfig_t cfg = split_config(p, plan, cooperative, s, attr);
        if (!cooperative) cfg.numAttrs += overlap_attr(plan.overlap, s, attr);
        const cudaError_t e = cudaLaunchKernelExC(&cfg, fn, args);
        if (e != cudaSuccess) (void)cudaGetLastError();  // a rejected launch leaves no error for the next one
        return e;
    }
    if (cooperative)
        return cudaLaunchCooperativeKernel(fn, dim3(p.R), dim3(plan.threads), args, plan.smem_bytes, s);
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(p.R);
    cfg.blockDim = dim3(plan.threads);
    cfg.dynamicSmemBytes = plan.smem_bytes;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = overlap_attr(plan.overlap, s, attr);
    const cudaError_t e = cudaLaunchKernelExC(&cfg, fn, args);
    if (e != cudaSuccess) (void)cudaGetLastError();
    return e;
}

cudaError_t launch_init(const DevProblem& p, cudaStream_t s) {
    init_kernel<<<p.R, 256, 0, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_energy(const DevProblem& p, cudaStream_t s) {
    energy_kernel<<<p.R, 256, 0, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_swap(const DevProblem& p, long long q, cudaStream_t s, bool overlap) {
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1);
    cfg.blockDim = dim3(256);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = overlap_attr(overlap, s, attr);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, swap_kernel, p, q);
    if (e != cudaSuccess) (void)cudaGetLastError();
    return e;
}

cudaError_t launch_gather_state(const DevProblem& p, int8_t* out, cudaStream_t s) {
    gather_kernel<<<p.R, 256, 0, s>>>(p, out);
    return cudaGetLastError();
}

cudaError_t launch_scatter_state(const DevProblem& p, const int8_t* in, cudaStream_t s) {
    scatter_kernel<<<p.R, 256, 0, s>>>(p, in);
    return cudaGetLastError();
}

}  // namespace ptq
