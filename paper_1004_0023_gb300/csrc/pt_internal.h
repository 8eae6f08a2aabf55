// pt_internal.h -- structures shared by the host side (pt_host.cu) and the kernels
// (pt_kernels.cu) of the PT-QMC library. Not part of the public ABI (include/pt.h).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "pt.h"

namespace ptq {

// Stream tags in the top nibble of Philox counter word 3.
constexpr uint32_t kTagFlip = 0u;
constexpr uint32_t kTagSwap = 1u;
constexpr uint32_t kTagInit = 2u;

// One (pass, rung) mailbox of the in-kernel swap: two self-validating 64-bit words that the
// chain on rung r writes after the sweep preceding pass q,
//   a = E << 24 | tag,   b = (uint32)M << 32 | tag,   tag = q mod (2^24 - 1) + 1 (never 0),
// so a partner that sees the pass's tag in both words has a consistent (E, M) from one round
// trip of two relaxed loads. |E| < 2^39 and |M| < 2^31 are checked at create; the host
// clears the mailboxes before a tag value could repeat.
struct alignas(16) Mailbox {
    unsigned long long a;
    unsigned long long b;
};
constexpr long long kTagPeriod = 16777215ll;
constexpr int kMaxChunks = 8;          // path 8: pieces of a sweep whose random words are made at a time
constexpr int kClusterMailPasses = 4;  // path 9: swap passes whose mailboxes each CTA holds at once

// Multiplicative inverses modulo 2^32 (Newton's iteration doubles the correct low bits).
constexpr uint32_t inverse32(uint32_t a) {
    uint32_t x = a;  // 3 correct bits for odd a
    for (int k = 0; k < 4; ++k) x *= 2u - a * x;
    return x;
}
constexpr uint32_t kInv127 = inverse32(127u), kInv255 = inverse32(255u);
static_assert(kInv127 * 127u == 1u && kInv255 * 255u == 1u, "inverses modulo 2^32");

// How the packed kernels index their threshold rows. A row in shared memory holds three
// columns of S entries, entry col S + (L + Lmax) with col = m/2 + 1 (the public layout
// [L + Lmax][col] is rearranged when a row is loaded). For Lmax <= 41 the whole entry index
// fits one byte per copy (at most 6 Lmax + 4 = 250) and is formed for four copies at once;
// S = 2 Lmax + 2 is even then, because the Trotter differences come doubled. Larger Lmax
// ("wide") combine L and the column per copy, with S a multiple of 16 so that a column's
// stride is a byte multiplier.
struct IndexRule {
    int Lmax, S, bias;   // bias: added to every byte L + Lmax, so that no column makes it negative
    bool wide;
    uint32_t kM;         // x -> 2 Lmax + 2 bias - x for the bytes under a sign mask m: (x ^ m) + kM m
    __host__ __device__ explicit IndexRule(int Lmax_) : Lmax(Lmax_) {
        wide = Lmax > 41;
        S = wide ? (2 * Lmax + 16) / 16 * 16 : 2 * Lmax + 2;
        bias = wide ? 0 : 2 * S;
        kM = (uint32_t)(2 * Lmax + 2 * bias - 255) * kInv255;
    }
    __host__ __device__ int zero() const { return Lmax + bias; }  // the byte of L = 0
    __host__ __device__ int row_words() const { return 3 * S; }
};

constexpr int kWordBitsLmax = 31;  // bit words: 4 (2 Lmax) fits a byte

// Per-rung statistics, in this order, as unsigned 64-bit two's-complement sums.
enum { kAccN = 0, kAccE, kAccE2, kAccM, kAccM2, kAccFlip, kAccCount };

// Device view of one PT problem. All pointers are device pointers.
struct DevProblem {
    // instance (read-only)
    const uint32_t* nbr;       // [N][dmax]: (j << 8) | (uint8_t)J; padding has J = 0, j = i
    const int8_t* h;           // [N]
    const uint32_t* items;     // [2N] (i << 1) | parity, grouped by dependency level
    const int32_t* level_off;  // [n_levels + 1]
    const uint32_t* desc;      // [N][8 or 12] packed-path site descriptors
    const uint32_t* thr;       // [R][nL*3] Metropolis thresholds
    const double* coef;        // [2(R-1)] a_r then c_r
    // state
    int8_t* spins;             // [R slots][slot_stride] int8, copy index fastest
    long long* E;              // [slot]
    long long* M;              // [slot]
    int32_t* rung_of_slot;     // [slot]
    int32_t* slot_of_rung;     // [rung]
    unsigned long long* acc;   // [rung][kAccCount]
    unsigned long long* swap_stats;  // [pair][2] attempts, accepts
    Mailbox* mbox;             // [max_passes][R]
    int* status;               // 0 or a PT_E* code set by a kernel
    int N, P, R, Lmax, nL3, n_levels;
    int dmax;                  // row stride of `nbr` (4, 8 or 32)
    int slot_stride;           // bytes between slots in `spins` (multiple of 16)
    int withhold_rung;         // test hook: rung whose chain never publishes (-1 = off)
    int acc_in_smem;           // 1: per-rung statistics gathered in shared memory per launch
    int tables_in_smem;        // 1: every rung's threshold row resident in shared memory
    int slots;                 // path 1: neighbour slots of a site descriptor (a multiple of 4) when the
                               // word-wise kernel runs, 0: the byte-wise one
    // Path 8: a sweep's random words come in n_chunks pieces, the words of levels chunk_level[c] to
    // chunk_level[c + 1] - 1 (at most chunk_items updates); n_chunks <= 1: the whole sweep at once.
    int n_chunks, chunk_items;
    int16_t chunk_level[kMaxChunks + 1];
    int records;               // 1: per-update records in schedule order in shared memory (see record_words)
    int nibble;                // path 4: 1 = the nibble form of the bit-packed chain
    int exact_swaps;           // test hook: 1 = always take the FP64 swap decision
    uint32_t key0, key1;
};

// Sweep kernel variants: any shape (word-wise, one copy a thread, or byte-wise), packed with Philox
// inline, packed with the random words produced one sweep ahead by dedicated warps, bit-packed, and
// the produced-words kernel with each chain split over a cluster of two CTAs.
// Path 7 runs the batched kernel on the one problem: all chains packed on the CTAs of one
// cluster (thread groups per chain), resident in shared memory, swaps in shared memory.
enum {
    kPathGeneric = 1,
    kPathPackedInline = 2,
    kPathPacked = 3,
    kPathBits = 4,
    kPathSplit = 5,
    kPathSplitInline = 6,
    kPathPackedChains = 7,
    kPathPeer = 8,  // path 3's sweep on every thread of rank 0 of a two-CTA cluster; rank 1 makes its random words
    kPathCluster = 9,   // paths 2 / 3 with every chain's CTA in one cluster; swap mailboxes in shared memory
    kPathClassical = 10  // P = 1: chains packed several to a CTA, one cluster, swap mailboxes in shared memory
};

struct LaunchPlan {
    int path;            // kPath*
    int threads;         // threads per CTA
    int n_consumer;      // threads running the levels (the rest produce random words)
    int dclass;          // padded neighbour slots the kernel is built for
    size_t smem_bytes;   // dynamic shared memory per CTA
    int cluster = 1;     // path 7: CTAs in the one cluster
    int group_threads = 0;  // path 7: threads sweeping one chain
    int mail_smem = 1;      // path 7: the swap mailboxes in shared memory
    int thr_resident = 0;   // path 7: every rung's threshold row in shared memory
    int form = 0, form_t = 0;  // path 7: kForm* of a chain
    int n_groups = 0;       // path 7: chain groups of a CTA
    // a context's own launches: set-up overlaps the kernel before (wait_for_earlier_kernels)
    int overlap = 0;
    int pieces = 0;         // path 8: > 1 where the random words come in pieces of a sweep
    int copy = 0;           // paths 1, 3 and 9: one copy a thread (sweep_copy_kernel)
    int nibble = 0;         // path 4: neighbour slots of the nibble form, 0 = one bit a copy
    int rows = 0;           // path 1: the word-wise kernel (DevProblem::slots > 0)
    int records = 0;        // the instance with records (DevProblem::records)
    int lean = 0;           // paths 2, 3, 4, 6 and 8: the instance with less registers a thread
    int chains_per_cta = 1; // path 10: chains packed on one CTA (cluster = ceil(R / chains_per_cta))
};

// Sizes of the dynamic shared-memory carve-up of the sweep kernel for a path.
// cluster_pre: path 9 with producer warps (its plan's n_consumer < threads)
size_t sweep_smem_bytes(const DevProblem& p, int path, int dclass, bool cluster_pre = false);
// Path 1: neighbour slots of the word-wise kernel's descriptors when its layout fits max_smem
// (with threshold rows and statistics in global memory if need be), else 0: byte-wise.
int rows_slots(const DevProblem& p, int max_degree, size_t max_smem);
// Shared memory of the one-copy-a-thread kernels (cluster: path 9).
size_t copy_smem_bytes(const DevProblem& p, bool cluster);
// path 10: the shared memory of a CTA holding `chains` classical chains
size_t classical_smem_bytes(const DevProblem& p, int chains);

// Forms of a batched chain in shared memory: int8 rows with update units of 1, 2 or 4 words of
// four copies, or bit words of 16 (nibbles) or 32 copies (bits_unit).
enum { kFormBytes1 = 0, kFormBytes2, kFormBytes4, kFormNibbles, kFormBits, kFormCount };
__host__ __device__ inline size_t form_row_bytes(int form, int P) {
    return form == kFormBits ? P / 8 : (form == kFormNibbles ? P / 4 : P);
}
__host__ __device__ inline int form_unit_copies(int form) { return 4 << (form == kFormNibbles ? 2 : form == kFormBits ? 3 : form); }

// One request of a batched launch (device view). Every chain of the request is swept by
// one CTA of the thread-block cluster that takes the request; the cluster's CTAs split the
// chains and exchange (E, M) through distributed shared memory for the swap passes.
struct BatchInstance {
    const uint32_t* sdesc;     // [N][DW] packed-path site descriptors (int8 rows)
    const uint32_t* wdesc;     // the same for bit words ("plain"), null for byte forms
    const uint32_t* items;     // [2N] schedule, grouped by level
    const int32_t* level_off;  // [n_levels + 1]
    const uint32_t* titems;    // the same levels balanced for form_t on one-warp groups
    const int32_t* tlevel_off;
    const uint32_t* thr;       // [R][nL3]
    const double* coef;        // [2(R-1)] (at least 2 entries)
    int8_t* spins;             // [R][slot_stride]
    long long* E;              // [R] by replica
    long long* M;
    int32_t* rung_of_slot;     // [R]
    int32_t* slot_of_rung;     // [R]
    unsigned long long* acc;   // [R][kAccCount] by rung
    unsigned long long* swap_stats;  // [R][2] by pair
    Mailbox* mail;             // [kClusterMailPasses][R], used when the swap mailboxes are not in shared memory
    int N, P, R, Lmax, nL3, n_levels, dc, slot_stride;
    int group_threads;         // threads sweeping one chain (a divisor of the CTA size)
    int resident;              // 1: a CTA keeps all its chains in shared memory for the run
    int thr_resident;          // 1: every rung's threshold row stays in shared memory for the run
    int mail_smem;             // 1: the swap mailboxes in every CTA's shared memory
    int form;                  // kForm*: how a chain lies in shared memory (form_t, or kFormBytes1)
    int form_t;                // the form with the least instructions for the chain on one-warp groups
    int n_groups;              // groups of group_threads threads at work in a CTA
    int withhold;              // test hook: 1 + the rung whose chain never publishes (0 = off)
    uint32_t key0, key1;
    long long t0, q0;          // counters before this run
    int n_sweeps, sweeps_per_swap;
};

// CTA `rank` of a cluster of K: its chains of the problem, and where they are during a run.
struct CtaShare {
    int begin, count;
    bool keep;      // no more chains than groups: each group keeps one
    bool in_place;  // chain lc stays in buffer lc; else chains are streamed, a buffer a group
    __host__ __device__ CtaShare(const BatchInstance& I, int rank, int K) {
        const int C = (I.R + K - 1) / K;
        begin = rank * C;
        count = I.R - begin < C ? I.R - begin : C;
        if (count < 0) count = 0;
        keep = count <= I.n_groups;
        // The last CTA of a streamed problem has fewer chains than the others, and may keep them: a
        // kept chain has its group's buffer to itself, so it stays there. (Streaming it would need a
        // wait between the store after one sweep and the load before the next: bulk copies have no
        // order among themselves.)
        in_place = I.resident != 0 || keep;
    }
    // chain buffers of every CTA of the cluster
    __host__ __device__ static int buffers(const BatchInstance& I, int K) {
        return I.resident ? (I.R + K - 1) / K : I.n_groups;
    }
};

// A group's place in its CTA's sequence of tasks: task number s * count + lc is sweep s of chain
// lc. Group g begins with task g (there are more chains than groups); the others are numbered by a
// counter from the groups' number on. The number can pass 2^32 (2^30 sweeps of 1024 chains), but the
// counter only has to tell a group's next task from its last one: a group takes the next while the
// chain of its last is still to be marked done, and until then each sweep of that chain holds up one
// other group, so fewer than (groups + 1) x chains tasks lie between the two.
struct TaskCursor {
    unsigned task;
    int s, lc;
    __host__ __device__ explicit TaskCursor(int group) : task((unsigned)group), s(0), lc(group) {}
    __host__ __device__ void move_to(unsigned next, int count) {
        const unsigned x = (unsigned)lc + (next - task);
        const unsigned sweeps = x / (unsigned)count;
        task = next;
        s += (int)sweeps;
        lc = (int)(x - sweeps * (unsigned)count);
    }
};

struct BatchParams {
    BatchInstance* inst;        // [count]; t0 / q0 of a finished problem advance in place
    const int32_t* order;       // [count] request indices, most work first
    int count;
    int* next_job;              // work counter, zero at launch
    int* status;
    long long timeout_ns = 5000000000ll;  // limit of every wait inside the launch
    int* done = nullptr;        // [count] or null: done[k] = done_token once problem k is written back
    int done_token = 1;         // nonzero, different per launch, so stale flags never match
    int single = 0;             // 1: one cluster runs `one` (passed by value) once; inst, order,
                                // next_job and done are unused and the counters stay on the host
    BatchInstance one;
};

// Kernel launchers (pt_kernels.cu). Each returns a cudaError_t from the launch.
cudaError_t launch_init(const DevProblem& p, cudaStream_t s);
cudaError_t launch_energy(const DevProblem& p, cudaStream_t s);
cudaError_t launch_sweeps(const DevProblem& p, const LaunchPlan& plan, long long t0,
                          long long q0, int n_sweeps, int sweeps_per_swap, long long timeout_ns,
                          bool cooperative, cudaStream_t s);
cudaError_t launch_swap(const DevProblem& p, long long q, cudaStream_t s, bool overlap = false);
cudaError_t launch_gather_state(const DevProblem& p, int8_t* out, cudaStream_t s);
cudaError_t launch_scatter_state(const DevProblem& p, const int8_t* in, cudaStream_t s);
cudaError_t sweep_kernel_occupancy(const DevProblem& p, const LaunchPlan& plan, int* blocks_per_sm);
// Chains that can be resident at once for a plan (CTAs, or clusters of the split kernel).
cudaError_t sweep_resident_chains(const DevProblem& p, const LaunchPlan& plan, long long* chains);
cudaError_t prepare_sweep_kernel(const LaunchPlan& plan);

// One problem of a multi-problem cooperative launch (one CTA per chain of every problem).
struct MultiProblem {
    DevProblem p;
    int dc;                    // packed neighbour slots: 4 or 8
    int n_sweeps, sweeps_per_swap;
    long long t0, q0, timeout_ns;
};
size_t multi_smem_bytes(const DevProblem& p, int dc);
cudaError_t multi_prepare(int threads, size_t smem, int* blocks_per_sm);
cudaError_t launch_multi(const MultiProblem* probs, const int2* map, int n_blocks, int threads, size_t smem,
                         cudaStream_t s);

// Host-side preparation shared by single and batched problems (pt_host.cu).
void build_tables(int R, int P, int Lmax, const pt_rung* ladder, std::vector<uint32_t>& thr,
                  std::vector<double>& coef);
// per_round > 0: levels balanced for a kernel that takes per_round items of a level at a
// time (same level count, same dependencies); 0: every update as early as possible.
// row_words > 0: each level's items ordered for a packed kernel whose rows are row_words
// 4-byte words (see level_schedule); 0: in site order.
void level_schedule(int N, const std::vector<std::vector<int>>& adj, std::vector<uint32_t>& items,
                    std::vector<int32_t>& level_off, int per_round = 0, int row_words = 0);
void build_site_desc(int N, int row_bytes, int dclass, int Lmax, const std::vector<std::vector<int>>& adj,
                     const std::vector<std::vector<int>>& adjJ, const int32_t* h, std::vector<uint32_t>& desc,
                     bool plain = false);  // plain: J itself and an unbiased constant (path 4's nibble form)

// Host-side preparation of one batched request (pt_batch.cu).
struct Prepared {
    int N, P, R, Lmax, dc, n_levels, slot_stride, form;
    std::vector<uint32_t> sdesc, wdesc, items, titems, thr;
    std::vector<int32_t> level_off, tlevel_off;
    std::vector<double> coef;
    size_t off_sdesc, off_wdesc, off_items, off_loff, off_titems, off_tloff, off_thr, off_coef, off_spins, off_E, off_M, off_rung, off_slot, off_acc,
        off_sw, off_mbox = 0, off_inst = 0, off_map = 0, off_status = 0;
    long long sweep_limit;
};
// per_round > 0: the level schedule is balanced for a kernel taking per_round items at a time.
int prepare_request(const pt_request& r, Prepared& pr, char* why, size_t why_len, int per_round = 0);
size_t request_block_layout(Prepared& p, size_t mailbox_entries = 0);
void fill_instance(BatchInstance& I, const Prepared& p, unsigned char* base, const pt_request& r);
// Group width of a fixed layout: narrowest that fits (one warp per chain where possible),
// which the autotuner picks on the batched size mix.
constexpr int kGroupWidenDefault = -4;
// Cycles the n_sweeps of a request take on one cluster, by the model choose_groups compares forms
// with (the layout choose_groups picked for that cluster).
double request_cycles(const BatchInstance& I, int cluster);
void choose_groups(BatchInstance& I, int cluster, int threads, size_t smem_cap, int widen = kGroupWidenDefault);
// Every chain resident, swept by groups of the given width: as many groups as fit, at least `least`,
// with every rung's threshold row and the swap mailboxes in shared memory where those fit too.
// False (I unchanged) when the chains don't fit.
bool resident_groups(BatchInstance& I, int cluster, int threads, size_t smem_cap, int group_threads, int least);

// Batched launchers (pt_batch.cu).
size_t batch_smem_bytes(const BatchInstance& I, int cluster, int threads);
cudaError_t launch_batch(const BatchParams& bp, int cluster, int n_clusters, int threads, size_t smem,
                         cudaStream_t s);
cudaError_t batch_max_clusters(int cluster, int threads, size_t smem, int* n_clusters);
cudaError_t launch_batch_init(const BatchInstance* inst, const int2* map, int n_chains, cudaStream_t s);
// One problem on one cluster of `cluster` CTAs (path 7); I carries t0, q0, n_sweeps, sweeps_per_swap.
cudaError_t launch_batch_single(const BatchInstance& I, int cluster, int threads, size_t smem, int* status,
                                long long timeout_ns, cudaStream_t s);
// The largest shared-memory need of the batched kernel: the device's opt-in maximum less
// the kernel's static shared memory.
size_t batch_smem_cap();

}  // namespace ptq
