// pt_device.cuh -- device building blocks shared by the PT-QMC kernels: Philox4x32-10,
// the deterministic exp and swap rule, PTX helpers and the packed 4-copy update unit.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "pt.h"
#include "pt_internal.h"

namespace ptq {


// ------------------------------------------------------------------------- Philox4x32-10
// Salmon, Moraes, Dror, Shaw, SC'11: round (c0,c1,c2,c3) -> (hi(M1 c2)^c1^k0, lo(M1 c2),
// hi(M0 c0)^c3^k1, lo(M0 c0)); the round-r key is (k0 + r W0, k1 + r W1).
struct PhiloxKey {
    uint32_t k0[10];
    uint32_t k1[10];
    __device__ __forceinline__ uint32_t a(int r) const { return k0[r]; }
    __device__ __forceinline__ uint32_t b(int r) const { return k1[r]; }
};

__device__ __forceinline__ PhiloxKey philox_schedule(uint32_t key0, uint32_t key1) {
    PhiloxKey k;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        k.k0[r] = key0 + (uint32_t)r * 0x9E3779B9u;
        k.k1[r] = key1 + (uint32_t)r * 0xBB67AE85u;
    }
    return k;
}

__device__ __forceinline__ uint4 philox_round(uint4 c, uint32_t ka, uint32_t kb) {
    const unsigned long long p0 = (unsigned long long)0xD2511F53u * c.x;
    const unsigned long long p1 = (unsigned long long)0xCD9E8D57u * c.z;
    return make_uint4((uint32_t)(p1 >> 32) ^ c.y ^ ka, (uint32_t)p1, (uint32_t)(p0 >> 32) ^ c.w ^ kb, (uint32_t)p0);
}

__device__ __forceinline__ uint4 philox(uint4 c, const PhiloxKey& k) {
#pragma unroll
    for (int r = 0; r < 10; ++r) c = philox_round(c, k.a(r), k.b(r));
    return c;
}


// ------------------------------------------------------------------------- det_exp
// exp(x) for x in (-23, 0] from IEEE round-to-nearest basic operations only (Cody & Waite
// argument reduction with a two-part ln 2, then the degree-13 Taylor series of exp by
// Horner's rule, then an exact scaling by 2^n). Each operation is an explicit _rn
// intrinsic so no multiply-add is fused; the host computes the same sequence.
__device__ __forceinline__ double det_exp(double x) {
    const double LN2_HI = 0x1.62e42ff000000p-1;
    const double LN2_LO = -0x1.718432a1b0e26p-35;
    const double INV_LN2 = 0x1.71547652b82fep+0;
    // 1/k! rounded to nearest (k! is exact in double for k <= 13); folded at compile time
    const double inv_fact[14] = {1.0, 1.0, 1.0 / 2.0, 1.0 / 6.0, 1.0 / 24.0, 1.0 / 120.0, 1.0 / 720.0,
                                 1.0 / 5040.0, 1.0 / 40320.0, 1.0 / 362880.0, 1.0 / 3628800.0,
                                 1.0 / 39916800.0, 1.0 / 479001600.0, 1.0 / 6227020800.0};
    const double nd = rint(__dmul_rn(x, INV_LN2));
    const double r = __dsub_rn(__dsub_rn(x, __dmul_rn(nd, LN2_HI)), __dmul_rn(nd, LN2_LO));
    double poly = inv_fact[13];
#pragma unroll
    for (int k = 12; k >= 0; --k) poly = __dadd_rn(__dmul_rn(poly, r), inv_fact[k]);
    const int n = (int)nd;  // in [-34, 0]
    const double scale = __hiloint2double((1023 + n) << 20, 0);
    return __dmul_rn(poly, scale);
}

// The uniform word of swap pass q for the pair (rl, rl + 1).
__device__ __forceinline__ uint32_t swap_word(uint32_t q, uint32_t rl, const PhiloxKey& key) {
    return philox(make_uint4(q, rl, 0u, kTagSwap << 28), key).x;
}

// Swap decision for X on rung rl and Y on rung rl + 1, with the pass's uniform word from
// word() (called only when Delta falls in the band where it matters).
template <typename WordFn>
__device__ __forceinline__ bool swap_accept_by(long long EX, long long EY, long long MX, long long MY, double a,
                                               double c, WordFn word) {
    const double dE = __ll2double_rn(EX - EY);
    const double dM = __ll2double_rn(MX - MY);
    const double delta = __dadd_rn(__dmul_rn(a, dE), __dmul_rn(c, dM));
    if (delta >= 0.0) return true;
    if (!(delta > -23.0)) return false;
    const double v = floor(__dmul_rn(det_exp(delta), 4294967296.0));
    const uint32_t ts = (v >= 4294967295.0) ? 0xFFFFFFFFu : (uint32_t)v;
    return word() < ts;
}

// The same decision without FP64 in the common case. GB300's FP64 pipe makes the ~40
// dependent FP64 operations of swap_accept_by cost over a microsecond, so Delta and exp(Delta)
// are first estimated in FP32 with an error bound:
//   |D - Delta| <= err = 5*2^-24 * (|a dE| + |c dM|)   (conversions of a, c, dE, dM, two
//   products, one sum, and the FP64 roundings of Delta itself, with room to spare), and
//   2^32 exp(D) within a relative 1e-5 + 1.01 err of 2^32 exp(Delta) (expf is within 2 ulp).
// The estimate decides only when u is farther than that margin (plus float rounding of u)
// from the threshold, or Delta's sign and the -23 cut are certain; otherwise swap_accept_by
// decides. Either way the result equals swap_accept_by's.
template <typename WordFn>
__device__ __forceinline__ bool swap_accept_fast_by(long long EX, long long EY, long long MX, long long MY,
                                                    double a, double c, WordFn word, bool exact_only) {
    if (!exact_only) {
        const float pa = (float)a * (float)(EX - EY);
        const float pc = (float)c * (float)(MX - MY);
        const float D = pa + pc;
        const float err = (fabsf(pa) + fabsf(pc)) * 2.99e-7f + 1e-30f;
        if (D >= 2.0f * err) return true;                       // Delta >= 0
        if (err < 0.25f) {
            if (D < -23.5f) return false;                         // Delta <= -23
            if (D + 2.0f * err < 0.0f && D > -22.5f) {
                const float v = 4294967296.0f * expf(D);
                const float margin = v * (1.0e-5f + 1.01f * err) + 512.0f;
                const float uf = (float)word();
                if (uf + margin < v) return true;
                if (uf - margin > v) return false;
            }
        }
    }
    return swap_accept_by(EX, EY, MX, MY, a, c, word);
}

// The two rules with the word drawn from (q, rl) under `key` when needed.
__device__ __forceinline__ bool swap_accept_fast(long long EX, long long EY, long long MX, long long MY,
                                                 double a, double c, uint32_t q, uint32_t rl,
                                                 const PhiloxKey& key, bool exact_only) {
    return swap_accept_fast_by(EX, EY, MX, MY, a, c, [&] { return swap_word(q, rl, key); }, exact_only);
}

// ------------------------------------------------------------------------- PTX helpers
__device__ __forceinline__ unsigned long long globaltimer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed_u64(unsigned long long* p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Tag of pass q0 + pass, from qmod0 = q0 mod kTagPeriod (taken once per launch): a 32-bit
// remainder by a constant instead of a 64-bit one on the path to the partner.
__device__ __forceinline__ unsigned long long mbox_tag(uint32_t qmod0, int pass) {
    return (unsigned long long)((qmod0 + (uint32_t)pass) % (uint32_t)kTagPeriod) + 1ull;
}

// ------------------------------------------------------------------------- misc
__host__ __device__ inline size_t up16(size_t x) { return (x + 15) & ~(size_t)15; }

// Every thread of every CTA of the cluster: release this CTA's shared-memory writes (own and
// remote) and acquire the others'. The non-.aligned form, so threads of a warp may arrive
// from different branches.
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// The two halves of a cluster barrier, for CTAs whose arrival orders none of their own
// earlier writes for the peers (relaxed) or does (release), and whose wait must see the
// peers' writes (acquire). A release arrival also waits for the thread's earlier global
// stores, which a relaxed one does not.
__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory"); }
__device__ __forceinline__ void cluster_arrive_release() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait_acquire() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// Two adjacent 64-bit words (16-byte aligned) into CTA `rank`'s copy of a shared-memory
// location (distributed shared memory), in one store, relaxed at cluster scope: each word
// carries its own tag and the readers poll the words themselves, so no other ordering is
// needed.
__device__ __forceinline__ void st_cluster_u64x2(const void* local, unsigned rank, unsigned long long a,
                                                 unsigned long long b) {
    const unsigned l = (unsigned)__cvta_generic_to_shared(local);
    unsigned ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(l), "r"(rank));
    asm volatile("st.relaxed.cluster.shared::cluster.v2.u64 [%0], {%1, %2};" ::"r"(ra), "l"(a), "l"(b) : "memory");
}

// This CTA's shared-memory word, as the other CTAs of the cluster last wrote it.
__device__ __forceinline__ unsigned long long ld_cluster_local_u64(const void* local) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(local);
    unsigned long long v;
    asm volatile("ld.relaxed.cluster.shared::cta.u64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
    return v;
}

__device__ __forceinline__ void named_barrier(int id, int count) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}

// Shared-memory rows of the int8 packed path are split by parity: row i holds the P/2 even
// copies of site i, then its P/2 odd copies, so the 4 copies of one parity in an update
// unit are one aligned word. Global rows interleave the copies (k fastest); these convert
// one 8-copy chunk (copies 8g..8g+7) between the two layouts.
__device__ __forceinline__ void split_chunk(uint2 v, uint32_t& even, uint32_t& odd) {
    even = __byte_perm(v.x, v.y, 0x6420u);
    odd = __byte_perm(v.x, v.y, 0x7531u);
}
__device__ __forceinline__ uint2 join_chunk(uint32_t even, uint32_t odd) {
    return make_uint2(__byte_perm(even, odd, 0x5140u), __byte_perm(even, odd, 0x7362u));
}

// ceil(2^32 / G) for G > 1: with it, __umulhi(x, ginv) = x / G exactly while x * G < 2^32,
// which holds for every chunk index of a chain that fits in shared memory. 0 for G = 1.
__host__ __device__ inline uint32_t chunk_ginv(int G) {
    return G > 1 ? (uint32_t)((0x100000000ull + (unsigned long long)G - 1ull) / (unsigned long long)G) : 0u;
}
__device__ __forceinline__ int chunk_of_row(int x, int G, uint32_t ginv) {
    return ginv ? x - G * (int)__umulhi((uint32_t)x, ginv) : 0;
}

// Copy an interleaved chain (N sites x P copies, global) into the split layout (shared),
// threads [tid0, tid0 + nthr) taking 8-copy chunks; and back. G = P / 8, ginv = chunk_ginv(G).
__device__ __forceinline__ void load_split(int8_t* dst, const int8_t* src, int N, int P, int G, uint32_t ginv,
                                           int tid0, int nthr) {
    const uint2* s2 = reinterpret_cast<const uint2*>(src);
    const int half = P >> 1;
    const int n = N * G;
    // eight loads in flight per thread before any shared store (the stores could alias the
    // loads as far as the compiler knows, which would otherwise serialise every load)
    for (int x0 = tid0; x0 < n; x0 += 8 * nthr) {
        uint2 v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int x = x0 + k * nthr;
            v[k] = x < n ? s2[x] : make_uint2(0u, 0u);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int x = x0 + k * nthr;
            if (x < n) {
                const int g = chunk_of_row(x, G, ginv);
                const int row = 8 * x - 8 * g;  // i * P
                uint32_t ev, od;
                split_chunk(v[k], ev, od);
                *reinterpret_cast<uint32_t*>(dst + row + 4 * g) = ev;
                *reinterpret_cast<uint32_t*>(dst + row + half + 4 * g) = od;
            }
        }
    }
}
__device__ __forceinline__ void store_split(int8_t* dst, const int8_t* src, int N, int P, int G, uint32_t ginv,
                                            int tid0, int nthr) {
    uint2* d2 = reinterpret_cast<uint2*>(dst);
    const int half = P >> 1;
    for (int x = tid0; x < N * G; x += nthr) {
        const int g = chunk_of_row(x, G, ginv);
        const int row = 8 * x - 8 * g;
        d2[x] = join_chunk(*reinterpret_cast<const uint32_t*>(src + row + 4 * g),
                           *reinterpret_cast<const uint32_t*>(src + row + half + 4 * g));
    }
}

// The same copies for rows of a multiple of 16 copies, 16 copies (one 16-byte word) at a
// time: half the loads, stores and index arithmetic of the 8-copy form per byte. H = P / 16,
// hinv = chunk_ginv(H).
__device__ __forceinline__ void load_split16(int8_t* dst, const int8_t* src, int N, int P, int H, uint32_t hinv,
                                             int tid0, int nthr) {
    const uint4* s4 = reinterpret_cast<const uint4*>(src);
    const int half = P >> 1;
    const int n = N * H;
    for (int x0 = tid0; x0 < n; x0 += 4 * nthr) {
        uint4 v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int x = x0 + k * nthr;
            v[k] = x < n ? s4[x] : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int x = x0 + k * nthr;
            if (x < n) {
                const int h = chunk_of_row(x, H, hinv);
                const int row = 16 * x - 16 * h;  // i * P
                uint2 ev, od;
                split_chunk(make_uint2(v[k].x, v[k].y), ev.x, od.x);  // copies 16h .. 16h+7
                split_chunk(make_uint2(v[k].z, v[k].w), ev.y, od.y);  // copies 16h+8 .. 16h+15
                *reinterpret_cast<uint2*>(dst + row + 8 * h) = ev;
                *reinterpret_cast<uint2*>(dst + row + half + 8 * h) = od;
            }
        }
    }
}
__device__ __forceinline__ void store_split16(int8_t* dst, const int8_t* src, int N, int P, int H, uint32_t hinv,
                                              int tid0, int nthr) {
    uint4* d4 = reinterpret_cast<uint4*>(dst);
    const int half = P >> 1;
    const int n = N * H;
    for (int x0 = tid0; x0 < n; x0 += 4 * nthr) {
        uint2 ev[4], od[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int x = min(x0 + k * nthr, n - 1);
            const int h = chunk_of_row(x, H, hinv);
            const int row = 16 * x - 16 * h;
            ev[k] = *reinterpret_cast<const uint2*>(src + row + 8 * h);
            od[k] = *reinterpret_cast<const uint2*>(src + row + half + 8 * h);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int x = x0 + k * nthr;
            if (x < n) {
                const uint2 lo = join_chunk(ev[k].x, od[k].x), hi = join_chunk(ev[k].y, od[k].y);
                d4[x] = make_uint4(lo.x, lo.y, hi.x, hi.y);
            }
        }
    }
}

// ------------------------------------------------------------------------- update unit
// A unit is the W * 4 copies of one parity of one site that one thread updates together:
// bytes 4 W u .. 4 W (u + 1) - 1 of that parity's half of the site's row, one +-1 byte a copy.
//
// All of a unit's arithmetic up to the table lookup is done on four copies at once, as plain
// 32-bit integer multiply-adds on the words of +-1 bytes. A word V of +-1 bytes is
// 0x01010101 + 254 B with B the word of 0 / 1 bytes "spin is -1", so with k = -J / 127 modulo
// 2^32 (127 is odd) k V = k 0x01010101 - 2 J B: a sum of such products over the neighbours,
// plus a constant word, is exactly the word whose four bytes are h + sum_j J_j s_j + Lmax,
// because each byte of the result is in [0, 2 Lmax] and everything is exact modulo 2^32. One
// multiply-add per neighbour word replaces the byte transposes and dp4a a per-copy field takes.
// The product with the own spin mirrors the byte where the spin is -1 (x -> 2 Lmax - x): an
// exclusive-or with the spin's sign mask and one multiply-add. The Trotter term enters as
// D = [left differs] + [right differs] per byte (doubled). What bounds the packed kernels is
// the ALU pipe (logic, permute, compare: half the issue width); the multiply-adds run on the
// FMA pipe beside it.
//
// Site descriptor of a class of NS = DC - 1 neighbour slots (unused slots: J = 0, own row),
// row offsets in bytes:
//   DC = 4:  C4, off0..2 | k0..2, own row offset                        (8 words)
//   DC = 8:  C4, J0..3 and J4..6 as bytes, own row offset | off0..3 | off4..6, 0   (12 words)
// C4 carries h + sum J + Lmax + the index bias in every byte, less the 0x01010101 terms. With
// seven slots the products are taken with J itself and the sum is scaled by -1/127 once.
template <int DC>
struct SiteDesc {
    static constexpr int DW = (DC == 4) ? 8 : 12;
    static constexpr int NS = DC - 1;
};

template <int DC>
struct SiteTerms {
    uint32_t off[DC - 1];
    uint32_t k[DC - 1];
    uint32_t c4, row;
};

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
    return d;
}

template <int DC>
__device__ __forceinline__ SiteTerms<DC> load_site(const uint32_t* desc) {
    SiteTerms<DC> s;
    const uint4 d0 = *reinterpret_cast<const uint4*>(desc);
    const uint4 d1 = *reinterpret_cast<const uint4*>(desc + 4);
    if constexpr (DC == 4) {
        s.c4 = d0.x;
        s.off[0] = d0.y;
        s.off[1] = d0.z;
        s.off[2] = d0.w;
        s.k[0] = d1.x;
        s.k[1] = d1.y;
        s.k[2] = d1.z;
        s.row = d1.w;
    } else {
        const uint4 d2 = *reinterpret_cast<const uint4*>(desc + 8);
        s.c4 = d0.x;
        s.row = d0.w;
        s.off[0] = d1.x;
        s.off[1] = d1.y;
        s.off[2] = d1.z;
        s.off[3] = d1.w;
        s.off[4] = d2.x;
        s.off[5] = d2.y;
        s.off[6] = d2.z;
        // byte b of a J word, sign-extended (a selector nibble with its top bit set repeats the sign)
        s.k[0] = prmt(d0.y, 0u, 0x8880u);
        s.k[1] = prmt(d0.y, 0u, 0x9991u);
        s.k[2] = prmt(d0.y, 0u, 0xAAA2u);
        s.k[3] = prmt(d0.y, 0u, 0xBBB3u);
        s.k[4] = prmt(d0.z, 0u, 0x8880u);
        s.k[5] = prmt(d0.z, 0u, 0x9991u);
        s.k[6] = prmt(d0.z, 0u, 0xAAA2u);
    }
    return s;
}

// Bytes L + Lmax + bias of four copies from their neighbour words a[], own word V and its
// sign mask (0xFF in the bytes of -1 spins).
template <int DC>
__device__ __forceinline__ uint32_t site_index(const SiteTerms<DC>& s, const uint32_t* a, uint32_t V, uint32_t kM) {
    uint32_t f;
    if constexpr (DC == 4) {
        f = s.c4;
#pragma unroll
        for (int d = 0; d < DC - 1; ++d) f += s.k[d] * a[d];
    } else {
        uint32_t g = s.k[0] * a[0];
#pragma unroll
        for (int d = 1; d < DC - 1; ++d) g += s.k[d] * a[d];
        f = s.c4 + (0u - kInv127) * g;
    }
    const uint32_t m = prmt(V, 0u, 0xBA98u);  // every byte's sign, repeated
    return (f ^ m) + kM * m;
}

// u.s8 x s.s8 dot product of four bytes: the flip masks' bytes are 0xFE, -2 as signed.
__device__ __forceinline__ int dp4a_us(uint32_t a, uint32_t b, int c) {
    int d;
    asm("dp4a.u32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}

// The attempt with random word u is accepted against threshold th: u < th, and always for
// the entry 0xFFFFFFFF, for which inline words (PRE = false) are first capped at 2^32 - 2
// (produced words already are).
template <bool PRE>
__device__ __forceinline__ bool accepts(uint32_t u, uint32_t th) {
    if (!PRE) u = min(u, 0xFFFFFFFEu);
    return u < th;
}

// How one launch or problem finds its table entries (see IndexRule). The Trotter differences
// are taken at the mask's bit, so D counts kUnit per neighbour that differs.
template <bool WIDE>
struct UnitRule {
    static constexpr uint32_t kMask = WIDE ? 0x40404040u : 0x02020202u;
    static constexpr int kUnit = WIDE ? 64 : 2;
    uint32_t kM;  // site_index's mirror multiplier
    uint32_t sD;  // entries (narrow) or bytes (wide) of a column's stride, per unit of D
    int zero;     // the index byte of L = 0
    __device__ __forceinline__ explicit UnitRule(int Lmax) {
        const IndexRule r(Lmax);
        kM = r.kM;
        zero = r.zero();
        sD = WIDE ? (uint32_t)r.S / 16u : (uint32_t)r.S / 2u;
    }
};

// 0xFE in byte w when copy w flips: L = biased L bytes, D = Trotter differences, thr = byte
// offset in shared memory of the threshold row (wide: of its last column).
template <bool PRE, bool WIDE>
__device__ __forceinline__ uint32_t flips4(const unsigned char* smem, const UnitRule<WIDE>& rule, uint32_t L,
                                           uint32_t D, const uint32_t* u, uint32_t thr) {
    uint32_t off[4];
    if constexpr (!WIDE) {
        const uint32_t idx = L - rule.sD * D;
#pragma unroll
        for (int w = 0; w < 4; ++w) off[w] = __dp4a(idx, 4u << (8 * w), thr);
    } else {
        const uint32_t m = 0u - rule.sD;  // -S / 16 as a signed byte
#pragma unroll
        for (int w = 0; w < 4; ++w)
            off[w] = __dp4a(L, 4u << (8 * w), (uint32_t)dp4a_us(D, (m & 0xFFu) << (8 * w), (int)thr));
    }
    uint32_t F = 0u;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        const uint32_t th = *reinterpret_cast<const uint32_t*>(smem + off[w]);
        if (accepts<PRE>(u[w], th)) F |= 0xFEu << (8 * w);
    }
    return F;
}
// The row offset flips4 takes for a row that starts at byte `row`.
template <bool WIDE>
__device__ __forceinline__ uint32_t thr_base(uint32_t row, int Lmax) {
    return WIDE ? row + 8u * (uint32_t)IndexRule(Lmax).S : row;
}

// Sums of a sweep over the flipped copies, each times -2: flips, biased L bytes, D.
struct FlipSums {
    int n, L, D;
    __device__ __forceinline__ void clear() { n = L = D = 0; }
    __device__ __forceinline__ void add4(uint32_t F, uint32_t Lb, uint32_t Db) {
        n = dp4a_us(0x01010101u, F, n);
        L = dp4a_us(Lb, F, L);
        D = dp4a_us(Db, F, D);
    }
    __device__ __forceinline__ void add(const FlipSums& o) {
        n += o.n;
        L += o.L;
        D += o.D;
    }
    // the changes the flips make: E by -2 sum L, M by -2 sum m with m = 2 - (neighbours that differ) * 2
    template <bool WIDE>
    __device__ __forceinline__ int dE(const UnitRule<WIDE>& r) const { return L - r.zero * n; }
    template <bool WIDE>
    __device__ __forceinline__ int dM(const UnitRule<WIDE>&) const { return 2 * n - D / (UnitRule<WIDE>::kUnit / 2); }
    __device__ __forceinline__ int flips() const { return -n / 2; }
};

// Byte offsets, within a shared-memory row, of what a unit of one fixed column reads: its
// own words, the opposite-parity words at the same copies, and the one Trotter neighbour
// outside those. [0] for an even-copy unit, [1] for an odd one.
struct UnitOffsets {
    uint32_t own[2], opp[2], edge[2];
    __device__ __forceinline__ uint32_t own_of(uint32_t par) const { return own[0] + par * (own[1] - own[0]); }
    __device__ __forceinline__ uint32_t opp_of(uint32_t par) const { return opp[0] + par * (opp[1] - opp[0]); }
    __device__ __forceinline__ uint32_t edge_of(uint32_t par) const { return edge[0] + par * (edge[1] - edge[0]); }
};

// W consecutive words at an address aligned to 4 W bytes, in one access.
template <int W>
__device__ __forceinline__ void load_words(const int8_t* p, uint32_t* v) {
    if constexpr (W == 1) {
        v[0] = *reinterpret_cast<const uint32_t*>(p);
    } else if constexpr (W == 2) {
        const uint2 x = *reinterpret_cast<const uint2*>(p);
        v[0] = x.x;
        v[1] = x.y;
    } else {
        const uint4 x = *reinterpret_cast<const uint4*>(p);
        v[0] = x.x;
        v[1] = x.y;
        v[2] = x.z;
        v[3] = x.w;
    }
}
template <int W>
__device__ __forceinline__ void store_words(int8_t* p, const uint32_t* v) {
    if constexpr (W == 1)
        *reinterpret_cast<uint32_t*>(p) = v[0];
    else if constexpr (W == 2)
        *reinterpret_cast<uint2*>(p) = make_uint2(v[0], v[1]);
    else
        *reinterpret_cast<uint4*>(p) = make_uint4(v[0], v[1], v[2], v[3]);
}

// The unit in three steps, so that a unit can be evaluated before the threshold row it needs
// is known: evaluate (loads, index bytes, random words), decide the flips against one
// threshold row, commit (flip store and the sweep's sums).
template <int W>
struct UnitEval {
    int8_t* own;        // the unit's words in shared memory
    uint32_t V[W];      // its copies as +-1 bytes
    uint32_t L[W];      // biased L bytes
    uint32_t D[W];      // Trotter differences
    uint32_t u[4 * W];  // random words
};

// The Trotter differences of a unit's words V with opposite-parity words O: their left and
// right neighbours are O itself and O shifted by one copy with the edge copy coming in (at
// the low end for even copies, at the high end for odd ones).
template <int W, bool WIDE>
__device__ __forceinline__ void trotter_differences(const uint32_t* V, const uint32_t* O, uint32_t edge, uint32_t par,
                                                    uint32_t* D, uint32_t last_odd_sel = 0x4321u) {
    constexpr uint32_t mask = UnitRule<WIDE>::kMask;
#pragma unroll
    for (int x = 0; x < W; ++x) {
        const uint32_t lo = x == 0 ? edge : O[x > 0 ? x - 1 : 0], hi = x == W - 1 ? edge : O[x < W - 1 ? x + 1 : x];
        const uint32_t even_sel = x == 0 ? 0x2104u : 0x2107u;
        const uint32_t odd_sel = x == W - 1 ? last_odd_sel : 0x4321u;
        const uint32_t in = (W == 1) ? edge : (par ? hi : lo);
        const uint32_t sh = prmt(O[x], in, even_sel + par * (odd_sel - even_sel));
        D[x] = ((V[x] ^ O[x]) & mask) + ((V[x] ^ sh) & mask);
    }
}

// Random words of a unit: read from rbq[0 .. W-1] (PRE), else word w of philox((t, i, slot,
// par<<24 | gg + x)) for word x, gg the unit's first 8-copy chunk in the whole chain.
template <int W, bool PRE>
__device__ __forceinline__ void unit_words(uint32_t* u, uint32_t item, const uint4* rbq, uint32_t t, uint32_t slot,
                                           uint32_t gg, const PhiloxKey& key) {
#pragma unroll
    for (int x = 0; x < W; ++x) {
        const uint4 r =
            PRE ? rbq[x] : philox(make_uint4(t, item >> 1, slot, ((item & 1u) << 24) | (gg + (uint32_t)x)), key);
        u[4 * x + 0] = r.x;
        u[4 * x + 1] = r.y;
        u[4 * x + 2] = r.z;
        u[4 * x + 3] = r.w;
    }
}

// The unit's spins, index bytes and Trotter differences, from its site's terms.
template <int DC, int W, bool WIDE>
__device__ __forceinline__ void unit_eval_site(UnitEval<W>& e, int8_t* sp, const SiteTerms<DC>& s, uint32_t par,
                                               const UnitOffsets& o, const UnitRule<WIDE>& rule) {
    const uint32_t own_off = o.own_of(par);
    const uint32_t edge = (uint8_t)sp[s.row + o.edge_of(par)];
    e.own = sp + s.row + own_off;
    uint32_t O[W], a[DC - 1][W];
    load_words<W>(e.own, e.V);
    load_words<W>(sp + s.row + o.opp_of(par), O);
#pragma unroll
    for (int d = 0; d < DC - 1; ++d) load_words<W>(sp + s.off[d] + own_off, a[d]);
    trotter_differences<W, WIDE>(e.V, O, edge, par, e.D);
#pragma unroll
    for (int x = 0; x < W; ++x) {
        uint32_t ax[DC - 1];
#pragma unroll
        for (int d = 0; d < DC - 1; ++d) ax[d] = a[d][x];
        e.L[x] = site_index<DC>(s, ax, e.V[x], rule.kM);
    }
}

template <int DC, int W, bool PRE, bool WIDE>
__device__ __forceinline__ UnitEval<W> unit_eval(int8_t* sp, const uint32_t* s_sdesc, uint32_t item,
                                                 const UnitOffsets& o, const uint4* rbq, uint32_t t, uint32_t slot,
                                                 uint32_t gg, const UnitRule<WIDE>& rule, const PhiloxKey& key) {
    UnitEval<W> e;
    const SiteTerms<DC> s = load_site<DC>(s_sdesc + (item >> 1) * SiteDesc<DC>::DW);
    unit_words<W, PRE>(e.u, item, rbq, t, slot, gg, key);
    unit_eval_site<DC, W, WIDE>(e, sp, s, item & 1u, o, rule);
    return e;
}

template <int W, bool PRE, bool WIDE>
__device__ __forceinline__ void unit_flips(const UnitEval<W>& e, const unsigned char* smem, const UnitRule<WIDE>& rule,
                                           uint32_t thr, uint32_t* F) {
#pragma unroll
    for (int x = 0; x < W; ++x) F[x] = flips4<PRE, WIDE>(smem, rule, e.L[x], e.D[x], e.u + 4 * x, thr);
}

template <int W>
__device__ __forceinline__ void unit_commit(const UnitEval<W>& e, const uint32_t* F, FlipSums& sums) {
    uint32_t any = 0u, v[W];
#pragma unroll
    for (int x = 0; x < W; ++x) {
        sums.add4(F[x], e.L[x], e.D[x]);
        any |= F[x];
        v[x] = e.V[x] ^ F[x];  // a +-1 byte flips by an exclusive-or with 0xFE
    }
    if (any) store_words<W>(e.own, v);
}

// Row offsets of column u of a one-CTA chain (half = P / 2 bytes a parity).
template <int W>
__device__ __forceinline__ UnitOffsets row_offsets(uint32_t u, uint32_t half) {
    const uint32_t b = 4u * W * u;
    UnitOffsets o;
    o.own[0] = b;
    o.own[1] = half + b;
    o.opp[0] = half + b;
    o.opp[1] = b;
    o.edge[0] = half + (u == 0 ? half - 1u : b - 1u);
    o.edge[1] = b + 4u * W == half ? 0u : b + 4u * W;
    return o;
}

// Records: what an update reads of its site, one record for every update in schedule order, its
// parity worked in. A descriptor takes the item first (another shared-memory latency) and about
// eight instructions of parity arithmetic a unit, on a path whose every instruction costs a
// level five to six cycles; a record takes twice the descriptors' memory and more.
//   DC = 4:  C4, own words, opposite parity's, parity | off0..2, k0 | k1, k2, item, 0
//   DC = 8:  C4, own words, opposite parity's, parity | J bytes (2), item, 0 | off0..3 | off4..6, 0
template <int DC>
struct UnitRecord {
    static constexpr int kWords = DC == 4 ? 12 : 16;
};
__host__ __device__ inline int record_words(int dc) { return dc == 4 ? 12 : 16; }
template <int DC>
__device__ __forceinline__ void make_record(uint32_t* rec, const uint32_t* desc, uint32_t item, uint32_t half) {
    const uint32_t par = item & 1u, shift = par * half;
    const uint32_t row = DC == 4 ? desc[7] : desc[3];
    rec[0] = desc[0];
    rec[1] = row + shift;
    rec[2] = row + half - shift;
    rec[3] = par;
    if constexpr (DC == 4) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            rec[4 + d] = desc[1 + d] + shift;
            rec[7 + d] = desc[4 + d];
        }
        rec[10] = item;
        rec[11] = 0u;
    } else {
        rec[4] = desc[1];
        rec[5] = desc[2];
        rec[6] = item;
        rec[7] = 0u;
#pragma unroll
        for (int d = 0; d < 7; ++d) rec[8 + d] = desc[4 + d] + shift;
        rec[15] = 0u;
    }
}
// A record in registers: loaded a level ahead, it leaves the spins, the table and the flip
// between two barriers.
template <int DC>
struct LoadedRecord {
    SiteTerms<DC> s;  // (row: unused; offsets and own / opp carry the parity)
    uint32_t own, opp, par, item;
};
template <int DC>
__device__ __forceinline__ LoadedRecord<DC> load_record(const uint32_t* rec) {
    LoadedRecord<DC> l;
    const uint4 r0 = *reinterpret_cast<const uint4*>(rec), r1 = *reinterpret_cast<const uint4*>(rec + 4);
    l.s.c4 = r0.x;
    l.own = r0.y;
    l.opp = r0.z;
    l.par = r0.w;
    if constexpr (DC == 4) {
        const uint4 r2 = *reinterpret_cast<const uint4*>(rec + 8);
        l.s.off[0] = r1.x;
        l.s.off[1] = r1.y;
        l.s.off[2] = r1.z;
        l.s.k[0] = r1.w;
        l.s.k[1] = r2.x;
        l.s.k[2] = r2.y;
        l.item = r2.z;
    } else {
        const uint4 r2 = *reinterpret_cast<const uint4*>(rec + 8), r3 = *reinterpret_cast<const uint4*>(rec + 12);
        l.s.off[0] = r2.x;
        l.s.off[1] = r2.y;
        l.s.off[2] = r2.z;
        l.s.off[3] = r2.w;
        l.s.off[4] = r3.x;
        l.s.off[5] = r3.y;
        l.s.off[6] = r3.z;
        l.s.k[0] = prmt(r1.x, 0u, 0x8880u);
        l.s.k[1] = prmt(r1.x, 0u, 0x9991u);
        l.s.k[2] = prmt(r1.x, 0u, 0xAAA2u);
        l.s.k[3] = prmt(r1.x, 0u, 0xBBB3u);
        l.s.k[4] = prmt(r1.y, 0u, 0x8880u);
        l.s.k[5] = prmt(r1.y, 0u, 0x9991u);
        l.s.k[6] = prmt(r1.y, 0u, 0xAAA2u);
        l.item = r1.z;
    }
    return l;
}
// A unit of one word at column byte g4 = 4 g of its row half, edge copies at e0 (even) and e1 (odd)
// of the opposite half.
template <int DC, bool PRE, bool WIDE>
__device__ __forceinline__ UnitEval<1> record_eval(int8_t* sp, const LoadedRecord<DC>& l, uint32_t g4, uint32_t e0,
                                                   uint32_t e1, const uint4* rbq, uint32_t t, uint32_t slot,
                                                   const UnitRule<WIDE>& rule, const PhiloxKey& key) {
    UnitEval<1> e;
    int8_t* spg = sp + g4;
    e.own = spg + l.own;
    uint32_t O[1], a[DC - 1];
    load_words<1>(e.own, e.V);
    load_words<1>(spg + l.opp, O);
    const uint32_t edge = (uint8_t)sp[l.opp + e0 + l.par * (e1 - e0)];
#pragma unroll
    for (int d = 0; d < DC - 1; ++d) load_words<1>(spg + l.s.off[d], a + d);
    unit_words<1, PRE>(e.u, l.item, rbq, t, slot, g4 >> 2, key);
    trotter_differences<1, WIDE>(e.V, O, edge, l.par, e.D);
    e.L[0] = site_index<DC>(l.s, a, e.V[0], rule.kM);
    return e;
}

// ------------------------------------------------------------------------- any even P, any degree
// The same unit (W = 1) for the shapes the classes above leave out: P not a multiple of 8, or
// more than seven neighbours. Each parity's half of a row is padded to whole words (G words;
// pad bytes hold +1 and never flip) and a site lists its neighbours' (row offset, multiplier)
// pairs, padded to a multiple of four, so the neighbour loop runs to the site's own degree.
// Descriptor of a site: C4, own row offset, neighbour slots in use, 0 | off, k, off, k | ...
__host__ __device__ inline int rows_desc_words(int slots) { return 4 + 2 * slots; }

struct RowsColumn {
    UnitOffsets o;
    uint32_t odd_sel;  // where the edge copy enters an odd unit's last word
    uint32_t live;     // mask of the bytes that are copies
};
__device__ __forceinline__ RowsColumn rows_column(uint32_t g, uint32_t G, uint32_t n_par) {
    RowsColumn c;
    const uint32_t half = 4u * G, b = 4u * g;
    c.o.own[0] = b;
    c.o.own[1] = half + b;
    c.o.opp[0] = half + b;
    c.o.opp[1] = b;
    c.o.edge[0] = half + (g == 0 ? n_par - 1u : b - 1u);
    c.o.edge[1] = g + 1u == G ? 0u : b + 4u;
    const uint32_t r = g + 1u == G ? n_par - 4u * (G - 1u) : 4u;  // copies in this word, 1..4
    c.odd_sel = r == 4u ? 0x4321u : (r == 3u ? 0x4421u : (r == 2u ? 0x4441u : 0x4444u));
    c.live = 0xFFFFFFFFu >> (8u * (4u - r));
    return c;
}

// What a unit of that form needs of its site: the header, the first four neighbours, and
// where the others are listed.
struct RowsTerms {
    uint4 head, n0, n1;
    const uint32_t* rest;
};
__device__ __forceinline__ RowsTerms load_rows_site(const uint32_t* desc) {
    RowsTerms s;
    s.head = *reinterpret_cast<const uint4*>(desc);
    s.n0 = *reinterpret_cast<const uint4*>(desc + 4);
    s.n1 = *reinterpret_cast<const uint4*>(desc + 8);
    s.rest = desc + 12;
    return s;
}

template <bool WIDE>
__device__ __forceinline__ void rows_eval_site(UnitEval<1>& e, int8_t* sp, const RowsTerms& s, uint32_t par,
                                               const RowsColumn& c, const UnitRule<WIDE>& rule) {
    const uint32_t own_off = c.o.own_of(par);
    const uint32_t edge = (uint8_t)sp[s.head.y + c.o.edge_of(par)];
    e.own = sp + s.head.y + own_off;
    uint32_t O[1], a[4], f = s.head.x;
    load_words<1>(e.own, e.V);
    load_words<1>(sp + s.head.y + c.o.opp_of(par), O);
    load_words<1>(sp + s.n0.x + own_off, a);
    load_words<1>(sp + s.n0.z + own_off, a + 1);
    load_words<1>(sp + s.n1.x + own_off, a + 2);
    load_words<1>(sp + s.n1.z + own_off, a + 3);
    f += s.n0.y * a[0] + s.n0.w * a[1] + s.n1.y * a[2] + s.n1.w * a[3];
#pragma unroll 2
    for (uint32_t d = 4; d < s.head.z; d += 4) {
        const uint4 p0 = *reinterpret_cast<const uint4*>(s.rest + 2 * d - 8);
        const uint4 p1 = *reinterpret_cast<const uint4*>(s.rest + 2 * d - 4);
        load_words<1>(sp + p0.x + own_off, a);
        load_words<1>(sp + p0.z + own_off, a + 1);
        load_words<1>(sp + p1.x + own_off, a + 2);
        load_words<1>(sp + p1.z + own_off, a + 3);
        f += p0.y * a[0] + p0.w * a[1] + p1.y * a[2] + p1.w * a[3];
    }
    trotter_differences<1, WIDE>(e.V, O, edge, par, e.D, c.odd_sel);
    const uint32_t m = prmt(e.V[0], 0u, 0xBA98u);
    e.L[0] = (f ^ m) + rule.kM * m;
}

// ------------------------------------------------------------------------- one copy a thread
// For chains whose levels hold no more copies than a CTA has threads: a level then costs the
// latency of one update, about 4.7 cycles per instruction of the thread that runs it, so a
// thread takes one copy (about 40 instructions against about 95 for the four-copy unit).
// Rows and descriptors are those of the word-wise form above, with J and h themselves.
struct CopyEval {
    int8_t* own;
    int s, L, m;  // spin, s (h + sum_j J_j s_j), s (left + right)
    uint32_t u;   // random word
};
struct CopySums {
    int n, L, M;  // over flipped copies: count, sum of L, sum of m
};
__device__ __forceinline__ UnitOffsets copy_offsets(uint32_t h, uint32_t half, uint32_t n_par) {
    UnitOffsets o;
    o.own[0] = h;
    o.own[1] = half + h;
    o.opp[0] = half + h;
    o.opp[1] = h;
    o.edge[0] = half + (h == 0u ? n_par - 1u : h - 1u);
    o.edge[1] = h + 1u == n_par ? 0u : h + 1u;
    return o;
}
__device__ __forceinline__ CopyEval copy_eval(int8_t* sp, const uint32_t* desc, uint32_t par, const UnitOffsets& o,
                                              uint32_t word) {
    CopyEval e;
    const RowsTerms t = load_rows_site(desc);
    const uint32_t own_off = o.own_of(par);
    e.own = sp + t.head.y + own_off;
    e.s = *e.own;
    const int nn = sp[t.head.y + o.opp_of(par)] + sp[t.head.y + o.edge_of(par)];
    int f = (int)t.head.x;
    f += (int)t.n0.y * sp[t.n0.x + own_off] + (int)t.n0.w * sp[t.n0.z + own_off];
    f += (int)t.n1.y * sp[t.n1.x + own_off] + (int)t.n1.w * sp[t.n1.z + own_off];
#pragma unroll 2
    for (uint32_t d = 4; d < t.head.z; d += 4) {
        const uint4 p0 = *reinterpret_cast<const uint4*>(t.rest + 2 * d - 8);
        const uint4 p1 = *reinterpret_cast<const uint4*>(t.rest + 2 * d - 4);
        f += (int)p0.y * sp[p0.x + own_off] + (int)p0.w * sp[p0.z + own_off];
        f += (int)p1.y * sp[p1.x + own_off] + (int)p1.w * sp[p1.z + own_off];
    }
    e.L = e.s * f;
    e.m = e.s * nn;
    e.u = word;
    return e;
}
// The same from a record: the word-wise form's descriptor with the parity worked into every
// offset (head: h, own row half, slots, opposite row half).
__device__ __forceinline__ CopyEval copy_record_eval(int8_t* sp, const RowsTerms& t, uint32_t g, uint32_t e0,
                                                     uint32_t e1, uint32_t word) {
    CopyEval e;
    int8_t* spg = sp + g;
    e.own = spg + t.head.y;
    e.s = *e.own;
    const int nn = spg[t.head.w] + sp[t.head.w + (t.head.w < t.head.y ? e1 : e0)];
    int f = (int)t.head.x;
    f += (int)t.n0.y * spg[t.n0.x] + (int)t.n0.w * spg[t.n0.z];
    f += (int)t.n1.y * spg[t.n1.x] + (int)t.n1.w * spg[t.n1.z];
#pragma unroll 2
    for (uint32_t d = 4; d < t.head.z; d += 4) {
        const uint4 p0 = *reinterpret_cast<const uint4*>(t.rest + 2 * d - 8);
        const uint4 p1 = *reinterpret_cast<const uint4*>(t.rest + 2 * d - 4);
        f += (int)p0.y * spg[p0.x] + (int)p0.w * spg[p0.z];
        f += (int)p1.y * spg[p1.x] + (int)p1.w * spg[p1.z];
    }
    e.L = e.s * f;
    e.m = e.s * nn;
    e.u = word;
    return e;
}
// thr: byte offset of the entry L = 0, m = 0; S: entries of a column.
__device__ __forceinline__ bool copy_flips(const CopyEval& e, const unsigned char* smem, int thr, int S) {
    return e.u < *reinterpret_cast<const uint32_t*>(smem + (thr + 4 * e.L + 2 * S * e.m));
}
__device__ __forceinline__ void copy_commit(const CopyEval& e, bool flip, CopySums& sums) {
    if (flip) {
        *e.own = (int8_t)(-e.s);
        sums.n += 1;
        sums.L += e.L;
        sums.M += e.m;
    }
}

// Bit-packed chains (shared memory only), one bit a copy: row i is P/8 bytes, bit k of byte g is copy 8g+k,
// set = spin -1. lut[p*256 + b] spreads the four parity-p bits (p, p+2, p+4, p+6) of byte b
// into four +1/-1 bytes, so each neighbour contributes one byte load and one table load and
// the index arithmetic of the int8 unit is reused unchanged.
template <int DC, bool WIDE>
__device__ __forceinline__ void packed_unit_bits(uint8_t* bp, const uint32_t* s_sdesc, uint32_t item,
                                                 int g, int G, const uint32_t* lut,
                                                 uint32_t t, uint32_t slot, const PhiloxKey& key,
                                                 const unsigned char* smem, const UnitRule<WIDE>& rule, uint32_t thr,
                                                 FlipSums& sums) {
    const uint32_t par = item & 1u;
    const SiteTerms<DC> s = load_site<DC>(s_sdesc + (item >> 1) * SiteDesc<DC>::DW);
    const uint32_t ug = (uint32_t)g, last = (uint32_t)G - 1u;
    const uint32_t own = bp[s.row + ug];
    // the one Trotter neighbour outside the byte: copy 8g-1 (bit 7 of byte g-1) for even
    // copies, copy 8g+8 (bit 0 of byte g+1) for odd ones, periodic in the row
    const uint32_t eb = par ? (bp[s.row + (ug == last ? 0u : ug + 1u)] & 1u)
                            : ((uint32_t)bp[s.row + (ug == 0 ? last : ug - 1u)] >> 7);
    const uint32_t* lut_p = lut + (par << 8);
    uint32_t nbyte[DC - 1];
#pragma unroll
    for (int d = 0; d < DC - 1; ++d) nbyte[d] = bp[s.off[d] + ug];
    uint32_t u[4];
    unit_words<1, false>(u, item, nullptr, t, slot, ug, key);
    const uint32_t V = lut_p[own];
    const uint32_t Rn = par ? lut[256 + (((own >> 1) | (eb << 7)) & 0xFFu)] : lut[256 + own];
    const uint32_t Ln = par ? lut[own] : lut[((own << 1) | eb) & 0xFFu];
    const uint32_t D = ((V ^ Ln) & UnitRule<WIDE>::kMask) + ((V ^ Rn) & UnitRule<WIDE>::kMask);
    uint32_t a[DC - 1];
#pragma unroll
    for (int d = 0; d < DC - 1; ++d) a[d] = lut_p[nbyte[d]];
    const uint32_t L = site_index<DC>(s, a, V, rule.kM);
    const uint32_t F = flips4<false, WIDE>(smem, rule, L, D, u, thr);
    sums.add4(F, L, D);
    // bits 0, 2, 4, 6 from bytes 0..3
    const uint32_t f1 = (F >> 1) & 0x01010101u, fb = f1 | (f1 >> 6);
    if (F) bp[s.row + ug] = (uint8_t)(own ^ (((fb | (fb >> 12)) & 0x55u) << par));
}

// Bit-packed chains, whole words: a word holds 4 U copies of one parity of a site (U = 8, or
// U = 4 with the upper nibbles empty when the copies don't fill words of 32), unit k as bit k
// of its four bytes: copy 4 U c + 4 k + w of that parity is bit 8 w + k of word c. A row is
// its even words, then its odd ones. A thread takes a whole word: one load per neighbour, one
// descriptor and one address serve 4 U copies, and no other thread writes its word. The
// one-bit form above costs a byte load and a table load per neighbour and four copies; this
// one an AND and a multiply-add. The arithmetic is the int8 unit's with 0 / 1 bytes:
// sum_j J_j B_j of unit k comes from the words masked at bit k, that is scaled by 2^k, and is
// shifted down once the sum is formed. Every byte has to hold 2^k 2 Lmax until then: k <= 2
// for Lmax <= 31 (kWordBitsLmax), so the units go in threes, each from words shifted by 3
// more. Descriptors hold J itself and C4 = h + sum J + Lmax in every byte ("plain"). With the
// Trotter column taken as the count of equal neighbours no index bias is needed.
struct BitSums {
    int n, L, C;  // minus the sums over flipped copies of 1, L + Lmax and the Trotter column
    __device__ __forceinline__ void clear() { n = L = C = 0; }
    __device__ __forceinline__ int dE(int Lmax) const { return 2 * (L - Lmax * n); }
    __device__ __forceinline__ int dM() const { return 4 * (C - n); }
    __device__ __forceinline__ int flips() const { return -n; }
};
// Row offsets of word c of `cols`: own word, the opposite parity's, and the one its edge copy is
// in (the word before for even copies, after for odd ones).
__device__ __forceinline__ UnitOffsets word_offsets(uint32_t c, uint32_t cols) {
    UnitOffsets o;
    o.own[0] = 4u * c;
    o.own[1] = 4u * (cols + c);
    o.opp[0] = o.own[1];
    o.opp[1] = o.own[0];
    o.edge[0] = 4u * (cols + (c == 0u ? cols - 1u : c - 1u));
    o.edge[1] = 4u * (c + 1u == cols ? 0u : c + 1u);
    return o;
}
template <int DC, int NS, int U>
__device__ __forceinline__ void bits_unit(int8_t* sp, const uint32_t* s_sdesc, uint32_t item, const UnitOffsets& o,
                                          uint32_t c, uint32_t t, uint32_t slot, const PhiloxKey& key,
                                          const unsigned char* smem, uint32_t S, uint32_t kM, uint32_t thr,
                                          BitSums& sums) {
    const uint32_t par = item & 1u;
    const SiteTerms<DC> s = load_site<DC>(s_sdesc + (item >> 1) * SiteDesc<DC>::DW);
    const uint32_t own_off = o.own_of(par);
    uint32_t* own = reinterpret_cast<uint32_t*>(sp + s.row + own_off);
    const uint32_t V = *own;
    const uint32_t O = *reinterpret_cast<const uint32_t*>(sp + s.row + o.opp_of(par));
    const uint32_t E = *reinterpret_cast<const uint32_t*>(sp + s.row + o.edge_of(par));
    uint32_t W[NS];
#pragma unroll
    for (int d = 0; d < NS; ++d) W[d] = *reinterpret_cast<const uint32_t*>(sp + s.off[d] + own_off);
    // the opposite parity shifted by one copy: bytes up (even copies) or down (odd copies) by
    // one, and the byte that comes in from the next unit, its last unit's from the edge word
    // (with U = 4, bits above the nibble are never looked at)
    const uint32_t in = par ? ((O >> 1) & (U == 8 ? 0x7Fu : ~0u)) | (E << (U - 1))
                            : ((O >> 23) & (U == 8 ? ~1u : ~0u)) | (E >> (23 + U));
    const uint32_t sh = prmt(O, in, 0x2104u + par * (0x4321u - 0x2104u));
    uint32_t flip = 0u;
#pragma unroll
    for (int k = 0; k < U; ++k) {
        uint32_t u[4];
        unit_words<1, false>(u, item, nullptr, t, slot, (uint32_t)U * c + (uint32_t)k, key);
        const uint32_t mk = 0x01010101u << k;
        constexpr int kGroup = 3;
        const int ks = k % kGroup, kb = k - ks;  // the scale of this unit's sum, the words' shift
        uint32_t g = 0u;
#pragma unroll
        for (int d = 0; d < NS; ++d) g += s.k[d] * ((W[d] >> kb) & (0x01010101u << ks));
        const uint32_t f = ((s.c4 << ks) - 2u * g) >> ks;
        const uint32_t m = prmt(V << (7 - k), 0u, 0xBA98u);  // 0xFF where the spin is -1
        const uint32_t L = (f ^ m) + kM * m;
        // neighbours equal to the spin; at k = 7 a byte cannot hold both
        const uint32_t C = k < 7 ? ((~(V ^ O) & mk) + (~(V ^ sh) & mk)) >> k
                                 : ((~(V ^ O) >> 7) & 0x01010101u) + ((~(V ^ sh) >> 7) & 0x01010101u);
        const uint32_t idx = L + S * C;
        uint32_t F = 0u;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const uint32_t th = *reinterpret_cast<const uint32_t*>(smem + __dp4a(idx, 4u << (8 * w), thr));
            if (accepts<false>(u[w], th)) F |= 0xFFu << (8 * w);
        }
        sums.n = dp4a_us(0x01010101u, F, sums.n);
        sums.L = dp4a_us(L, F, sums.L);
        sums.C = dp4a_us(C, F, sums.C);
        flip |= F & mk;
    }
    if (flip) *own = V ^ flip;
}

// Chains between global memory (interleaved +-1 bytes) and bit words, threads tid0, tid0 + nthr, ...
// taking whole words of both parities: 8 U copies.
template <int U>
__device__ __forceinline__ void load_bits(uint32_t* words, const int8_t* chain, int N, int cols, int tid0, int nthr) {
    const uint4* src = reinterpret_cast<const uint4*>(chain);
    for (int x = tid0; x < N * cols; x += nthr) {
        const int i = x / cols, c = x - i * cols;
        uint4 v[U / 2];
#pragma unroll
        for (int y = 0; y < U / 2; ++y) v[y] = src[(U / 2) * x + y];
        uint32_t even = 0u, odd = 0u;
#pragma unroll
        for (int y = 0; y < U / 2; ++y) {
            uint32_t e, d;
            split_chunk(make_uint2(v[y].x, v[y].y), e, d);
            even |= ((e >> 7) & 0x01010101u) << (2 * y);
            odd |= ((d >> 7) & 0x01010101u) << (2 * y);
            split_chunk(make_uint2(v[y].z, v[y].w), e, d);
            even |= ((e >> 7) & 0x01010101u) << (2 * y + 1);
            odd |= ((d >> 7) & 0x01010101u) << (2 * y + 1);
        }
        words[2 * i * cols + c] = even;
        words[(2 * i + 1) * cols + c] = odd;
    }
}
template <int U>
__device__ __forceinline__ void store_bits(int8_t* chain, const uint32_t* words, int N, int cols, int tid0, int nthr) {
    uint4* dst = reinterpret_cast<uint4*>(chain);
    for (int x = tid0; x < N * cols; x += nthr) {
        const int i = x / cols, c = x - i * cols;
        const uint32_t even = words[2 * i * cols + c], odd = words[(2 * i + 1) * cols + c];
#pragma unroll
        for (int y = 0; y < U / 2; ++y) {
            uint2 v[2];
#pragma unroll
            for (int z = 0; z < 2; ++z) {
                const int k = 2 * y + z;  // +-1 bytes: 1 + 0xFE where the bit is set
                v[z] = join_chunk(0x01010101u + 0xFEu * ((even >> k) & 0x01010101u),
                                  0x01010101u + 0xFEu * ((odd >> k) & 0x01010101u));
            }
            dst[(U / 2) * x + y] = make_uint4(v[0].x, v[0].y, v[1].x, v[1].y);
        }
    }
}

}  // namespace ptq
