// qsg_sweep.cuh -- device pieces shared by the sweep kernels (k_wavefront.cu,
// k_sweep_unit.cu): the shared-memory plane ring, the threshold search and the
// bitsliced site update on multispin words.
#pragma once
#include "qsg_device.cuh"

namespace qsg {
namespace sweep {

constexpr int kRing = 16;  // planes held in shared memory (a power of two)

__device__ __forceinline__ void cp_async8(void *smem, const void *gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

struct Thresh {
    uint32_t t[7];  // Metropolis: t[0..2]; heat bath: t[0..6]; non-increasing
};

template <int LUT>
__device__ __forceinline__ uint32_t lop3(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, %4;" : "=r"(r) : "r"(a), "r"(b), "r"(c), "n"(LUT));
    return r;
}
constexpr int kXor3 = 0x96, kMaj3 = 0xE8, kMux = 0xCA;  // a ^ b ^ c, majority, a ? b : c

// All ones where u < t, else zero: the borrow of a subtraction, spread by a
// second one.  Two additions of either pipe in place of a comparison and a
// select of the integer pipe (16 LOP3 with two of them: 1.12 of the time of 16
// LOP3 alone, with a compare and select 1.25).
__device__ __forceinline__ uint32_t below(uint32_t u, uint32_t t) {
    uint32_t r;
    asm("{.reg .u32 d; sub.cc.u32 d, %1, %2; subc.u32 %0, 0, 0;}" : "=r"(r) : "r"(u), "r"(t));
    return r;
}

// Bits of the scalar threshold a site's count is compared with, as all-ones /
// all-zero masks, found by a binary search over the monotone table.  Heat bath:
// m = #{n : u < T[n]} (S = -1 iff n_neg >= m), its bits m2 m1 m0; T[3] = 2^31 (h
// = 0).  Metropolis: a = #{c : u < T[c]} (flip iff n_unsat >= 3 - a), its bits
// m1 m0.
template <int ALGO>
__device__ __forceinline__ void threshold_masks(uint32_t u, const Thresh &T, uint32_t &m0, uint32_t &m1,
                                                uint32_t &m2) {
    if (ALGO == 0) {
        m2 = 0u;
        m1 = below(u, T.t[1]);
        m0 = below(u, lop3<kMux>(m1, T.t[2], T.t[0]));
    } else {
        m2 = ~(uint32_t)((int32_t)u >> 31);
        m1 = below(u, lop3<kMux>(m2, T.t[5], T.t[1]));
        m0 = below(u, lop3<kMux>(m1, lop3<kMux>(m2, T.t[6], T.t[2]), lop3<kMux>(m2, T.t[4], T.t[0])));
    }
}

// One site update on one half of the multispin words.  Terms: n1 .. n4 spatial
// neighbours with couplings j1 .. j4, tp / tm time neighbours (APBC sign folded
// in).  The six terms a_i (neighbour XOR coupling) are counted by two full
// adders (s1, c1), (s2, c2); with k = s1 & s2 the count is b = (s1 ^ s2) + 2 B1 +
// 4 B2, and [b >= m] is the carry of b + ~m + 1 (three steps, the first merged
// with s1 ^ s2): 14 LOP3 for the heat bath.  The new spin is [b >= m].
// Metropolis: with c the old spin the unsatisfied bonds number b (c = 0) or 6 -
// b (c = 1), and the spin flips iff that count is >= m = 3 - a; so the new spin
// is [b >= m] for c = 0 and [6 - b < m] = [b >= 7 - m] for c = 1, that is [b >=
// m XOR 7c], and ~m = a + 4 on three bits: 16 LOP3.  Written as lop3 because the
// compiler's own choice for the plain expressions took 15 % more of them (L = 24,
// L_tau = 2048 heat-bath sweep 1.14 -> 1.04 ms).
template <int ALGO>
__device__ __forceinline__ uint32_t update_half(uint32_t c, uint32_t n1, uint32_t n2, uint32_t n3, uint32_t n4,
                                                uint32_t tp, uint32_t tm, uint32_t j1, uint32_t j2, uint32_t j3,
                                                uint32_t j4, uint32_t m0, uint32_t m1, uint32_t m2) {
    const uint32_t a = n1 ^ j1, b = n2 ^ j2, d = n3 ^ j3, e = n4 ^ j4;
    const uint32_t s1 = lop3<kXor3>(a, b, d), c1 = lop3<kMaj3>(a, b, d);
    const uint32_t s2 = lop3<kXor3>(e, tp, tm), c2 = lop3<kMaj3>(e, tp, tm);
    const uint32_t k = s1 & s2, B1 = lop3<kXor3>(c1, c2, k), B2 = lop3<kMaj3>(c1, c2, k);
    if (ALGO == 0) {
        const uint32_t e0 = lop3<0xBE>(s1, s2, m0 ^ c);   // (s1 ^ s2) | ~m0'
        const uint32_t e1 = lop3<kMaj3>(B1, m1 ^ c, e0);  // carry of B1 + ~m1' + e0
        return lop3<0xB2>(B2, c, e1);                     // carry of B2 + ~c + e1
    }
    const uint32_t e0 = lop3<0x7D>(s1, s2, m0);  // (s1 ^ s2) | ~m0
    const uint32_t e1 = lop3<0xB2>(B1, m1, e0);  // carry of B1 + ~m1 + e0
    return lop3<0xB2>(B2, m2, e1);
}

// One site update on whole words: nr/nl/nu/nd and jr/jl/ju/jd are the spatial
// neighbours and their couplings.
template <int ALGO>
__device__ __forceinline__ uint64_t update_site(uint64_t c, uint64_t nr, uint64_t nl, uint64_t nu, uint64_t nd,
                                                uint64_t ntp, uint64_t ntm, uint64_t jr, uint64_t jl, uint64_t ju,
                                                uint64_t jd, uint32_t u, const Thresh &T) {
    uint32_t m0, m1, m2;
    threshold_masks<ALGO>(u, T, m0, m1, m2);
    auto lo = [](uint64_t v) { return (uint32_t)v; };
    auto hi = [](uint64_t v) { return (uint32_t)(v >> 32); };
    const uint32_t a = update_half<ALGO>(lo(c), lo(nr), lo(nl), lo(nu), lo(nd), lo(ntp), lo(ntm), lo(jr), lo(jl),
                                         lo(ju), lo(jd), m0, m1, m2);
    const uint32_t b = update_half<ALGO>(hi(c), hi(nr), hi(nl), hi(nu), hi(nd), hi(ntp), hi(ntm), hi(jr), hi(jl),
                                         hi(ju), hi(jd), m0, m1, m2);
    return ((uint64_t)b << 32) | a;
}

}  // namespace sweep
}  // namespace qsg
