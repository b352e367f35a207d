// Switching noise (Sec. 2): the counter-based draws and the redraw of one site.
#pragma once

#include <cmath>
#include <cstdint>

// Philox4x64-10 (Salmon et al., SC'11): ten rounds of two 64 x 64 -> 128-bit
// products with the key bumped by the Weyl constants; four output words.
struct Philox4 {
    unsigned long long w[4];
};

static __device__ __forceinline__ Philox4 philox4x64(unsigned long long c0, unsigned long long c1,
                                              unsigned long long c2, unsigned long long c3,
                                              unsigned long long k0, unsigned long long k1) {
    const unsigned long long M0 = 0xD2E7470EE14C6C93ull, M1 = 0xCA5A826395121157ull;
    const unsigned long long W0 = 0x9E3779B97F4A7C15ull, W1 = 0xBB67AE8584CAA73Bull;
#pragma unroll
    for (int round = 0; round < 10; ++round) {
        const unsigned long long hi0 = __umul64hi(M0, c0), lo0 = M0 * c0;
        const unsigned long long hi1 = __umul64hi(M1, c2), lo1 = M1 * c2;
        const unsigned long long n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
        c0 = n0;
        c1 = lo1;
        c2 = n2;
        c3 = lo0;
        k0 += W0;
        k1 += W1;
    }
    return Philox4{{c0, c1, c2, c3}};
}

static __device__ __forceinline__ double unit_double(unsigned long long w) {
    return (double)(w >> 11) * 0x1.0p-53;
}

// What a Hamiltonian update needs beside the parameters themselves.
struct SwitchLaw {
    unsigned long long seed = 0;
    unsigned long long below = 0;   // a 53-bit draw under this switches (probability p: p 2^53, rounded up)
    const double *eps_mean = nullptr, *J_mean = nullptr;   // or null: 0 and J0
    double eps_hw = 0.0, J_hw = 0.0, J0 = 0.0;
    int round_f32 = 1, periodic = 0;
};

// u < p for a draw u = w 2^-53 in [0, 1) is w < p 2^53; the product by a power
// of two is exact.
inline unsigned long long switch_below(double p) {
    return (unsigned long long)std::ceil(p * 9007199254740992.0);
}

// Site i of realization r (N sites) after step `step`: Philox block
// (step, r, i, 0) under key (seed, 0); words 0, 1 decide and redraw eps_i,
// words 2, 3 the hopping of bond i (not the absent wrap bond of an open
// chain).  Returns bit 0: e was redrawn, bit 1: j was.
static __device__ __forceinline__ int switch_site(const SwitchLaw &law, unsigned long long step, int r, int i, int N,
                                                  double &e, double &j) {
    const Philox4 b = philox4x64(step, (unsigned long long)r, (unsigned long long)i, 0ull, law.seed, 0ull);
    int changed = 0;
    if ((b.w[0] >> 11) < law.below) {
        const double em = law.eps_mean ? law.eps_mean[i] : 0.0;
        e = __dadd_rn(em, __dmul_rn(law.eps_hw, __dadd_rn(__dmul_rn(2.0, unit_double(b.w[1])), -1.0)));
        if (law.round_f32) e = (double)__double2float_rn(e);
        changed |= 1;
    }
    if ((law.periodic || i < N - 1) && (b.w[2] >> 11) < law.below) {
        const double jm = law.J_mean ? law.J_mean[i] : law.J0;
        j = __dadd_rn(jm, __dmul_rn(law.J_hw, __dadd_rn(__dmul_rn(2.0, unit_double(b.w[3])), -1.0)));
        if (law.round_f32) j = (double)__double2float_rn(j);
        changed |= 2;
    }
    return changed;
}
