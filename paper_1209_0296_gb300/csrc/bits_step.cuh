// bits_step.cuh -- acceptance of 32 bit-packed sites, shared by the streaming
// (kernels_bitpacked.cu) and the band-resident (kernels_band.cu) kernels.
#pragma once

#include "accept16.cuh"

#if defined(__CUDACC__)
namespace lat {
namespace {

// ---------------------------------------------------------------------
// Ising with a symmetric table (J >= 0, h = 0): thresholds K0, K1 for no and
// one unlike neighbour, every other move certain.  Turning the four
// bit planes of the table index into 32 byte offsets and looking 32
// thresholds up cost 15 instructions a site beside Philox's 9.5; here the
// top 16 bits of two draws are compared at a time (accept16.cuh).  Sites t,
// t + 8, t + 16, t + 24 go together: their "one unlike" bits sit at bit t of
// the four bytes, and their rejections, spread over four bytes by one byte
// permute, go back to those bits under a constant mask.
// ---------------------------------------------------------------------
struct SymK {
    uint32_t k0, k1;   // the top 16 bits of a threshold in both halves
};

// Bit i: site i of the word may not flip.  odd: sites with one (or three)
// unlike neighbours; tie as in reject4.
LAT_D uint32_t bits_rejected(const SymK &k, const PhiloxPre &pp, uint32_t g0, uint32_t colour, uint32_t odd,
                             uint32_t &tie)
{
    uint32_t rej = 0;
#pragma unroll
    for (int half = 0; half < 2; ++half) {   // sites 4 half + w + {0, 8, 16, 24}, w = 0..3
        U4 u[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) u[c] = philox_item(pp, g0 + (uint32_t)(half + 2 * c), colour);
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const int t = 4 * half + w;
            const uint32_t one = odd << (7 - t);   // bit 7 of each byte
            const uint32_t m01 = prmt(one, one, 0x9988u), m23 = prmt(one, one, 0xBBAAu);
            const uint32_t t01 = (k.k1 & m01) | (k.k0 & ~m01), t23 = (k.k1 & m23) | (k.k0 & ~m23);
            const uint32_t p01 = prmt(word_of(u[0], w), word_of(u[1], w), 0x7632u);
            const uint32_t p23 = prmt(word_of(u[2], w), word_of(u[3], w), 0x7632u);
            rej |= reject4(t01, t23, p01, p23, tie) & (0x01010101u << t);
        }
    }
    return rej;
}

// The same from full 32-bit draws (rare; by value, out of line).
__device__ __noinline__ uint32_t bits_rejected_exact(uint32_t thr0, uint32_t thr1, unsigned long long sweep,
                                                     uint32_t key0, uint32_t key1, uint32_t g0, uint32_t colour,
                                                     uint32_t odd)
{
    PhiloxPre pp;
    philox_prepare(pp, (uint32_t)sweep, (uint32_t)(sweep >> 32), key0, key1);
    uint32_t rej = 0;
#pragma unroll 1
    for (uint32_t q = 0; q < 8u; ++q) {
        const U4 u = philox_item(pp, g0 + q, colour);
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const uint32_t i = 4u * q + (uint32_t)w;
            if (word_of(u, w) > ((odd >> i) & 1u ? thr1 : thr0)) rej |= 1u << i;
        }
    }
    return rej;
}

// The word after the other plane's row word O in the direction its sites'
// side neighbours lie (x = 2j: west, bit j - 1; x = 2j + 1: east, bit j + 1).
LAT_D uint32_t bits_shifted(bool odd, uint32_t O, uint32_t next)
{
    return odd ? __funnelshift_r(O, next, 1) : __funnelshift_l(next, O, 1);
}

// A word's new spins from its neighbour words (exact).
LAT_D uint32_t bits_step(const SymK &sk, const uint32_t *thr16, const PhiloxPre &pp, unsigned long long sweep,
                         uint32_t key0, uint32_t key1, uint32_t g0, uint32_t colour, const Nbr &n, uint32_t S)
{
    const uint32_t odd = n.s1 ^ n.R;                              // an odd number unlike
    const uint32_t ge2 = (n.c1 ^ S) | ((n.s1 ^ S) & (n.R ^ S));   // two or more unlike
    uint32_t tie = kNoTie;
    uint32_t rej = bits_rejected(sk, pp, g0, colour, odd, tie);
    if (tie_hit(tie)) rej = bits_rejected_exact(thr16[0], thr16[1], sweep, key0, key1, g0, colour, odd);
    return S ^ (ge2 | ~rej);
}

LAT_D SymK bits_sym(const uint32_t *thr16)
{
    return SymK{__byte_perm(thr16[0], 0, 0x3232), __byte_perm(thr16[1], 0, 0x3232)};
}

// Unlike bonds of a word (sum and carry of three neighbours, and the fourth).
LAT_D int bits_unlike(const Nbr &n, uint32_t Sn) { return __popc(n.s1 ^ Sn) + 2 * __popc(n.c1 ^ Sn) + __popc(n.R ^ Sn); }

}  // namespace
}  // namespace lat
#endif
