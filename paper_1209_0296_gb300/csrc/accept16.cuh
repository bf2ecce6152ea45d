// accept16.cuh -- acceptance of 2D spin-1/2 moves, two sites per 32-bit
// operation.
//
// A move is accepted iff its 32-bit draw u <= t' (t' = thr - 1, all ones =
// always).  Looking t' up per site in shared memory and comparing per site
// costs about nine logic-pipe instructions a site, more than the Philox
// draws do, and the logic pipe is what bounds these kernels.  Here the top
// 16 bits decide: the thresholds of two sites come from a byte permute of a
// register table, one subtraction compares both, and the borrow bits of
// its two halves are the rejections.  Where the top 16 bits are equal (one
// site in 2^16) they do not decide, and the word is done again with full
// 32-bit compares, so the result is exact.
#pragma once

#include "lattice_internal.cuh"

#if defined(__CUDACC__)
namespace lat {

// Byte permute in PTX's generic mode: selector nibble bits 0-2 pick one of
// the eight bytes of (b, a), bit 3 replicates its sign over the output byte.
LAT_D uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel)
{
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
    return r;
}

// Neighbour words of one word of four sites, bytes 0x01 / 0xFF (bits 1-7 of
// a byte all say "down"): sum and carry of three of them, and the fourth.
struct Nbr {
    uint32_t s1, c1, R;
};

LAT_D Nbr nbr_sum(uint32_t a, uint32_t b, uint32_t c, uint32_t r)
{
    return Nbr{a ^ b ^ c, (a & b) | (a & c) | (b & c), r};
}

// Rejections of one word: t01, t23 are the 16-bit thresholds of sites 0, 1
// and 2, 3, p01, p23 the top halves of their draws.  0xFF at rejected sites;
// tie keeps track of pairs that may be undecided: its low half is 0 when a
// low half tied, its upper half <= 1 when an upper half did (the low half's
// borrow enters the upper half, so there a difference of -1 counts too).
LAT_D uint32_t reject4(uint32_t t01, uint32_t t23, uint32_t p01, uint32_t p23, uint32_t &tie)
{
    const uint32_t d01 = t01 - p01, d23 = t23 - p23;
    tie = __viaddmin_u16x2(d01, 0x00010000u, tie);
    tie = __viaddmin_u16x2(d23, 0x00010000u, tie);
    const uint32_t b01 = (~t01 & p01) | (~(t01 ^ p01) & d01);   // borrow out of every bit
    const uint32_t b23 = (~t23 & p23) | (~(t23 ^ p23) & d23);
    return prmt(b01, b23, 0xFDB9u);
}

constexpr uint32_t kNoTie = 0xFFFFFFFFu;
LAT_D bool tie_hit(uint32_t tie) { return (tie & 0xFFFFu) == 0u || tie < 0x20000u; }

// Thresholds when flipping all spins changes nothing and a move with two or
// more unlike neighbours is free (J >= 0, h = 0): three values, by the
// number of unlike neighbours 0, 1, >= 2.  The class bits of a site go
// straight into the two selector nibbles that fetch its 16-bit threshold.
LAT_D void sym_thresholds(const uint32_t (&acc)[8], const Nbr &n, uint32_t S, uint32_t &t01, uint32_t &t23)
{
    const uint32_t t = (n.s1 ^ S) & (n.R ^ S);
    const uint32_t ge2 = (n.c1 ^ S) | t;               // two or more unlike
    const uint32_t odd = n.s1 ^ n.R;                   // an odd number unlike
    const uint32_t sel = (ge2 & 0x44444444u) | ((odd & 0x22222222u) | 0x10101010u);
    t01 = prmt(acc[0], acc[1], sel);
    t23 = prmt(acc[0], acc[1], sel >> 16);
}

// Thresholds from a general table (any J and h), two words at a time: the
// down-neighbour counts (0..4) of both words, one nibble a site, select the
// low and high threshold bytes of an up and of a down spin.
LAT_D void gen_thresholds2(const uint32_t (&acc)[8], const Nbr &n0, const Nbr &n1, uint32_t S0, uint32_t S1,
                           uint32_t (&t01)[2], uint32_t (&t23)[2])
{
    const uint32_t M = 0x0F0F0F0Fu;
    const uint32_t z0 = ((n0.s1 ^ n0.R) & M) | ((n1.s1 ^ n1.R) & ~M);
    const uint32_t x0 = n0.c1 ^ (n0.s1 & n0.R), x1 = n1.c1 ^ (n1.s1 & n1.R);
    const uint32_t z1 = (x0 & M) | (x1 & ~M);
    const uint32_t y0 = n0.c1 & n0.s1 & n0.R, y1 = n1.c1 & n1.s1 & n1.R;
    const uint32_t z2 = (y0 & M) | (y1 & ~M);
    const uint32_t X = ((z0 & 0x22222222u) | (z1 & 0x44444444u) | (z2 & 0x88888888u)) >> 1;
#pragma unroll
    for (int h = 0; h < 2; ++h) {   // sites 0, 1 of both words, then sites 2, 3
        const uint32_t sel = h ? X >> 16 : X;
        const uint32_t dn = prmt(S0, S1, h ? 0xFBEAu : 0xD9C8u);   // 0xFF at down spins
        const uint32_t lo = (prmt(acc[4], acc[5], sel) & dn) | (prmt(acc[0], acc[1], sel) & ~dn);
        const uint32_t hi = (prmt(acc[6], acc[7], sel) & dn) | (prmt(acc[2], acc[3], sel) & ~dn);
        (h ? t23 : t01)[0] = prmt(lo, hi, 0x6240u);
        (h ? t23 : t01)[1] = prmt(lo, hi, 0x7351u);
    }
}

// The exact rejections of one word from full 32-bit draws and the t' table;
// far: 0x40 at the sites whose entries are 16 on.
LAT_D uint32_t reject4_exact(const uint32_t *sthr, const Nbr &n, uint32_t S, const U4 &u, uint32_t far = 0u)
{
    const uint32_t b0 = n.s1 ^ n.R, b1 = n.c1 ^ (n.s1 & n.R), b2 = n.c1 & n.s1 & n.R;
    const uint32_t idx = ((b0 & 0x04040404u) | (b1 & 0x08080808u) | (b2 & 0x10101010u) | (S & 0x20202020u) | far) >> 2;
    return (u.x > sthr[idx & 0x1Fu] ? 0xFFu : 0u) | (u.y > sthr[(idx >> 8) & 0x1Fu] ? 0xFF00u : 0u) |
           (u.z > sthr[(idx >> 16) & 0x1Fu] ? 0xFF0000u : 0u) | (u.w > sthr[idx >> 24] ? 0xFF000000u : 0u);
}

// Top halves of a Philox call's four words, in pairs.
LAT_D void top_halves(const U4 &u, uint32_t &p01, uint32_t &p23)
{
    p01 = prmt(u.x, u.y, 0x7632u);
    p23 = prmt(u.z, u.w, 0x7632u);
}

// Sum over four int8 products, added to c.
LAT_D int dot4(uint32_t a, uint32_t b, int c) { return __dp4a((int)a, (int)b, c); }

// Sixteen sites: 0xFE at flipped sites by the 16-bit compare; true when it
// may not have decided some site.
template <bool kSym>
LAT_D bool flips16(const uint32_t (&acc)[8], const Nbr (&n)[4], const uint32_t (&S)[4], const uint32_t (&p01)[4],
                   const uint32_t (&p23)[4], uint32_t (&F)[4])
{
    uint32_t tie = kNoTie;
#pragma unroll
    for (int v = 0; v < 4; v += 2) {
        uint32_t t01[2], t23[2];
        if constexpr (kSym) {
            sym_thresholds(acc, n[v], S[v], t01[0], t23[0]);
            sym_thresholds(acc, n[v + 1], S[v + 1], t01[1], t23[1]);
        } else {
            gen_thresholds2(acc, n[v], n[v + 1], S[v], S[v + 1], t01, t23);
        }
        F[v] = ~reject4(t01[0], t23[0], p01[v], p23[v], tie) & 0xFEFEFEFEu;
        F[v + 1] = ~reject4(t01[1], t23[1], p01[v + 1], p23[v + 1], tie) & 0xFEFEFEFEu;
    }
    return tie_hit(tie);
}

}  // namespace lat
#endif
