// ising_walk.cuh -- one colour of one thread's column of 16-site chunks for
// 2D spin-1/2 Ising lattices (uniform, or with the disorder of Eq. 1): the
// two-launch kernels of a lone lattice (kernels_wide.cu), and the neighbours and
// counters of a chunk, which the band-resident forms use too.
//
// The thread walks consecutive rows.  The three rows of the other plane
// that a chunk touches stay in registers and turn over by renaming, so a row
// costs one new load of each plane; the next row's loads and Philox draws
// share each instruction block with this row's acceptance.  Acceptance looks
// every threshold up, or, on long walks of symmetric tables, goes by the top 16
// bits (accept16.cuh); there rows with an undecided site are marked and done
// again exactly, from memory, after the walk (one chunk in 2700).
#pragma once

#include <type_traits>

#include "accept16.cuh"
#include "wide_common.cuh"

#if defined(__CUDACC__)
namespace lat {
namespace {

// Disorder of Eq. 1: none, bond signs, bond and field signs.
enum IsingDisorder { kUniform = 0, kBonds = 1, kFields = 2 };

// Acceptance: every threshold from the table in shared memory, or the top 16
// bits (accept16.cuh) of a general or a symmetric table.
enum IsingAccept { kLookUp = 0, kTopGen = 1, kTopSym = 2 };

// The planes of one colour's pass: colour 0 reads both planes of the old
// buffer; colour 1 its own old sites and the new colour-0 sites.  Each
// writes only its own plane of the new buffer.
template <int kColour>
struct IsingPlanes {
    const int8_t *pS, *pO;
    int8_t *dS;
    const int8_t *r1, *r0;   // reference planes 1 and 0 (or null)
    const int8_t *pC;        // this colour's disorder bytes (or null)
    uint32_t half, L, G;
};

template <int kColour>
LAT_D IsingPlanes<kColour> ising_planes(const SweepView &v, unsigned long long sweep)
{
    const int8_t *old = (sweep & 1) ? v.s1 : v.s0;
    int8_t *nw = (sweep & 1) ? v.s0 : v.s1;
    const size_t plane = (size_t)v.plane;
    IsingPlanes<kColour> p;
    p.pS = old + kColour * plane;
    p.pO = (kColour == 0 ? old : nw) + (1 - kColour) * plane;
    p.dS = nw + kColour * plane;
    p.r1 = v.ref ? v.ref + plane : nullptr;
    p.r0 = v.ref;
    p.pC = v.cpl ? reinterpret_cast<const int8_t *>(v.cpl) + kColour * plane : nullptr;
    p.half = v.half;
    p.L = (uint32_t)v.L;
    p.G = v.G;
    return p;
}

// A chunk's sites and neighbours (U north, D south, O same index, X
// shifted), disorder applied to the neighbours; E: 0xFE where eta_i = -1.
struct IsingChunk {
    uint32_t S[4], U[4], D[4], O[4], X[4], E[4];
    Nbr n[4];
    uint32_t St[4];   // the spins as the table sees them
};

// C: the chunk's disorder bytes; odd: x = 2j + 1 in this row.  kFold: field
// signs go into the neighbours and spins (else into the table index).
template <int kDis, bool kFold = true>
LAT_D void ising_neighbours(IsingChunk &c, const uint32_t (&C)[4], bool odd)
{
    if constexpr (kDis != kUniform) {
        // a negative bond enters as a flipped neighbour (XOR 0xFE turns +1
        // into -1 and back); bits 0-3 of a disorder byte are the west, east,
        // north and south bonds
        const uint32_t sX = odd ? 1u : 0u, sO = odd ? 0u : 1u;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            c.X[w] ^= ((C[w] >> sX) & 0x01010101u) * 0xFEu;
            c.O[w] ^= ((C[w] >> sO) & 0x01010101u) * 0xFEu;
            c.U[w] ^= ((C[w] >> 2) & 0x01010101u) * 0xFEu;
            c.D[w] ^= ((C[w] >> 3) & 0x01010101u) * 0xFEu;
        }
    }
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        c.n[w] = nbr_sum(c.U[w], c.D[w], c.O[w], c.X[w]);
        c.St[w] = c.S[w];
        if constexpr (kDis == kFields) c.E[w] = ((C[w] >> 6) & 0x01010101u) * 0xFEu;
        if constexpr (kDis == kFields && kFold) {
            // eta_i = -1: the move has the energy of the flipped spin among
            // flipped neighbours at eta_i = +1 (sum and carry are self-dual)
            c.n[w].s1 ^= c.E[w];
            c.n[w].c1 ^= c.E[w];
            c.n[w].R ^= c.E[w];
            c.St[w] ^= c.E[w];
        }
    }
}

// Counter terms of a chunk's new spins (and of the other plane's at the
// same indices for the magnetisation), as byte dot products on the multiply
// pipe: the logic pipe is the busier one.
template <int kColour, int kDis, bool kAligned>
LAT_D void ising_count(const IsingChunk &c, const uint32_t (&Sn)[4], const uint32_t (&vm)[4], Counts &cnt)
{
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        const uint32_t Sv = kAligned ? Sn[w] : Sn[w] & vm[w], one = 0x01010101u & vm[w];
        if constexpr (kDis == kFields) cnt.fld = dot4(Sv, c.E[w] ^ 0x01010101u, cnt.fld);
        if constexpr (kColour == 1) {
            cnt.bond = dot4(Sv, c.U[w], cnt.bond);
            cnt.bond = dot4(Sv, c.D[w], cnt.bond);
            cnt.bond = dot4(Sv, c.O[w], cnt.bond);
            cnt.bond = dot4(Sv, c.X[w], cnt.bond);
            cnt.mag = dot4(Sn[w], one, cnt.mag);
        }
    }
}

// Row y's chunk again with full 32-bit draws; where the stored result
// differs, put it right.  Returns what to add to the counters.  (A call, with
// everything by value, so that the walk's registers and code stay small.)
template <int kColour, bool kRef, int kDis, bool kAligned>
__device__ __noinline__ Counts ising_redo(const IsingPlanes<kColour> p, const uint32_t *sthr,
                                          unsigned long long sweep, uint32_t key0, uint32_t key1, uint32_t k,
                                          uint32_t y)
{
    PhiloxPre pp;
    philox_prepare(pp, (uint32_t)sweep, (uint32_t)(sweep >> 32), key0, key1);
    Counts cnt;
    const ChunkCol<kAligned> cc = chunk_col<kAligned>(k, p.half);
    const size_t at = (size_t)y * p.half + cc.j0;
    const bool odd = ((kColour + y) & 1u) != 0u;
    IsingChunk c;
    uint32_t C[4] = {0, 0, 0, 0}, got[4], Sn[4];
    load16_any<kAligned>(p.pS + at, cc.nv, c.S);
    load16_any<kAligned>(p.pO + at, cc.nv, c.O);
    load16_any<kAligned>(p.pO + (size_t)(y == 0u ? p.L - 1u : y - 1u) * p.half + cc.j0, cc.nv, c.U);
    load16_any<kAligned>(p.pO + (size_t)(y + 1u == p.L ? 0u : y + 1u) * p.half + cc.j0, cc.nv, c.D);
    load16_any<kAligned>(p.dS + at, cc.nv, got);
    if constexpr (kDis != kUniform) load_words<4>(p.pC + at, C);
    shifted_row<kAligned>(cc, odd, (uint32_t)(uint8_t)p.pO[(size_t)y * p.half + (odd ? cc.jn : cc.jp)], c.O, c.X);
    ising_neighbours<kDis>(c, C, odd);
    uint32_t diff = 0;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        const U4 u = philox_item(pp, y * p.G + 4u * k + (uint32_t)w, (uint32_t)kColour);
        Sn[w] = c.S[w] ^ (~reject4_exact(sthr, c.n[w], c.St[w], u) & 0xFEFEFEFEu);
        diff |= (Sn[w] ^ got[w]) & cc.vm[w];
    }
    if (diff == 0u) return cnt;
    Counts was, now;
    ising_count<kColour, kDis, kAligned>(c, got, cc.vm, was);
    ising_count<kColour, kDis, kAligned>(c, Sn, cc.vm, now);
    cnt.bond = now.bond - was.bond;
    cnt.mag = now.mag - was.mag;
    cnt.fld = now.fld - was.fld;
    if constexpr (kColour == 1 && kRef) {
        uint32_t R1[4];
        load16_any<kAligned>(p.r1 + at, cc.nv, R1);
#pragma unroll
        for (int w = 0; w < 4; ++w)
            cnt.acf += dot4(Sn[w] & cc.vm[w], R1[w], 0) - dot4(got[w] & cc.vm[w], R1[w], 0);
    }
    store16_any<kAligned>(p.dS + at, cc.nv, Sn);
    return cnt;
}

template <bool kTop>
struct IsingDraws {
    uint32_t p01[4], p23[4];   // top halves of the chunk's draws
};
template <>
struct IsingDraws<false> {
    U4 u[4];
};

// The table of ising_flips: the t' table, and with field signs a second half
// for eta_i = -1 (the energy of the flipped spin among flipped neighbours).
template <int kDis>
LAT_D void ising_table(const uint32_t *thr16, uint32_t *sthr)
{
    const uint32_t i = threadIdx.x;
    if (i < 16u) sthr[i] = thr16[i];
    if constexpr (kDis == kFields)
        if (i >= 16u && i < 32u && (i & 7u) <= 4u) sthr[i] = thr16[((i & 8u) ^ 8u) | (4u - (i & 7u))];
}

// 0xFE at the chunk's flipped sites, from full 32-bit draws.
template <int kDis>
LAT_D void ising_flips(const IsingChunk &c, const uint32_t *sthr, const U4 (&u)[4], uint32_t (&F)[4])
{
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        uint32_t far = 0;   // bit 6 of a byte: the second half
        if constexpr (kDis == kFields) far = c.E[w] & 0x40404040u;
        F[w] = ~reject4_exact(sthr, c.n[w], c.St[w], u[w], far) & 0xFEFEFEFEu;
    }
}

// Rows [y, y1), y < y1, of chunk column k.
template <int kColour, bool kRef, int kDis, int kAcc, bool kAligned>
LAT_D void ising_walk(const IsingPlanes<kColour> &p, const uint32_t (&acc)[8], const uint32_t *sthr,
                      unsigned long long sweep, uint32_t key0, uint32_t key1, uint32_t k, uint32_t y,
                      const uint32_t y1, Counts &cnt)
{
    constexpr bool kSym = kAcc == kTopSym;
    static_assert(kAcc != kTopGen, "general tables walk by look-ups");
    PhiloxPre pp;
    philox_prepare(pp, (uint32_t)sweep, (uint32_t)(sweep >> 32), key0, key1);
    const ChunkCol<kAligned> cc = chunk_col<kAligned>(k, p.half);
    const uint32_t rows = y1 - y;
    uint32_t R[4][4];   // rows of the other plane, row y - 1 + i in R[(s + i) & 3] at step s
    Row16<kAligned> nS, nD;
    uint32_t nC[4] = {0, 0, 0, 0}, nb_next;
    IsingDraws<kSym> draws[2];
    auto other_row = [&](uint32_t r) { return p.pO + (size_t)r * p.half + cc.j0; };
    auto fetch = [&](uint32_t r) {   // row r's own sites and neighbour byte, row r + 1 of the other plane
        const size_t at = (size_t)r * p.half;
        row_load<kAligned>(p.pS + at + cc.j0, cc.nv, nS);
        row_load<kAligned>(other_row(r + 1u == p.L ? 0u : r + 1u), cc.nv, nD);
        nb_next = (uint32_t)(uint8_t)p.pO[at + (((kColour + r) & 1u) ? cc.jn : cc.jp)];
        if constexpr (kDis != kUniform) load_words<4>(p.pC + at + cc.j0, nC);
    };
    auto draw = [&](uint32_t r, IsingDraws<kSym> &d) {
        const uint32_t g0 = r * p.G + 4u * k;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const U4 u = philox_item(pp, g0 + (uint32_t)w, (uint32_t)kColour);
            if constexpr (kSym) top_halves(u, d.p01[w], d.p23[w]);
            else d.u[w] = u;
        }
    };
    {
        Row16<kAligned> a, b;
        const int8_t *qa = other_row(y == 0u ? p.L - 1u : y - 1u), *qb = other_row(y);
        row_load<kAligned>(qa, cc.nv, a);
        row_load<kAligned>(qb, cc.nv, b);
        fetch(y);
        draw(y, draws[0]);
        row_words<kAligned>(qa, a, R[0]);
        row_words<kAligned>(qb, b, R[1]);
    }
    uint32_t redo = 0, first = y;   // undecided rows first + i
    // Row y at step s of four (a constant, so that R and draws stay in registers); whether there is another.
    auto row = [&](auto which) {
        constexpr int s = decltype(which)::value;
        const uint32_t at = y * p.half + cc.j0;
        const bool odd = ((kColour + y) & 1u) != 0u, more = y + 1u < y1;
        IsingChunk c;
        uint32_t C[4];
        row_words<kAligned>(p.pS + at, nS, c.S);
        row_words<kAligned>(other_row(y + 1u == p.L ? 0u : y + 1u), nD, R[(s + 2) & 3]);
        shifted_row<kAligned>(cc, odd, nb_next, R[(s + 1) & 3], c.X);
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            c.U[w] = R[s][w];
            c.O[w] = R[(s + 1) & 3][w];
            c.D[w] = R[(s + 2) & 3][w];
            C[w] = nC[w];
        }
        [[maybe_unused]] uint32_t R1[4], R0[4];
        if constexpr (kColour == 1 && kRef) {   // (asked for here, not where they are used: L = 8192, 76 us for 80)
            load16_any<kAligned>(p.r1 + at, cc.nv, R1);
            load16_any<kAligned>(p.r0 + at, cc.nv, R0);
        }
        auto step = [&]() {
            ising_neighbours<kDis, false>(c, C, odd);
            uint32_t F[4], Sn[4];
            bool tie = false;
            if constexpr (kSym) tie = flips16<true>(acc, c.n, c.St, draws[s & 1].p01, draws[s & 1].p23, F);
            else ising_flips<kDis>(c, sthr, draws[s & 1].u, F);
#pragma unroll
            for (int w = 0; w < 4; ++w) Sn[w] = c.S[w] ^ F[w];
            store16_any<kAligned>(p.dS + at, cc.nv, Sn);
            ising_count<kColour, kDis, kAligned>(c, Sn, cc.vm, cnt);
            if constexpr (kColour == 1) {
#pragma unroll
                for (int w = 0; w < 4; ++w) cnt.mag = dot4(R[(s + 1) & 3][w], 0x01010101u & cc.vm[w], cnt.mag);
                if constexpr (kRef) {
#pragma unroll
                    for (int w = 0; w < 4; ++w)
                        cnt.acf = dot4(Sn[w] & cc.vm[w], R1[w], dot4(R[(s + 1) & 3][w] & cc.vm[w], R0[w], cnt.acf));
                }
            }
            if (tie) redo |= 1u << (y - first);
        };
        if (more) {   // the next row's loads and draws in the same block
            fetch(y + 1u);
            draw(y + 1u, draws[(s + 1) & 1]);
            step();
            ++y;
        } else {
            step();
        }
        return more;
    };
    for (bool more = true; more;) {
        more = row(std::integral_constant<int, 0>()) && row(std::integral_constant<int, 1>()) &&
               row(std::integral_constant<int, 2>()) && row(std::integral_constant<int, 3>());
        if constexpr (kSym) {
            if (!more || y - first >= 28u) {
                while (redo != 0u) {
                    const uint32_t i = (uint32_t)__ffs((int)redo) - 1u;
                    redo &= redo - 1u;
                    const Counts d =
                        ising_redo<kColour, kRef, kDis, kAligned>(p, sthr, sweep, key0, key1, k, first + i);
                    cnt.bond += d.bond;
                    cnt.mag += d.mag;
                    cnt.fld += d.fld;
                    cnt.acf += d.acf;
                }
                first = y;
            }
        }
    }
    if constexpr (kColour == 1) cnt.up += (cnt.mag + 2 * (int)(cc.nv * rows)) / 2;
}

// Row y's chunk of column k alone (lattices with little more than one chunk
// a thread).  Everything it reads is asked for before its draws.
template <int kColour, bool kRef, int kDis, int kAcc, bool kAligned>
LAT_D void ising_one(const IsingPlanes<kColour> &p, const uint32_t (&acc)[8], const uint32_t *sthr, unsigned long long sweep, uint32_t key0, uint32_t key1, uint32_t k, uint32_t y, Counts &cnt)
{
    const ChunkCol<kAligned> cc = chunk_col<kAligned>(k, p.half);
    const size_t at = (size_t)y * p.half + cc.j0;
    const bool odd = ((kColour + y) & 1u) != 0u;
    IsingChunk c;
    uint32_t C[4] = {0, 0, 0, 0}, O[4], F[4], Sn[4];
    load16_any<kAligned>(p.pS + at, cc.nv, c.S);
    load16_any<kAligned>(p.pO + at, cc.nv, O);
    load16_any<kAligned>(p.pO + (size_t)(y == 0u ? p.L - 1u : y - 1u) * p.half + cc.j0, cc.nv, c.U);
    load16_any<kAligned>(p.pO + (size_t)(y + 1u == p.L ? 0u : y + 1u) * p.half + cc.j0, cc.nv, c.D);
    const uint32_t nb = (uint32_t)(uint8_t)p.pO[(size_t)y * p.half + (odd ? cc.jn : cc.jp)];
    if constexpr (kDis != kUniform) load_words<4>(p.pC + at, C);
    [[maybe_unused]] uint32_t R1[4], R0[4];
    if constexpr (kColour == 1 && kRef) {
        load16_any<kAligned>(p.r1 + at, cc.nv, R1);
        load16_any<kAligned>(p.r0 + at, cc.nv, R0);
    }
    U4 u[4];
    {   // while the loads are on their way
        PhiloxPre pp;
        philox_prepare(pp, (uint32_t)sweep, (uint32_t)(sweep >> 32), key0, key1);
#pragma unroll
        for (int w = 0; w < 4; ++w)
            u[w] = philox_item(pp, y * p.G + 4u * k + (uint32_t)w, (uint32_t)kColour);
    }
    shifted_row<kAligned>(cc, odd, nb, O, c.X);
#pragma unroll
    for (int w = 0; w < 4; ++w) c.O[w] = O[w];
    ising_neighbours<kDis, false>(c, C, odd);
    if constexpr (kAcc == kLookUp) {
        ising_flips<kDis>(c, sthr, u, F);
    } else {
        uint32_t p01[4], p23[4];
#pragma unroll
        for (int w = 0; w < 4; ++w) top_halves(u[w], p01[w], p23[w]);
        if (flips16<kAcc == kTopSym>(acc, c.n, c.St, p01, p23, F)) ising_flips<kDis>(c, sthr, u, F);
    }
#pragma unroll
    for (int w = 0; w < 4; ++w) Sn[w] = c.S[w] ^ F[w];
    store16_any<kAligned>(p.dS + at, cc.nv, Sn);
    ising_count<kColour, kDis, kAligned>(c, Sn, cc.vm, cnt);
    if constexpr (kColour == 1) {
#pragma unroll
        for (int w = 0; w < 4; ++w) cnt.mag = dot4(O[w], 0x01010101u & cc.vm[w], cnt.mag);
        if constexpr (kRef) {
#pragma unroll
            for (int w = 0; w < 4; ++w)
                cnt.acf = dot4(Sn[w] & cc.vm[w], R1[w], dot4(O[w] & cc.vm[w], R0[w], cnt.acf));
        }
    }
    if constexpr (kColour == 1) cnt.up += (cnt.mag + 2 * (int)cc.nv) / 2;
}

}  // namespace
}  // namespace lat
#endif
