// ne_walk.cuh -- the pieces of a c-mode North-East half-sweep: the constraint
// and the certain moves of a 16-site chunk and its counters, which the streaming
// kernels (kernels_ne.cu) and the band-resident ones (band.cuh) share, and the
// streaming kernels' queued draws.
#pragma once

#include "accept16.cuh"
#include "wide_common.cuh"

#if defined(__CUDACC__)
namespace lat {
namespace {

constexpr int kNeQueue = 32 + 4 * 32; // jobs per warp: under 32 left over, 4 per lane new
constexpr uint32_t kB1 = 0x02020202u; // one copy of a byte's "down" flag

// A queued group: Philox group index, byte offset of its first site in the
// colour's plane, flags of the sites whose draw decides, and the west (bit 1)
// and south (bit 2) neighbours' flags (colour 1).
struct __align__(16) NeJob {
    uint32_t g, at, cand, ws;
};

// The draw threshold (accept iff u <= K), the flag flip that marks the state
// which draws (0: down spins, all ones: up spins), and whether any does (all
// ones; 0 at c = 1/2, where both moves are certain).
struct NeRate {
    uint32_t K, inv, draws;
};

LAT_D NeRate ne_rate(const uint32_t *thr16)
{
    // index sd << 3 | nd; in c-mode every nd has the same entry
    const bool up_draws = thr16[8] == 0xFFFFFFFFu && thr16[0] != 0xFFFFFFFFu;
    const uint32_t K = up_draws ? thr16[0] : thr16[8];
    return NeRate{K, up_draws ? 0xFFFFFFFFu : 0u, K == 0xFFFFFFFFu ? 0u : 0xFFFFFFFFu};
}

// Where a queued move is applied: the colour's spins, its persistence bytes
// (one per group) and the reference plane 1.
struct NePlanes {
    uint8_t *spins, *flags;
    const int8_t *ref;
};

// 0xFF at the sites whose draw is above K.
LAT_D uint32_t ne_rejected(const U4 &u, uint32_t K)
{
    auto above = [&](uint32_t x) {   // all ones where x > K: the borrow of K - x
        uint32_t m;
        asm("{\n\t.reg .u32 d;\n\tsub.cc.u32 d, %1, %2;\n\tsubc.u32 %0, 0, 0;\n\t}" : "=r"(m) : "r"(K), "r"(x));
        return m;
    };
    const uint32_t m0 = above(u.x), m1 = above(u.y), m2 = above(u.z), m3 = above(u.w);
    const uint32_t lo = (m0 & 0x000000FFu) | (m1 & 0xFFFFFF00u), hi = (m2 & 0x00FFFFFFu) | (m3 & 0xFF000000u);
    return (lo & 0x0000FFFFu) | (hi & 0xFFFF0000u);
}

// One queued group: draw, accept, apply.
template <bool kRef>
LAT_D void ne_job(const NePlanes &p, const PhiloxPre &pp, const NeRate rate, const NeJob job, uint32_t colour,
                  Counts &cnt)
{
    const U4 u = philox_item(pp, job.g, colour);
    const uint32_t rej = ne_rejected(u, rate.K);
    const uint32_t f = job.cand & ~rej & kB1;   // accepted moves
    if (f == 0u) return;
    const uint8_t now = rate.inv ? 0xFFu : 0x01u;   // the spin after the move
    uint8_t *d = p.spins + job.at;
#pragma unroll
    for (int b = 0; b < 4; ++b)
        if (f & (2u << (8 * b))) d[b] = now;
    const uint32_t bits = (uint32_t)dot4(f, 0x08040201u, 0) >> 1;
    uint8_t *fl = p.flags + job.g;
    const uint32_t was = *fl;
    *fl = (uint8_t)(was | bits);
    cnt.unfl -= __popc(bits & ~was);
    if (colour == 1u) {
        // north and east are up, so a site's neighbour sum is 4 - 2 (west down + south down)
        const int n = __popc(f), side = __popc(f & job.ws) + __popc((f << 1) & job.ws), sg = rate.inv ? -2 : 2;
        cnt.mag += sg * n;
        cnt.bond += sg * (4 * n - 2 * side);
        if constexpr (kRef) {
#pragma unroll
            for (int b = 0; b < 4; ++b)
                if (f & (2u << (8 * b))) cnt.acf += sg * (int)p.ref[job.at + b];
        }
    }
}

// The moves of a chunk that need no draw: north U, south D, east E, west W,
// own spins S -> spins after the certain moves Sn, flags of those moves
// (sure), of the sites whose draw decides (cand) and of their west and south
// neighbours (ws), and which groups need a draw.  kHalf: looks whether any does.
template <bool kFull, bool kHalf = false>
LAT_D void ne_moves(const uint32_t (&U)[4], const uint32_t (&D)[4], const uint32_t (&E)[4], const uint32_t (&W)[4],
                    const uint32_t (&S)[4], const uint32_t (&vm)[4], const NeRate rate, uint32_t (&cand)[4],
                    uint32_t (&sure)[4], uint32_t (&ws)[4], uint32_t (&Sn)[4], bool (&need)[4])
{
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        const uint32_t open = kFull ? ~(U[w] | E[w]) : ~(U[w] | E[w]) & vm[w];
        const uint32_t undecided = kHalf ? (S[w] ^ rate.inv) & rate.draws : S[w] ^ rate.inv;
        cand[w] = open & undecided;
        sure[w] = open & ~undecided;
        need[w] = (cand[w] & kB1) != 0u;
        Sn[w] = S[w] ^ (sure[w] & 0xFEFEFEFEu);
        ws[w] = (W[w] & kB1) | (D[w] & ~kB1);
    }
}

// Persistence bits of the certain moves: byte w = group w, bit q = its site q.
LAT_D uint32_t ne_changed(const uint32_t (&sure)[4])
{
    int c = dot4(sure[3] & kB1, 0x08040201u, 0);
#pragma unroll
    for (int w = 2; w >= 0; --w) c = dot4(sure[w] & kB1, 0x08040201u, c * 256);
    return (uint32_t)c >> 1;
}

// The persistence bits of a chunk of nv sites, byte w = group w (the bytes of
// groups that do not exist are unspecified).  Unaligned: by whole words, so
// that a row waits for memory once and not once a group (L = 3000, c = 0.4,
// launches of a graph: 34.1 us a sweep with a byte read each, 21.4).  The
// words' other bytes are other threads'; a word that holds none of the
// chunk's is not read (the buffer is a multiple of 4 bytes, so every word read
// is in bounds).
template <bool kAligned>
LAT_D uint32_t ne_flags(const uint8_t *fp, uint32_t nv)
{
    if constexpr (kAligned) return *reinterpret_cast<const uint32_t *>(fp);
    const uintptr_t a = reinterpret_cast<uintptr_t>(fp);
    const uint32_t sh = (uint32_t)(a & 3u);
    const uint32_t *q = reinterpret_cast<const uint32_t *>(a - sh);
    return __funnelshift_r(q[0], sh + (nv + 3u) / 4u > 4u ? q[1] : 0u, 8u * sh);
}

// Write the bytes that changed.
template <bool kAligned>
LAT_D void ne_set_flags(uint8_t *fp, uint32_t was, uint32_t now)
{
    if constexpr (kAligned) {
        if (now != was) *reinterpret_cast<uint32_t *>(fp) = now;
    } else {
#pragma unroll
        for (int w = 0; w < 4; ++w)   // (only groups that exist have moves)
            if (((now ^ was) >> (8 * w) & 0xFFu) != 0u) fp[w] = (uint8_t)(now >> (8 * w));
    }
}

// Colour 1: bonds of the new spins, both planes' magnetisation.
LAT_D void ne_count(const uint32_t (&Sn)[4], const uint32_t (&U)[4], const uint32_t (&D)[4], const uint32_t (&O)[4],
                    const uint32_t (&X)[4], const uint32_t (&vm)[4], Counts &cnt)
{
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        const uint32_t Sv = Sn[w] & vm[w], one = 0x01010101u & vm[w];
        cnt.bond = dot4(Sv, U[w], cnt.bond);
        cnt.bond = dot4(Sv, D[w], cnt.bond);
        cnt.bond = dot4(Sv, O[w], cnt.bond);
        cnt.bond = dot4(Sv, X[w], cnt.bond);
        cnt.mag = dot4(Sn[w], one, dot4(O[w], one, cnt.mag));
    }
}

}  // namespace
}  // namespace lat
#endif
