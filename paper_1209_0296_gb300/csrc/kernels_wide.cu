// kernels_wide.cu -- two launches per sweep (one per colour, the kernel
// boundary being the device-wide barrier of §III.A steps 6-7) for 2D
// spin-1/2 lattices (Ising and North-East), int8 spins of +-1 in the
// checkerboard-planar layout, L a multiple of 32.
//
// A thread owns 16 consecutive same-colour sites of one plane row (one
// 16-byte load = four Philox groups), so the loads, index arithmetic and
// Philox set-up are shared by 16 sites.  The colour-c sites only read the
// other plane, so the colour-c pass never reads a byte another thread
// writes.  Neighbour counts, thresholds and acceptance are those of the
// tiled kernel (bytes 0x01 / 0xFF, bit-sliced adder, t' = thr - 1 table).
//
// The solo kernels (k_ising_walk for Ising at any even L, uniform or with
// per-bond and per-site disorder: ising_walk.cuh; k_wide_pipe_ne and
// k_any_pipe_ne for North-East rates that are not of the c-mode form, which
// kernels_ne.cu has) walk one chunk column per thread down the rows. They
// read s[sweep & 1] and write s[(sweep+1) & 1] without copying a plane:
// colour 1 takes the new colour-0 sites from the new buffer. Calls of
// several sweeps on lattices that fit the SMs' shared memory run in bands
// instead (kernels_band.cu). The resident kernels (wide_chunk or one word a
// thread, in place) keep the whole lattice in one CTA's shared memory.
#include <algorithm>

#include "ising_walk.cuh"

namespace lat {

namespace {

// Byte permute in PTX's generic mode, where bit 3 of a selector nibble
// replicates the sign bit of the selected byte over the output byte.
LAT_D uint32_t prmt_sign(uint32_t a, uint32_t sel)
{
    uint32_t r;
    asm("prmt.b32 %0, %1, 0, %2;" : "=r"(r) : "r"(a), "r"(sel));
    return r;
}

LAT_D int byte_sum(uint32_t x)
{
    const uint32_t s = (x & 0x00FF00FFu) + ((x >> 8) & 0x00FF00FFu);
    return (int)((s & 0xFFFFu) + (s >> 16));
}

// Sweep colour `colour` of the chunk k (16 sites, four Philox groups) of plane
// row y of the resident kernel's shared-memory lattice, in place (both
// buffer pointers of g are that array).
template <bool kNE>
LAT_D void wide_chunk(const SweepView g, const uint32_t *sthr, int colour, unsigned long long sweep,
                      const PhiloxPre &pp, int y, int k, Counts &cnt)
{
    constexpr int W = 4;
    const int8_t *src = g.s0;
    int8_t *dst = g.s0;
    const int L = g.L;
    const uint32_t half = g.half;
    const int oc = 1 - colour;
    const int ym = y == 0 ? L - 1 : y - 1, yp = y == L - 1 ? 0 : y + 1;
    const uint32_t nwr = half >> 2;  // 4-byte words per plane row
    auto row = [&](int c, int r) { return src + (uint64_t)c * g.plane + (uint64_t)r * half; };
    uint32_t S[W], O[W], U[W], D[W];
    load_words<W>(row(colour, y) + 4 * W * k, S);
    load_words<W>(row(oc, y) + 4 * W * k, O);
    load_words<W>(row(oc, ym) + 4 * W * k, U);   // north
    load_words<W>(row(oc, yp) + 4 * W * k, D);   // south
    const bool p1 = ((colour + y) & 1) != 0;
    uint32_t adj;
    {
        const uint32_t w = p1 ? (uint32_t)(W * k + W) : (uint32_t)(W * k - 1 + nwr);
        adj = reinterpret_cast<const uint32_t *>(row(oc, y))[wrap_once(w, nwr)];
    }
    U4 u[W];
#pragma unroll
    for (int w = 0; w < W; ++w) u[w] = U4{0, 0, 0, 0};
    uint32_t Lf[W], R[W];
#pragma unroll
    for (int w = 0; w < W; ++w) {
        if (!p1) {  // x = 2j: west is j-1 of the other plane, east is j
            Lf[w] = __funnelshift_l(w == 0 ? adj : O[w - 1], O[w], 8);
            R[w] = O[w];
        } else {    // x = 2j+1: west is j, east is j+1
            Lf[w] = O[w];
            R[w] = __funnelshift_r(O[w], w == W - 1 ? adj : O[w + 1], 8);
        }
    }
    uint32_t t[W][4], locked[W];
    bool need = false;
    const char *tb = reinterpret_cast<const char *>(sthr);
#pragma unroll
    for (int w = 0; w < W; ++w) {
        const uint32_t s1 = U[w] ^ D[w] ^ Lf[w];
        const uint32_t c1 = (U[w] & D[w]) | (U[w] & Lf[w]) | (D[w] & Lf[w]);
        const uint32_t b0 = s1 ^ R[w];
        const uint32_t b1 = c1 ^ (s1 & R[w]);
        const uint32_t b2 = c1 & s1 & R[w];
        // byte offset into the 16-entry table (index sd<<3 | nd, 4 bytes each)
        uint32_t idx = (b0 & 0x04040404u) | (b1 & 0x08080808u) | (b2 & 0x10101010u) | (S[w] & 0x20202020u);
        t[w][0] = *reinterpret_cast<const uint32_t *>(tb + (idx & 0xFFu));
        t[w][1] = *reinterpret_cast<const uint32_t *>(tb + ((idx >> 8) & 0xFFu));
        t[w][2] = *reinterpret_cast<const uint32_t *>(tb + ((idx >> 16) & 0xFFu));
        t[w][3] = *reinterpret_cast<const uint32_t *>(tb + (idx >> 24));
        locked[w] = 0;
        if constexpr (kNE) {
            // §III.B: north (U) and east (R) must be up; a locked site needs
            // no draw (t' all ones) and its flip is masked off below.
            locked[w] = U[w] | R[w];
            t[w][0] |= prmt_sign(locked[w], 0x8888u);
            t[w][1] |= prmt_sign(locked[w], 0x9999u);
            t[w][2] |= prmt_sign(locked[w], 0xAAAAu);
            t[w][3] |= prmt_sign(locked[w], 0xBBBBu);
        }
        need |= (t[w][0] & t[w][1] & t[w][2] & t[w][3]) != 0xFFFFFFFFu;
    }
    // An item that needs no draw has t' = all ones at every site, so any u
    // accepts exactly as "no draw" would.
    if (need) {
        const uint32_t g0 = (uint32_t)y * g.G + (uint32_t)(W * k);
#pragma unroll
        for (int w = 0; w < W; ++w) u[w] = philox_item(pp, g0 + (uint32_t)w, (uint32_t)colour);
    }
    uint32_t Sn[W], chg = 0;
    const uint32_t M1 = 0x02020202u;
    uint32_t ue = 0, dn = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) {
        const uint32_t acc = (u[w].x <= t[w][0] ? 1u : 0u) | (u[w].y <= t[w][1] ? 2u : 0u) |
                             (u[w].z <= t[w][2] ? 4u : 0u) | (u[w].w <= t[w][3] ? 8u : 0u);
        uint32_t F = ((acc * 0x00204081u) & 0x01010101u) * 0xFEu;  // 0xFE at flipped sites
        if constexpr (kNE) {
            F &= ~locked[w];
            chg |= ((((F >> 1) & 0x01010101u) * 0x01020408u) >> 24 & 0xFu) << (8 * w);
        }
        Sn[w] = S[w] ^ F;
        if (colour == 1) {
            // bond: 4 - 2 * (# unequal) per colour-1 site (2 per unequal bond below)
            ue += ((U[w] ^ Sn[w]) & M1) + ((D[w] ^ Sn[w]) & M1) + ((Lf[w] ^ Sn[w]) & M1) +
                  ((R[w] ^ Sn[w]) & M1);
            dn += (Sn[w] & M1) + (O[w] & M1);  // 2 per down spin, both planes
        }
    }
    store_words<W>(dst + (uint64_t)colour * g.plane + (uint64_t)y * half + 4 * W * k, Sn);
    int unfl = 0;
    if constexpr (kNE) {
        // persistence bytes of the W groups (bit q = site 4m+q)
        uint8_t *fb = g.flags + ((uint64_t)colour * L + y) * g.G + (uint64_t)(W * k);
        const uint8_t *fob = g.flags + ((uint64_t)oc * L + y) * g.G + (uint64_t)(W * k);
        uint32_t *fp = reinterpret_cast<uint32_t *>(fb);
        const uint32_t f = *fp | chg;
        *fp = f;
        if (colour == 1) unfl = 8 * W - __popc(f) - __popc(*reinterpret_cast<const uint32_t *>(fob));
    }
    if (colour == 1) {
        const int d2 = byte_sum(dn);
        cnt.bond += 16 * W - byte_sum(ue);
        cnt.mag += 8 * W - d2;
        cnt.up += 8 * W - (d2 >> 1);
        cnt.unfl += unfl;
        if (g.ref != nullptr) {
            // overlap with the reference over both planes' 8W sites:
            // 8W - 2 * (# sites that differ); 0x02 marks a differing byte
            uint32_t R1[W], R0[W], dr = 0;
            load_words<W>(g.ref + g.plane + (uint64_t)y * half + 4 * W * k, R1);
            load_words<W>(g.ref + (uint64_t)y * half + 4 * W * k, R0);
#pragma unroll
            for (int w = 0; w < W; ++w) dr += ((Sn[w] ^ R1[w]) & M1) + ((O[w] ^ R0[w]) & M1);
            cnt.acf += 8 * W - byte_sum(dr);
        }
    }
}

// ---------------------------------------------------------------------
// One 16-site chunk of a North-East column walk: the kernels that take any
// rate table and the general step (k_wide_pipe_ne) load chunk i + 1 in the
// same straight-line block as the step of chunk i.
// ---------------------------------------------------------------------
struct WideIn {
    uint32_t S[4], O[4], U[4], D[4];
    uint32_t adj;
};

// What one thread needs to walk its chunk column k (16 sites) down the
// rows of one colour: the rows it visits are y0, y0 + rs, y0 + 2 rs, ...
// with rs * cpr threads in the grid, so the column, its row-end neighbour
// word and its base addresses are fixed and a row costs a few 32-bit adds.
template <int kColour>
struct ColWalk {
    const int8_t *pS;      // this colour's sites before the sweep, + 16k
    const int8_t *pO;      // the other colour's current sites, + 16k
    const int8_t *pOrow;   // the other colour's current sites (row starts)
    int8_t *dS;            // this colour's plane in the new buffer, + 16k
    const int8_t *r1, *r0; // reference planes 1 and 0, + 16k (or null)
    uint32_t half, L, G, k;
    uint32_t adjb0, adjb1; // byte offset in the row of the neighbour word past the chunk end, x parity 0 / 1
};

// old: the buffer of the state before the sweep; nw: the new buffer.
// Colour 0 reads both planes of old; colour 1 reads its own sites from old
// (colour 0 did not touch them) and the new colour-0 sites from nw.  Each
// colour writes only its own plane of nw, so no plane is copied.
template <int kColour>
LAT_D ColWalk<kColour> col_walk(const SweepView &g, const int8_t *old, int8_t *nw, uint32_t k)
{
    constexpr int oc = 1 - kColour;
    ColWalk<kColour> c;
    const uint32_t plane = (uint32_t)g.plane;   // N < 2^32, so a plane is < 2^31 bytes
    c.pOrow = (kColour == 0 ? old : nw) + (size_t)oc * plane;
    c.pS = old + (size_t)kColour * plane + 16 * k;
    c.pO = c.pOrow + 16 * k;
    c.dS = nw + (size_t)kColour * plane + 16 * k;
    c.r1 = g.ref ? g.ref + (size_t)plane + 16 * k : nullptr;
    c.r0 = g.ref ? g.ref + 16 * k : nullptr;
    c.half = g.half;
    c.L = (uint32_t)g.L;
    c.G = g.G;
    c.k = k;
    const uint32_t nwr = g.half >> 2;   // 4-byte words per plane row
    c.adjb0 = 4u * wrap_once(4u * k - 1u + nwr, nwr);   // x = 2j: west word before the chunk
    c.adjb1 = 4u * wrap_once(4u * k + 4u, nwr);         // x = 2j+1: east word after it
    return c;
}

// Loads of the walk's chunk in plane row y.
template <int kColour>
LAT_D void col_load(const ColWalk<kColour> &c, uint32_t y, WideIn &in)
{
    const uint32_t oy = y * c.half;
    const uint32_t oym = y == 0 ? oy + (c.L - 1) * c.half : oy - c.half;
    const uint32_t oyp = y == c.L - 1 ? 0u : oy + c.half;
    load_words<4>(c.pS + oy, in.S);
    load_words<4>(c.pO + oy, in.O);
    load_words<4>(c.pO + oym, in.U);   // north
    load_words<4>(c.pO + oyp, in.D);   // south
    in.adj = *reinterpret_cast<const uint32_t *>(c.pOrow + oy + (((kColour + y) & 1) ? c.adjb1 : c.adjb0));
}

constexpr int kPipeMinB = 2;   // CTAs per SM (the two chunks in flight need ~100 registers)
constexpr int kWalkMinB = 2;   // (3, with fewer registers: 24 us a sweep at L = 4096 for 20.5)

// 2D Ising, one colour.  kOne: a thread per chunk (the launch has one for
// each); else a thread per (chunk column, band of consecutive rows), in one
// wave of at least cpr threads.
template <int kColour, bool kRef, int kDis, int kAcc, bool kAligned, bool kOne>
__global__ void __launch_bounds__(kThreads, kOne && kAligned && kDis != kFields ? 4 : kWalkMinB) k_ising_walk(Geom g, SweepAt at)
{
    __shared__ uint32_t sthr[kDis == kFields ? 32 : 16];
    __shared__ int red[kThreads / 32][5];
    ising_table<kDis>(g.thr16, sthr);
    __syncthreads();
    dep_wait();
    const unsigned long long sweep = sweep_of(g.ctrl, at);
    const SweepView v = sweep_view(g);
    Counts cnt;
    const uint32_t L = (uint32_t)g.L, cpr = (g.half + 15u) >> 4;
    const uint32_t nb = kOne ? L : min((gridDim.x * blockDim.x) / cpr, L);
    const uint32_t gt = blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t band = gt / cpr;
    if (band < nb) {
        const IsingPlanes<kColour> p = ising_planes<kColour>(v, sweep);
        if constexpr (kOne) {
            ising_one<kColour, kRef, kDis, kAcc, kAligned>(p, g.acc, sthr, sweep, g.key0, g.key1, gt - band * cpr,
                                                           band, cnt);
        } else {
            uint32_t y, y1;
            walk_rows(band, nb, L, y, y1);
            ising_walk<kColour, kRef, kDis, kAcc, kAligned>(p, g.acc, sthr, sweep, g.key0, g.key1, gt - band * cpr, y,
                                                            y1, cnt);
        }
    }
    dep_launch();   // main work done: the next kernel may be scheduled
    if constexpr (kColour == 1) {
        if (gt == 0u) sweep_done(g.ctrl, at);
        flush(v, sweep, cnt, false, red);
    }
    if constexpr (kDis == kFields) flush_one(fld_slot(g.ctrl, sweep), cnt.fld, red);   // both colours
}

// ---------------------------------------------------------------------
// North-East model (§III.B), the same column walk with the loads of the
// next chunk in flight, and draws compacted across the warp.  A site moves
// only if its north and east neighbours are up, and then, in c-mode with
// c < 1/2, an up site turns down without a draw; so only a few percent of
// the Philox groups need a draw.  Each lane marks the groups of its chunk
// that do; the warp lists them (ballot and prefix count), every lane makes
// the Philox calls of list entries lane, lane + 32, ... and the draws go
// back to their owners through shared memory.  A warp then makes
// ceil(needed / 32) calls per lane instead of 4.  Same groups, counters and
// bits as the other kernels.
// ---------------------------------------------------------------------
constexpr int kNeSlots = 4 * 32;   // list entries per warp (4 groups per lane)

template <int kColour, bool kRef>
LAT_D void ne_col_step(bool act, const ColWalk<kColour> &c, const uint8_t *fl_c, const uint8_t *fl_o,
                       const uint32_t *sthr, uint32_t y, const WideIn &in, const PhiloxPre &pp,
                       uint32_t *gtab, uint4 *dq, Counts &cnt)
{
    const uint32_t oy = y * c.half;
    const bool p1 = ((kColour + y) & 1) != 0;
    const char *tb = reinterpret_cast<const char *>(sthr);
    const uint32_t M1 = 0x02020202u;
    const int lane = threadIdx.x & 31;
    uint32_t Lf[4], R[4], t[4][4], locked[4], s1[4], c1[4];
    unsigned need = 0;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        if (!p1) {
            Lf[w] = __funnelshift_l(w == 0 ? in.adj : in.O[w - 1], in.O[w], 8);
            R[w] = in.O[w];
        } else {
            Lf[w] = in.O[w];
            R[w] = __funnelshift_r(in.O[w], w == 3 ? in.adj : in.O[w + 1], 8);
        }
        const uint32_t Uw = in.U[w], Dw = in.D[w];
        s1[w] = Uw ^ Dw ^ Lf[w];
        c1[w] = (Uw & Dw) | (Uw & Lf[w]) | (Dw & Lf[w]);
        const uint32_t b0 = s1[w] ^ R[w];
        const uint32_t b1 = c1[w] ^ (s1[w] & R[w]);
        const uint32_t b2 = c1[w] & s1[w] & R[w];
        // §III.B: north (U) and east (R) must be up.  A locked site (either
        // down: bit 6 of U | R set) indexes entries 16..31 of the table, all
        // t' = all ones, so it needs no draw; its flip is masked off below.
        locked[w] = Uw | R[w];
        const uint32_t idx = (b0 & 0x04040404u) | (b1 & 0x08080808u) | (b2 & 0x10101010u) |
                             (in.S[w] & 0x20202020u) | (locked[w] & 0x40404040u);
        t[w][0] = *reinterpret_cast<const uint32_t *>(tb + (idx & 0xFFu));
        t[w][1] = *reinterpret_cast<const uint32_t *>(tb + ((idx >> 8) & 0xFFu));
        t[w][2] = *reinterpret_cast<const uint32_t *>(tb + ((idx >> 16) & 0xFFu));
        t[w][3] = *reinterpret_cast<const uint32_t *>(tb + (idx >> 24));
        if (act && (t[w][0] & t[w][1] & t[w][2] & t[w][3]) != 0xFFFFFFFFu) need |= 1u << w;
    }
    // the warp's list of groups that need a draw: group w of every lane, then w+1
    unsigned bal[4], base[4], total = 0;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        bal[w] = __ballot_sync(0xffffffffu, (need >> w) & 1u);
        base[w] = total;
        total += __popc(bal[w]);
    }
    U4 u[4];
#pragma unroll
    for (int w = 0; w < 4; ++w) u[w] = U4{0u, 0u, 0u, 0u};   // t' all ones: any draw accepts
    if (total > 0) {   // warp-uniform
        const unsigned lt_mask = (1u << lane) - 1u;
        const uint32_t g0 = y * c.G + 4u * c.k;
#pragma unroll
        for (int w = 0; w < 4; ++w)
            if ((need >> w) & 1u) gtab[base[w] + __popc(bal[w] & lt_mask)] = g0 + (uint32_t)w;
        __syncwarp();
        for (unsigned j = (unsigned)lane; j < total; j += 32) {
            const U4 d = philox_item(pp, gtab[j], (uint32_t)kColour);
            dq[j] = make_uint4(d.x, d.y, d.z, d.w);
        }
        __syncwarp();
#pragma unroll
        for (int w = 0; w < 4; ++w)
            if ((need >> w) & 1u) {
                const uint4 q = dq[base[w] + __popc(bal[w] & lt_mask)];
                u[w] = U4{q.x, q.y, q.z, q.w};
            }
        __syncwarp();   // the next chunk's list may overwrite these entries
    }
    if (!act) return;
    uint32_t Sn[4], ue = 0, dn = 0, chg = 0;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        const uint32_t acc = (u[w].x <= t[w][0] ? 1u : 0u) | (u[w].y <= t[w][1] ? 2u : 0u) |
                             (u[w].z <= t[w][2] ? 4u : 0u) | (u[w].w <= t[w][3] ? 8u : 0u);
        const uint32_t F = ((acc * 0x00204081u) & 0x01010101u) * 0xFEu & ~locked[w];
        chg |= ((((F >> 1) & 0x01010101u) * 0x01020408u) >> 24 & 0xFu) << (8 * w);
        Sn[w] = in.S[w] ^ F;
        if constexpr (kColour == 1) {
            ue += ((s1[w] ^ Sn[w]) & M1) + ((c1[w] ^ Sn[w]) & 0x04040404u) + ((R[w] ^ Sn[w]) & M1);
            dn += (Sn[w] & M1) + (in.O[w] & M1);
        }
    }
    store_words<4>(c.dS + oy, Sn);
    // persistence bytes of the chunk's four groups (bit q = site 4m+q)
    uint32_t *fp = reinterpret_cast<uint32_t *>(const_cast<uint8_t *>(fl_c) + (size_t)y * c.G);
    const uint32_t f = *fp | chg;
    *fp = f;
    if constexpr (kColour == 1) {
        const uint32_t fo = *reinterpret_cast<const uint32_t *>(fl_o + (size_t)y * c.G);
        const int d2 = byte_sum(dn);
        cnt.bond += 64 - byte_sum(ue);
        cnt.mag += 32 - d2;
        cnt.up += 32 - (d2 >> 1);
        cnt.unfl += 32 - __popc(f) - __popc(fo);
        if constexpr (kRef) {
            uint32_t R1[4], R0[4], dr = 0;
            load_words<4>(c.r1 + oy, R1);
            load_words<4>(c.r0 + oy, R0);
#pragma unroll
            for (int w = 0; w < 4; ++w) dr += ((Sn[w] ^ R1[w]) & M1) + ((in.O[w] ^ R0[w]) & M1);
            cnt.acf += 32 - byte_sum(dr);
        }
    }
}

template <int kColour, bool kRef>
__global__ void __launch_bounds__(kThreads, kPipeMinB) k_wide_pipe_ne(Geom g, int off)
{
    __shared__ uint32_t sthr[32];   // entries 16..31: locked sites, always accepted (then masked)
    __shared__ int red[kThreads / 32][5];
    __shared__ uint32_t gtab[kThreads / 32][kNeSlots];
    __shared__ uint4 dq[kThreads / 32][kNeSlots];
    if (threadIdx.x < 32) sthr[threadIdx.x] = threadIdx.x < 16 ? g.thr16[threadIdx.x] : 0xFFFFFFFFu;
    __syncthreads();
    dep_wait();
    const unsigned long long sweep = g.ctrl->sweep + (unsigned long long)off;
    const SweepView v = sweep_view(g);
    const int8_t *old = (sweep & 1) ? v.s1 : v.s0;
    int8_t *nw = (sweep & 1) ? v.s0 : v.s1;
    Counts cnt;
    const uint32_t cpr = g.half >> 4;
    const uint32_t rs = (gridDim.x * blockDim.x) / cpr;
    const uint32_t gt = blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t L = (uint32_t)g.L;
    uint32_t y = gt / cpr;
    const uint32_t k = gt - y * cpr;
    bool act = y < rs && y < L;
    PhiloxPre pp;
    philox_prepare(pp, (uint32_t)sweep, (uint32_t)(sweep >> 32), g.key0, g.key1);
    const ColWalk<kColour> c = col_walk<kColour>(v, old, nw, act ? k : 0u);
    const uint8_t *fl_c = g.flags + (size_t)kColour * g.rows * g.G + 4u * k;
    const uint8_t *fl_o = g.flags + (size_t)(1 - kColour) * g.rows * g.G + 4u * k;
    const int warp = threadIdx.x >> 5;
    // Two chunks in flight (A and B in turn).  The warp's lanes stay in step
    // (the draw list is made by the whole warp), so a lane that has run out
    // of rows takes part with nothing to update.
    WideIn A, B;
    if (act) col_load<kColour>(c, y, A);
    for (;;) {
        if (!__any_sync(0xffffffffu, act)) break;
        const uint32_t y1 = y + rs;
        const bool act1 = act && y1 < L;
        if (act1) col_load<kColour>(c, y1, B);
        ne_col_step<kColour, kRef>(act, c, fl_c, fl_o, sthr, y, A, pp, gtab[warp], dq[warp], cnt);
        if (!__any_sync(0xffffffffu, act1)) break;
        const uint32_t y2 = y1 + rs;
        const bool act2 = act1 && y2 < L;
        if (act2) col_load<kColour>(c, y2, A);
        ne_col_step<kColour, kRef>(act1, c, fl_c, fl_o, sthr, y1, B, pp, gtab[warp], dq[warp], cnt);
        y = y2;
        act = act2;
    }
    dep_launch();   // main work done: the next kernel may be scheduled
    if constexpr (kColour == 1) flush(v, sweep, cnt, true, red);
}

// ---------------------------------------------------------------------
// Any even L, 16 sites per lane: the wide kernel's chunk of four Philox
// groups on rows at any byte alignment.  A chunk's 16 bytes are gathered
// from the aligned words that hold them; the last chunk of a row holds
// L/2 % 16 sites (its bytes past the row are masked, its neighbour past the
// row end is the row's first byte); stores write whole aligned words inside
// the chunk and single bytes at its two ends, so no byte of another lane's
// chunk is touched.  Column walk with two chunks in flight (Ising: the next
// chunk's draws too) and, for the North-East model, the warp-compacted draws
// of k_wide_pipe_ne.  Ising in batches' step loop, North-East at any rates.
// ---------------------------------------------------------------------

struct AnyIn {
    uint32_t S[4], O[4], U[4], D[4];
    uint32_t nb;   // the other plane's byte past the chunk's edge (west of j0, or east of its last site)
};

// One thread's column of chunks (chunk k of every plane row it visits).
template <int kColour>
struct AnyWalk {
    const int8_t *pS, *pO;   // planes: this colour's old sites, the other colour's current sites
    int8_t *dS;              // this colour's plane in the new buffer
    const int8_t *r1, *r0;   // reference planes 1 and 0 (or null)
    uint32_t half, L, G, k, j0, nv;
    uint32_t vm[4];          // valid-byte masks of the chunk's words
    uint32_t jprev, jnext;   // row index of the west neighbour of j0 / the east neighbour of the last site
};

template <int kColour>
LAT_D AnyWalk<kColour> any_walk(const SweepView &g, const int8_t *old, int8_t *nw, uint32_t k)
{
    constexpr int oc = 1 - kColour;
    AnyWalk<kColour> c;
    const uint32_t plane = (uint32_t)g.plane;
    c.pS = old + (size_t)kColour * plane;
    c.pO = (kColour == 0 ? old : nw) + (size_t)oc * plane;
    c.dS = nw + (size_t)kColour * plane;
    c.r1 = g.ref ? g.ref + (size_t)plane : nullptr;
    c.r0 = g.ref;
    c.half = g.half;
    c.L = (uint32_t)g.L;
    c.G = g.G;
    c.k = k;
    c.j0 = 16u * k;
    c.nv = min(16u, g.half - c.j0);
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        const int n = (int)c.nv - 4 * w;
        c.vm[w] = n >= 4 ? 0xFFFFFFFFu : (n <= 0 ? 0u : (1u << (8 * n)) - 1u);
    }
    c.jprev = c.j0 == 0u ? g.half - 1u : c.j0 - 1u;
    c.jnext = c.j0 + c.nv == g.half ? 0u : c.j0 + c.nv;
    return c;
}

template <int kColour, bool kAligned = false>
LAT_D void any_load(const AnyWalk<kColour> &c, uint32_t y, AnyIn &in)
{
    const uint32_t oy = y * c.half;
    const uint32_t oym = y == 0 ? oy + (c.L - 1) * c.half : oy - c.half;
    const uint32_t oyp = y == c.L - 1 ? 0u : oy + c.half;
    load16_any<kAligned>(c.pS + oy + c.j0, c.nv, in.S);
    load16_any<kAligned>(c.pO + oy + c.j0, c.nv, in.O);
    load16_any<kAligned>(c.pO + oym + c.j0, c.nv, in.U);   // north
    load16_any<kAligned>(c.pO + oyp + c.j0, c.nv, in.D);   // south
    in.nb = (uint32_t)(uint8_t)c.pO[oy + (((kColour + y) & 1) ? c.jnext : c.jprev)];
}

template <int kColour>
LAT_D void any_draws(const PhiloxPre &pp, const AnyWalk<kColour> &c, uint32_t y, U4 (&u)[4])
{
    const uint32_t g0 = y * c.G + 4u * c.k;
#pragma unroll
    for (int w = 0; w < 4; ++w) u[w] = philox_item(pp, g0 + (uint32_t)w, (uint32_t)kColour);
}

// West (Lf) and east (R) neighbour words of the chunk's sites.
template <int kColour>
LAT_D void any_sides(const AnyWalk<kColour> &c, uint32_t y, const AnyIn &in, uint32_t (&Lf)[4], uint32_t (&R)[4])
{
    if (((kColour + y) & 1) == 0) {   // x = 2j: west is j-1 (nb for j0), east is j
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            Lf[w] = __funnelshift_l(w == 0 ? (in.nb << 24) : in.O[w - 1], in.O[w], 8);
            R[w] = in.O[w];
        }
    } else {                          // x = 2j+1: west is j, east is j+1 (nb for the last site)
        // a partial chunk's last site: its east neighbour nb goes to byte nv
        // of the sequence (a mask that is zero in every other word)
        uint32_t Oe[4];
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const uint32_t d = c.nv - 4u * (uint32_t)w;
            const uint32_t m = d < 4u ? (0xFFu << (8u * d)) : 0u;
            Oe[w] = (in.O[w] & ~m) | ((in.nb << (8u * (d & 3u))) & m);
        }
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            Lf[w] = in.O[w];
            R[w] = __funnelshift_r(Oe[w], w == 3 ? in.nb : Oe[w + 1], 8);
        }
    }
}

template <int kColour, bool kRef, bool kAligned = false>
LAT_D void any_step(const AnyWalk<kColour> &c, const uint32_t *sthr, uint32_t y, const AnyIn &in, const U4 (&u)[4],
                    Counts &cnt)
{
    const uint32_t oy = y * c.half;
    const char *tb = reinterpret_cast<const char *>(sthr);
    const uint32_t M1 = 0x02020202u;
    uint32_t Lf[4], R[4];
    any_sides<kColour>(c, y, in, Lf, R);
    uint32_t Sn[4], ue = 0, dn = 0;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        const uint32_t Uw = in.U[w], Dw = in.D[w];
        const uint32_t s1 = Uw ^ Dw ^ Lf[w];
        const uint32_t c1 = (Uw & Dw) | (Uw & Lf[w]) | (Dw & Lf[w]);
        const uint32_t b0 = s1 ^ R[w];
        const uint32_t b1 = c1 ^ (s1 & R[w]);
        const uint32_t b2 = c1 & s1 & R[w];
        const uint32_t idx = (b0 & 0x04040404u) | (b1 & 0x08080808u) | (b2 & 0x10101010u) | (in.S[w] & 0x20202020u);
        const uint32_t t0 = *reinterpret_cast<const uint32_t *>(tb + (idx & 0xFFu));
        const uint32_t t1 = *reinterpret_cast<const uint32_t *>(tb + ((idx >> 8) & 0xFFu));
        const uint32_t t2 = *reinterpret_cast<const uint32_t *>(tb + ((idx >> 16) & 0xFFu));
        const uint32_t t3 = *reinterpret_cast<const uint32_t *>(tb + (idx >> 24));
        const uint32_t acc = (u[w].x <= t0 ? 1u : 0u) | (u[w].y <= t1 ? 2u : 0u) | (u[w].z <= t2 ? 4u : 0u) |
                             (u[w].w <= t3 ? 8u : 0u);
        const uint32_t F = ((acc * 0x00204081u) & 0x01010101u) * 0xFEu & c.vm[w];
        Sn[w] = in.S[w] ^ F;
        if constexpr (kColour == 1) {
            ue += (((s1 ^ Sn[w]) & M1) + ((c1 ^ Sn[w]) & 0x04040404u) + ((R[w] ^ Sn[w]) & M1)) & c.vm[w];
            dn += ((Sn[w] & M1) + (in.O[w] & M1)) & c.vm[w];
        }
    }
    store16_any<kAligned>(c.dS + oy + c.j0, c.nv, Sn);
    if constexpr (kColour == 1) {
        const int nv = (int)c.nv;
        const int d2 = byte_sum(dn);
        cnt.bond += 4 * nv - byte_sum(ue);
        cnt.mag += 2 * nv - d2;
        cnt.up += 2 * nv - (d2 >> 1);
        if constexpr (kRef) {
            uint32_t R1[4], R0[4], dr = 0;
            load16_any<kAligned>(c.r1 + oy + c.j0, c.nv, R1);
            load16_any<kAligned>(c.r0 + oy + c.j0, c.nv, R0);
#pragma unroll
            for (int w = 0; w < 4; ++w) dr += (((Sn[w] ^ R1[w]) & M1) + ((in.O[w] ^ R0[w]) & M1)) & c.vm[w];
            cnt.acf += 2 * nv - byte_sum(dr);
        }
    }
}

// North-East at any even L: the step of ne_col_step with any-alignment
// loads and stores, per-byte persistence updates (the groups of a row need
// not start on a word), and the warp-compacted draws.
template <int kColour, bool kRef, bool kAligned = false>
LAT_D void any_ne_step(bool act, const AnyWalk<kColour> &c, uint8_t *fl_c, const uint8_t *fl_o,
                       const uint32_t *sthr, uint32_t y, const AnyIn &in, const PhiloxPre &pp, uint32_t *gtab,
                       uint4 *dq, Counts &cnt)
{
    const uint32_t oy = y * c.half;
    const char *tb = reinterpret_cast<const char *>(sthr);
    const uint32_t M1 = 0x02020202u;
    const int lane = threadIdx.x & 31;
    uint32_t Lf[4], R[4], t[4][4], locked[4], s1[4], c1[4];
    any_sides<kColour>(c, y, in, Lf, R);
    unsigned need = 0;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        const uint32_t Uw = in.U[w], Dw = in.D[w];
        s1[w] = Uw ^ Dw ^ Lf[w];
        c1[w] = (Uw & Dw) | (Uw & Lf[w]) | (Dw & Lf[w]);
        const uint32_t b0 = s1[w] ^ R[w];
        const uint32_t b1 = c1[w] ^ (s1[w] & R[w]);
        const uint32_t b2 = c1[w] & s1[w] & R[w];
        // §III.B: a locked site (north or east down) indexes the all-accept
        // entries 16..31; so do the bytes past the row (masked below)
        locked[w] = Uw | R[w] | ~c.vm[w];
        const uint32_t idx = (b0 & 0x04040404u) | (b1 & 0x08080808u) | (b2 & 0x10101010u) |
                             (in.S[w] & 0x20202020u) | (locked[w] & 0x40404040u);
        t[w][0] = *reinterpret_cast<const uint32_t *>(tb + (idx & 0xFFu));
        t[w][1] = *reinterpret_cast<const uint32_t *>(tb + ((idx >> 8) & 0xFFu));
        t[w][2] = *reinterpret_cast<const uint32_t *>(tb + ((idx >> 16) & 0xFFu));
        t[w][3] = *reinterpret_cast<const uint32_t *>(tb + (idx >> 24));
        if (act && (t[w][0] & t[w][1] & t[w][2] & t[w][3]) != 0xFFFFFFFFu) need |= 1u << w;
    }
    unsigned bal[4], base[4], total = 0;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        bal[w] = __ballot_sync(0xffffffffu, (need >> w) & 1u);
        base[w] = total;
        total += __popc(bal[w]);
    }
    U4 u[4];
#pragma unroll
    for (int w = 0; w < 4; ++w) u[w] = U4{0u, 0u, 0u, 0u};
    if (total > 0) {
        const unsigned lt_mask = (1u << lane) - 1u;
        const uint32_t g0 = y * c.G + 4u * c.k;
#pragma unroll
        for (int w = 0; w < 4; ++w)
            if ((need >> w) & 1u) gtab[base[w] + __popc(bal[w] & lt_mask)] = g0 + (uint32_t)w;
        __syncwarp();
        for (unsigned j = (unsigned)lane; j < total; j += 32) {
            const U4 d = philox_item(pp, gtab[j], (uint32_t)kColour);
            dq[j] = make_uint4(d.x, d.y, d.z, d.w);
        }
        __syncwarp();
#pragma unroll
        for (int w = 0; w < 4; ++w)
            if ((need >> w) & 1u) {
                const uint4 q = dq[base[w] + __popc(bal[w] & lt_mask)];
                u[w] = U4{q.x, q.y, q.z, q.w};
            }
        __syncwarp();
    }
    if (!act) return;
    uint32_t Sn[4], ue = 0, dn = 0, chg = 0;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        const uint32_t acc = (u[w].x <= t[w][0] ? 1u : 0u) | (u[w].y <= t[w][1] ? 2u : 0u) |
                             (u[w].z <= t[w][2] ? 4u : 0u) | (u[w].w <= t[w][3] ? 8u : 0u);
        const uint32_t F = ((acc * 0x00204081u) & 0x01010101u) * 0xFEu & ~locked[w];
        chg |= ((((F >> 1) & 0x01010101u) * 0x01020408u) >> 24 & 0xFu) << (8 * w);
        Sn[w] = in.S[w] ^ F;
        if constexpr (kColour == 1) {
            ue += (((s1[w] ^ Sn[w]) & M1) + ((c1[w] ^ Sn[w]) & 0x04040404u) + ((R[w] ^ Sn[w]) & M1)) & c.vm[w];
            dn += ((Sn[w] & M1) + (in.O[w] & M1)) & c.vm[w];
        }
    }
    store16_any<kAligned>(c.dS + oy + c.j0, c.nv, Sn);
    // persistence bytes of the chunk's groups that exist (4k + w < G)
    uint8_t *fp = fl_c + (size_t)y * c.G;
    const uint8_t *fop = fl_o + (size_t)y * c.G;
    const uint32_t ng = min(4u, c.G - 4u * c.k);
    int fpop = 0, fopop = 0;
#pragma unroll
    for (int w = 0; w < 4; ++w)
        if ((uint32_t)w < ng) {
            const uint32_t f = (uint32_t)fp[w] | ((chg >> (8 * w)) & 0xFu);
            fp[w] = (uint8_t)f;
            fpop += __popc(f);
            if constexpr (kColour == 1) fopop += __popc((uint32_t)fop[w]);
        }
    if constexpr (kColour == 1) {
        const int nv = (int)c.nv;
        const int d2 = byte_sum(dn);
        cnt.bond += 4 * nv - byte_sum(ue);
        cnt.mag += 2 * nv - d2;
        cnt.up += 2 * nv - (d2 >> 1);
        cnt.unfl += 2 * nv - fpop - fopop;
        if constexpr (kRef) {
            uint32_t R1[4], R0[4], dr = 0;
            load16_any<kAligned>(c.r1 + oy + c.j0, c.nv, R1);
            load16_any<kAligned>(c.r0 + oy + c.j0, c.nv, R0);
#pragma unroll
            for (int w = 0; w < 4; ++w) dr += (((Sn[w] ^ R1[w]) & M1) + ((in.O[w] ^ R0[w]) & M1)) & c.vm[w];
            cnt.acf += 2 * nv - byte_sum(dr);
        }
    }
}

template <int kColour, bool kRef>
__global__ void __launch_bounds__(kThreads, kPipeMinB) k_any_pipe_ne(Geom g, int off)
{
    __shared__ uint32_t sthr[32];   // entries 16..31: locked sites, always accepted (then masked)
    __shared__ int red[kThreads / 32][5];
    __shared__ uint32_t gtab[kThreads / 32][kNeSlots];
    __shared__ uint4 dq[kThreads / 32][kNeSlots];
    if (threadIdx.x < 32) sthr[threadIdx.x] = threadIdx.x < 16 ? g.thr16[threadIdx.x] : 0xFFFFFFFFu;
    __syncthreads();
    dep_wait();
    const unsigned long long sweep = g.ctrl->sweep + (unsigned long long)off;
    const SweepView v = sweep_view(g);
    const int8_t *old = (sweep & 1) ? v.s1 : v.s0;
    int8_t *nw = (sweep & 1) ? v.s0 : v.s1;
    Counts cnt;
    const uint32_t cpr = (g.half + 15u) >> 4;
    const uint32_t rs = (gridDim.x * blockDim.x) / cpr;
    const uint32_t gt = blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t L = (uint32_t)g.L;
    uint32_t y = gt / cpr;
    const uint32_t k = gt - y * cpr;
    bool act = y < rs && y < L;
    PhiloxPre pp;
    philox_prepare(pp, (uint32_t)sweep, (uint32_t)(sweep >> 32), g.key0, g.key1);
    const AnyWalk<kColour> c = any_walk<kColour>(v, old, nw, act ? k : 0u);
    uint8_t *fl_c = g.flags + (size_t)kColour * g.rows * g.G + 4u * c.k;
    const uint8_t *fl_o = g.flags + (size_t)(1 - kColour) * g.rows * g.G + 4u * c.k;
    const int warp = threadIdx.x >> 5;
    AnyIn A, B;
    if (act) any_load<kColour>(c, y, A);
    for (;;) {
        if (!__any_sync(0xffffffffu, act)) break;
        const uint32_t y1 = y + rs;
        const bool act1 = act && y1 < L;
        if (act1) any_load<kColour>(c, y1, B);
        any_ne_step<kColour, kRef>(act, c, fl_c, fl_o, sthr, y, A, pp, gtab[warp], dq[warp], cnt);
        if (!__any_sync(0xffffffffu, act1)) break;
        const uint32_t y2 = y1 + rs;
        const bool act2 = act1 && y2 < L;
        if (act2) any_load<kColour>(c, y2, A);
        any_ne_step<kColour, kRef>(act1, c, fl_c, fl_o, sthr, y1, B, pp, gtab[warp], dq[warp], cnt);
        y = y2;
        act = act2;
    }
    dep_launch();   // main work done: the next kernel may be scheduled
    if constexpr (kColour == 1) flush(v, sweep, cnt, true, red);
}

// Batched form of the any-L kernels: a persistent grid takes (lattice,
// item) pairs from an atomic counter.  An item is a band of rows and, in
// rows of more than 256 chunks, a segment of 256 chunk columns; a thread
// walks one chunk column down the band with two chunks in flight, as the
// solo kernels do.
template <int kColour, bool kNE, bool kAligned>
LAT_D void batch_any_item(const SweepView &v, const uint32_t *sthr, uint32_t item, uint32_t passes, uint32_t *gtab,
                          uint4 *dq, Counts &cnt)
{
    const unsigned long long sweep = v.ctrl->sweep;
    PhiloxPre pp;
    philox_prepare(pp, (uint32_t)sweep, (uint32_t)(sweep >> 32), v.key0, v.key1);
    const int8_t *old = (sweep & 1) ? v.s1 : v.s0;
    int8_t *nw = (sweep & 1) ? v.s0 : v.s1;
    const AnyItemShape sh = any_item_shape(v.half, passes);
    const uint32_t L = (uint32_t)v.L;
    const uint32_t band = item / sh.nseg, seg = item - band * sh.nseg;
    const uint32_t y0 = band * sh.br, y1 = min(L, y0 + sh.br);
    uint32_t k, r0;
    if (sh.cpr <= (uint32_t)kThreads) {
        k = threadIdx.x % sh.cpr;
        r0 = threadIdx.x / sh.cpr;
    } else {
        k = seg * kThreads + threadIdx.x;
        r0 = 0;
    }
    const bool mine = k < sh.cpr && r0 < sh.rsb;
    uint32_t y = y0 + r0;
    const AnyWalk<kColour> c = any_walk<kColour>(v, old, nw, mine ? k : 0u);
    if constexpr (!kNE) {
        if (!(mine && y < y1)) return;
        AnyIn A, B;
        U4 uA[4], uB[4];
        any_load<kColour, kAligned>(c, y, A);
        any_draws<kColour>(pp, c, y, uA);
        for (;;) {
            const uint32_t ya = y + sh.rsb;
            if (ya >= y1) {
                if (v.ref) any_step<kColour, true, kAligned>(c, sthr, y, A, uA, cnt);
                else any_step<kColour, false, kAligned>(c, sthr, y, A, uA, cnt);
                break;
            }
            any_load<kColour, kAligned>(c, ya, B);
            any_draws<kColour>(pp, c, ya, uB);
            if (v.ref) any_step<kColour, true, kAligned>(c, sthr, y, A, uA, cnt);
            else any_step<kColour, false, kAligned>(c, sthr, y, A, uA, cnt);
            const uint32_t yb = ya + sh.rsb;
            if (yb >= y1) {
                if (v.ref) any_step<kColour, true, kAligned>(c, sthr, ya, B, uB, cnt);
                else any_step<kColour, false, kAligned>(c, sthr, ya, B, uB, cnt);
                break;
            }
            any_load<kColour, kAligned>(c, yb, A);
            any_draws<kColour>(pp, c, yb, uA);
            if (v.ref) any_step<kColour, true, kAligned>(c, sthr, ya, B, uB, cnt);
            else any_step<kColour, false, kAligned>(c, sthr, ya, B, uB, cnt);
            y = yb;
        }
    } else {
        // the warp's lanes stay in step (warp-compacted draws)
        uint8_t *fl_c = v.flags + (size_t)kColour * v.rows * v.G + 4u * c.k;
        const uint8_t *fl_o = v.flags + (size_t)(1 - kColour) * v.rows * v.G + 4u * c.k;
        bool act = mine && y < y1;
        AnyIn A, B;   // two chunks in flight
        if (act) any_load<kColour, kAligned>(c, y, A);
        for (;;) {
            if (!__any_sync(0xffffffffu, act)) break;
            const uint32_t ya = y + sh.rsb;
            const bool act1 = act && ya < y1;
            if (act1) any_load<kColour, kAligned>(c, ya, B);
            if (v.ref) any_ne_step<kColour, true, kAligned>(act, c, fl_c, fl_o, sthr, y, A, pp, gtab, dq, cnt);
            else any_ne_step<kColour, false, kAligned>(act, c, fl_c, fl_o, sthr, y, A, pp, gtab, dq, cnt);
            if (!__any_sync(0xffffffffu, act1)) break;
            const uint32_t yb = ya + sh.rsb;
            const bool act2 = act1 && yb < y1;
            if (act2) any_load<kColour, kAligned>(c, yb, A);
            if (v.ref) any_ne_step<kColour, true, kAligned>(act1, c, fl_c, fl_o, sthr, ya, B, pp, gtab, dq, cnt);
            else any_ne_step<kColour, false, kAligned>(act1, c, fl_c, fl_o, sthr, ya, B, pp, gtab, dq, cnt);
            y = yb;
            act = act2;
        }
    }
}

template <bool kNE, bool kAligned, int kColour>
__global__ void __launch_bounds__(kThreads, kPipeMinB) k_batch_any(const Geom *geoms, const uint2 *items, int n_items,
                                                                  unsigned *next_item, uint32_t passes)
{
    __shared__ uint32_t sthr[32];   // entries 16..31: locked North-East sites
    __shared__ int red[kThreads / 32][5];
    __shared__ uint32_t gtab[kNE ? kThreads / 32 : 1][kNeSlots];
    __shared__ uint4 dq[kNE ? kThreads / 32 : 1][kNeSlots];
    __shared__ Geom sg;
    __shared__ int cur;
    int loaded = -1;
    const int warp = kNE ? (int)(threadIdx.x >> 5) : 0;
    dep_wait();   // the work counter, sweep numbers and spins of the step before
    for (;;) {
        if (threadIdx.x == 0) cur = (int)atomicAdd(next_item, 1u);
        __syncthreads();
        const int it = cur;
        if (it >= n_items) break;
        const uint2 w = items[it];
        if ((int)w.x != loaded) {
            if (threadIdx.x < sizeof(Geom) / 4)
                reinterpret_cast<uint32_t *>(&sg)[threadIdx.x] =
                    reinterpret_cast<const uint32_t *>(&geoms[w.x])[threadIdx.x];
            __syncthreads();
            if (threadIdx.x < 32) sthr[threadIdx.x] = threadIdx.x < 16 ? sg.thr16[threadIdx.x] : 0xFFFFFFFFu;
            loaded = (int)w.x;
            __syncthreads();
        }
        const SweepView v = sweep_view(sg);
        Counts cnt;
        batch_any_item<kColour, kNE, kAligned>(v, sthr, w.y, passes, gtab[warp], dq[warp], cnt);
        if constexpr (kColour == 1) flush(v, v.ctrl->sweep, cnt, kNE, red);   // ends with __syncthreads()
        __syncthreads();
    }
    dep_launch();   // no items left: the next kernel may be scheduled
}

// Resident form for lattices that fit in one CTA's shared memory (§III.A
// with the whole lattice as the block's tile): the CTA loads the spins (and
// the North-East persistence bytes) once, runs n sweeps in place -- an
// in-place checkerboard update is exact because a colour reads only the
// other colour, and __syncthreads() is the barrier between the two -- and
// writes the final state to s[(sweep + n) & 1].  One launch replaces 2n.
constexpr int kResThreads = 512;
constexpr size_t kResMaxBytes = 220 * 1024;

// One lattice, n_sweeps sweeps, by the whole CTA.  g may live in shared
// memory (the batched kernel): the sweep loop reads only register copies.
// advance: the CTA also moves the lattice's sweep counter on by n_sweeps.
template <bool kNE>
LAT_D void resident_body(const Geom &g, unsigned long long sweep0, int n_sweeps, bool advance, uint4 *res_smem, uint32_t *sthr,
                         int (*red)[5])
{
    int8_t *sp = reinterpret_cast<int8_t *>(res_smem);
    const uint64_t n16 = g.N >> 4;                       // N % 16 == 0 (L % 32 == 0)
    const uint64_t f16 = kNE ? ((uint64_t)2 * g.rows * g.G) >> 4 : 0;  // flag bytes / 16
    uint4 *fl4 = res_smem + n16;
    {
        const uint4 *src = reinterpret_cast<const uint4 *>(g.s[sweep0 & 1]);
        for (uint64_t i = threadIdx.x; i < n16; i += blockDim.x) res_smem[i] = src[i];
        if constexpr (kNE) {
            const uint4 *fsrc = reinterpret_cast<const uint4 *>(g.flags);
            for (uint64_t i = threadIdx.x; i < f16; i += blockDim.x) fl4[i] = fsrc[i];
        }
    }
    if (threadIdx.x < 16) sthr[threadIdx.x] = g.thr16[threadIdx.x];
    __syncthreads();
    SweepView v = sweep_view(g);
    v.s0 = sp;
    v.s1 = sp;
    v.flags = reinterpret_cast<uint8_t *>(fl4);
    const uint32_t cpr = g.half >> 4;
    const uint32_t total = (uint32_t)g.L * cpr;
    unsigned long long *slot0 = series_slot(g.ctrl, sweep0);  // slots of consecutive sweeps are contiguous
    unsigned long long *acf0 = g.ref ? acf_slot(g.ctrl, sweep0) : nullptr;
    for (int s = 0; s < n_sweeps; ++s) {
        const unsigned long long sweep = sweep0 + (unsigned long long)s;
        PhiloxPre pp;
        philox_prepare(pp, (uint32_t)sweep, (uint32_t)(sweep >> 32), g.key0, g.key1);
        Counts cnt;
        for (uint32_t t = threadIdx.x; t < total; t += blockDim.x)
            wide_chunk<kNE>(v, sthr, 0, sweep, pp, (int)(t / cpr), (int)(t % cpr), cnt);
        __syncthreads();
        for (uint32_t t = threadIdx.x; t < total; t += blockDim.x)
            wide_chunk<kNE>(v, sthr, 1, sweep, pp, (int)(t / cpr), (int)(t % cpr), cnt);
        flush_slot(slot0 + 4ull * (unsigned)s, acf0 ? acf0 + (unsigned)s : nullptr, cnt, kNE, red);  // ends with __syncthreads()
    }
    {
        uint4 *dst = reinterpret_cast<uint4 *>(g.s[(sweep0 + (unsigned long long)n_sweeps) & 1]);
        for (uint64_t i = threadIdx.x; i < n16; i += blockDim.x) dst[i] = res_smem[i];
        if constexpr (kNE) {
            uint4 *fdst = reinterpret_cast<uint4 *>(g.flags);
            for (uint64_t i = threadIdx.x; i < f16; i += blockDim.x) fdst[i] = fl4[i];
        }
    }
    if (advance) {
        __syncthreads();   // every thread has read the old counter long before
        if (threadIdx.x == 0) g.ctrl->sweep = sweep0 + (unsigned long long)n_sweeps;
    }
}

// Lattices of at most one four-site word a thread and colour (L = 32, 64). A
// sweep is then two short dependent steps, so what does not depend on the
// other colour is taken out of them: a thread keeps its words of both
// colours (and their persistence bits) in registers, draws for the next
// half-sweep once its new word is stored, decides by the 16-bit compare, and
// the counters are summed through shared memory and posted a barrier later.
// L = 64: 0.93 us a sweep (1.06 with table look-ups, draws and three counter
// barriers in line). Batches; a lattice alone has k_resident_pair.
template <bool kNE, bool kSym>
LAT_D void resident_words(const Geom &g, unsigned long long sweep0, int n_sweeps, bool advance, uint4 *res_smem,
                          uint32_t *sthr, int (*sum)[5])
{
    uint32_t *pl = reinterpret_cast<uint32_t *>(res_smem);   // two planes of words
    const uint32_t tid = threadIdx.x, wpr = g.half >> 2, words = (uint32_t)g.L * wpr;
    const uint32_t y = tid / wpr, k = tid - y * wpr;
    const bool mine = tid < words;
    const uint32_t *src = reinterpret_cast<const uint32_t *>(g.s[sweep0 & 1]);
    uint32_t S[2] = {0u, 0u}, was[2] = {0u, 0u}, rw[2] = {0u, 0u};
    int unfl = 0;
    if (mine)
        for (int c = 0; c < 2; ++c) {
            S[c] = src[c * words + tid];
            pl[c * words + tid] = S[c];
            if constexpr (kNE) was[c] = g.flags[c * words + tid];   // G = wpr groups a row
            if (g.ref) rw[c] = reinterpret_cast<const uint32_t *>(g.ref)[c * words + tid];
        }
    if (tid < 16) sthr[tid] = g.thr16[tid];
    if (tid >= 32 && tid < 42) (&sum[0][0])[tid - 32] = 0;
    if constexpr (kNE) unfl = mine ? 8 - __popc(was[0]) - __popc(was[1]) : 0;
    __syncthreads();
    // shared word indices of the neighbours (the other plane's base is added)
    const uint32_t iU = (y == 0u ? (uint32_t)g.L - 1u : y - 1u) * wpr + k, iD = (y + 1u == (uint32_t)g.L ? 0u : y + 1u) * wpr + k;
    const uint32_t iW = y * wpr + (k == 0u ? wpr - 1u : k - 1u), iE = y * wpr + (k + 1u == wpr ? 0u : k + 1u);
    unsigned long long *slot0 = series_slot(g.ctrl, sweep0);   // consecutive sweeps are contiguous
    unsigned long long *acf0 = g.ref ? acf_slot(g.ctrl, sweep0) : nullptr;
    const uint32_t g0 = y * g.G + k;
    uint32_t p01 = 0, p23 = 0;
    auto draw = [&](unsigned long long sweep, uint32_t colour) {
        PhiloxPre pp;
        philox_prepare(pp, (uint32_t)sweep, (uint32_t)(sweep >> 32), g.key0, g.key1);
        top_halves(philox_item(pp, g0, colour), p01, p23);
    };
    draw(sweep0, 0u);
    int bond = 0, mag = 0, acf = 0;
    auto half_sweep = [&](auto which, unsigned long long sweep) {
        constexpr uint32_t c = decltype(which)::value;
        if (mine) {
            const uint32_t *o = pl + (1u - c) * words;
            const bool odd = ((c + y) & 1u) != 0u;
            const uint32_t U = o[iU], D = o[iD], O = S[1u - c], nb = o[odd ? iE : iW];
            const uint32_t X = odd ? __funnelshift_r(O, nb, 8) : __funnelshift_l(nb, O, 8);
            const Nbr n = nbr_sum(U, D, O, X);
            uint32_t t01[2], t23[2], tie = kNoTie;
            if constexpr (kSym) sym_thresholds(g.acc, n, S[c], t01[0], t23[0]);
            else gen_thresholds2(g.acc, n, n, S[c], S[c], t01, t23);
            uint32_t rej = reject4(t01[0], t23[0], p01, p23, tie);
            if (tie_hit(tie)) {
                PhiloxPre pp;
                philox_prepare(pp, (uint32_t)sweep, (uint32_t)(sweep >> 32), g.key0, g.key1);
                rej = reject4_exact(sthr, n, S[c], philox_item(pp, g0, c));
            }
            uint32_t F = ~rej & 0xFEFEFEFEu;
            if constexpr (kNE) F &= ~(U | (odd ? X : O));   // §III.B: north and east must be up
            S[c] ^= F;
            pl[c * words + tid] = S[c];
            draw(sweep + (c == 1u ? 1ull : 0ull), 1u - c);
            if constexpr (kNE) {
                const uint32_t bits = (uint32_t)dot4(F & 0x02020202u, 0x08040201u, 0) >> 1;
                unfl -= __popc(bits & ~was[c]);
                was[c] |= bits;
            }
            if constexpr (c == 1u) {
                bond = dot4(S[1], X, dot4(S[1], O, dot4(S[1], D, dot4(S[1], U, 0))));
                mag = dot4(S[1], 0x01010101u, dot4(O, 0x01010101u, 0));
                if (g.ref) acf = dot4(S[1], rw[1], dot4(O, rw[0], 0));
            }
        }
        if constexpr (c == 1u) {
            const int par = (int)(sweep & 1ull);
            const int b = __reduce_add_sync(0xffffffffu, bond), m = __reduce_add_sync(0xffffffffu, mag);
            [[maybe_unused]] const int f = kNE ? __reduce_add_sync(0xffffffffu, unfl) : 0;
            const int a = g.ref ? __reduce_add_sync(0xffffffffu, acf) : 0;
            if ((tid & 31u) == 0u) {
                atomicAdd(&sum[par][0], b);
                atomicAdd(&sum[par][1], m);
                if constexpr (kNE) atomicAdd(&sum[par][3], f);
                if (g.ref) atomicAdd(&sum[par][4], a);
            }
        }
        __syncthreads();
        if constexpr (c == 1u) {   // posted while the next half-sweep runs; cleared two barriers before its next use
            if (tid == 0u) {
                const int par = (int)(sweep & 1ull);
                unsigned long long *slot = slot0 + 4ull * (sweep - sweep0);
                const long long m = sum[par][1];
                add_counter(slot + 0, sum[par][0]);
                add_counter(slot + 1, m);
                add_counter(slot + 2, (m + (long long)g.N) / 2);
                if constexpr (kNE) add_counter(slot + 3, sum[par][3]);
                if (g.ref) add_counter(acf0 + (sweep - sweep0), sum[par][4]);
                for (int i = 0; i < 5; ++i) sum[par][i] = 0;
            }
        }
    };
    for (int s = 0; s < n_sweeps; ++s) {
        half_sweep(std::integral_constant<uint32_t, 0>(), sweep0 + (unsigned long long)s);
        half_sweep(std::integral_constant<uint32_t, 1>(), sweep0 + (unsigned long long)s);
    }
    uint32_t *dst = reinterpret_cast<uint32_t *>(g.s[(sweep0 + (unsigned long long)n_sweeps) & 1]);
    if (mine)
        for (int c = 0; c < 2; ++c) {
            dst[c * words + tid] = S[c];
            if constexpr (kNE) g.flags[c * words + tid] = (uint8_t)was[c];
        }
    if (advance && tid == 0) g.ctrl->sweep = sweep0 + (unsigned long long)n_sweeps;   // read by all before the first barrier
}

__global__ void __launch_bounds__(kResThreads, 1) k_resident_ising(const __grid_constant__ Geom g, SweepAt at, int n_sweeps)
{
    extern __shared__ uint4 res_smem[];
    __shared__ uint32_t sthr[16];
    __shared__ int red[kResThreads / 32][5];
    resident_body<false>(g, sweep_of(g.ctrl, at), n_sweeps, at.known != 0, res_smem, sthr, red);
}

__global__ void __launch_bounds__(kResThreads, 1) k_resident_ne(const __grid_constant__ Geom g, SweepAt at, int n_sweeps)
{
    extern __shared__ uint4 res_smem[];
    __shared__ uint32_t sthr[16];
    __shared__ int red[kResThreads / 32][5];
    resident_body<true>(g, sweep_of(g.ctrl, at), n_sweeps, at.known != 0, res_smem, sthr, red);
}

// L = 32 or 64 alone on the GPU: as resident_words, with threads of their own
// for either colour. While one colour steps, the other draws and sums its
// counters, so a half-sweep takes the longer of the two and not their sum.
// L = 64: 0.93 us a sweep with one thread for both colours, 0.81 here; 64% of
// issue on its one SM, waiting for the draws' multiply pipe.
template <bool kNE, bool kSym>
__global__ void __launch_bounds__(2 * kResThreads, 1) k_resident_pair(const __grid_constant__ Geom g, SweepAt at,
                                                                      int n_sweeps)
{
    __shared__ uint32_t pl[2 * kResThreads], sthr[16];
    __shared__ int sum[2][5];   // a sweep's counters: two sweeps in turn
    const unsigned long long sweep0 = sweep_of(g.ctrl, at);
    const uint32_t wpr = g.half >> 2, words = (uint32_t)g.L * wpr;   // a multiple of 32
    const uint32_t c = threadIdx.x >= words ? 1u : 0u, i = threadIdx.x - c * words;
    const uint32_t y = i / wpr, k = i - y * wpr;
    const uint32_t *src = reinterpret_cast<const uint32_t *>(g.s[sweep0 & 1]);
    uint32_t S = src[c * words + i], was = 0, rw[2] = {0u, 0u};
    pl[c * words + i] = S;
    if constexpr (kNE) was = g.flags[c * words + i];   // G = wpr groups a row
    if (g.ref != nullptr && c == 1u)
        for (int p = 0; p < 2; ++p) rw[p] = reinterpret_cast<const uint32_t *>(g.ref)[p * words + i];
    int unfl = 4 - __popc(was);
    if (threadIdx.x < 16) sthr[threadIdx.x] = g.thr16[threadIdx.x];
    if (threadIdx.x >= 32 && threadIdx.x < 42) (&sum[0][0])[threadIdx.x - 32] = 0;
    __syncthreads();
    // the other plane's words around this one
    const uint32_t *o = pl + (1u - c) * words;
    const bool odd = ((c + y) & 1u) != 0u;
    const uint32_t *pU = o + (y == 0u ? (uint32_t)g.L - 1u : y - 1u) * wpr + k;
    const uint32_t *pD = o + (y + 1u == (uint32_t)g.L ? 0u : y + 1u) * wpr + k;
    const uint32_t *pN = o + y * wpr + (odd ? (k + 1u == wpr ? 0u : k + 1u) : (k == 0u ? wpr - 1u : k - 1u));
    unsigned long long *slot0 = series_slot(g.ctrl, sweep0);   // consecutive sweeps are contiguous
    unsigned long long *acf0 = g.ref ? acf_slot(g.ctrl, sweep0) : nullptr;
    const uint32_t g0 = y * g.G + k;
    uint32_t p01 = 0, p23 = 0;
    int bond = 0, mag = 0, acf = 0;
    auto draw = [&](int s) {
        const unsigned long long sweep = sweep0 + (unsigned long long)s;
        PhiloxPre pp;
        philox_prepare(pp, (uint32_t)sweep, (uint32_t)(sweep >> 32), g.key0, g.key1);
        top_halves(philox_item(pp, g0, c), p01, p23);
    };
    auto step = [&](int s) {
        const uint32_t U = *pU, D = *pD, O = o[i], nb = *pN;
        const uint32_t X = odd ? __funnelshift_r(O, nb, 8) : __funnelshift_l(nb, O, 8);
        const Nbr n = nbr_sum(U, D, O, X);
        uint32_t t01[2], t23[2], tie = kNoTie;
        if constexpr (kSym) sym_thresholds(g.acc, n, S, t01[0], t23[0]);
        else gen_thresholds2(g.acc, n, n, S, S, t01, t23);
        uint32_t rej = reject4(t01[0], t23[0], p01, p23, tie);
        if (tie_hit(tie)) {
            const unsigned long long sweep = sweep0 + (unsigned long long)s;
            PhiloxPre pp;
            philox_prepare(pp, (uint32_t)sweep, (uint32_t)(sweep >> 32), g.key0, g.key1);
            rej = reject4_exact(sthr, n, S, philox_item(pp, g0, c));
        }
        uint32_t F = ~rej & 0xFEFEFEFEu;
        if constexpr (kNE) F &= ~(U | (odd ? X : O));   // §III.B: north and east must be up
        S ^= F;
        pl[c * words + i] = S;
        if constexpr (kNE) {
            const uint32_t bits = (uint32_t)dot4(F & 0x02020202u, 0x08040201u, 0) >> 1;
            unfl -= __popc(bits & ~was);
            was |= bits;
        }
        if (c == 1u) {
            bond = dot4(S, X, dot4(S, O, dot4(S, D, dot4(S, U, 0))));
            mag = dot4(S, 0x01010101u, dot4(O, 0x01010101u, 0));
            if (g.ref) acf = dot4(S, rw[1], dot4(O, rw[0], 0));
        }
    };
    // this colour's share of sweep s's counters, after its step
    auto reduce = [&](int s) {
        int *t = sum[s & 1];
        const bool first = (threadIdx.x & 31u) == 0u;
        if constexpr (kNE) {
            const int f = __reduce_add_sync(0xffffffffu, unfl);
            if (first) atomicAdd(&t[3], f);
        }
        if (c == 0u) return;
        const int b = __reduce_add_sync(0xffffffffu, bond), m = __reduce_add_sync(0xffffffffu, mag);
        const int a = g.ref ? __reduce_add_sync(0xffffffffu, acf) : 0;
        if (first) {
            atomicAdd(&t[0], b);
            atomicAdd(&t[1], m);
            if (g.ref) atomicAdd(&t[4], a);
        }
    };
    // a sweep's counters go out once both colours have summed theirs; cleared
    // two barriers before their next use
    auto post = [&](int s) {
        if (threadIdx.x != 0u || s < 0) return;
        int *t = sum[s & 1];
        unsigned long long *slot = slot0 + 4ull * (unsigned)s;
        const long long m = t[1];
        add_counter(slot + 0, t[0]);
        add_counter(slot + 1, m);
        add_counter(slot + 2, (m + (long long)g.N) / 2);
        if constexpr (kNE) add_counter(slot + 3, t[3]);
        if (g.ref) add_counter(acf0 + (unsigned)s, t[4]);
        for (int j = 0; j < 5; ++j) t[j] = 0;
    };
    if (c == 0u) {
        draw(0);
        for (int s = 0; s < n_sweeps; ++s) {
            step(s);
            __syncthreads();
            post(s - 1);
            reduce(s);
            if (s + 1 < n_sweeps) draw(s + 1);
            __syncthreads();
        }
    } else {
        for (int s = 0; s < n_sweeps; ++s) {
            if (s > 0) reduce(s - 1);
            draw(s);
            __syncthreads();
            step(s);
            __syncthreads();
        }
        reduce(n_sweeps - 1);
    }
    __syncthreads();
    post(n_sweeps - 1);
    reinterpret_cast<uint32_t *>(g.s[(sweep0 + (unsigned long long)n_sweeps) & 1])[c * words + i] = S;
    if constexpr (kNE) g.flags[c * words + i] = (uint8_t)was;
    if (at.known != 0 && threadIdx.x == 0) g.ctrl->sweep = sweep0 + (unsigned long long)n_sweeps;
}

// Batched form: CTA i sweeps lattice i (descriptor geoms[i]) by
// min(chunk, n[i] - done) sweeps and advances its counter; lattices of
// either model and width share the launch.
__global__ void __launch_bounds__(kResThreads, 1) k_batch_resident(const Geom *geoms, const long long *n,
                                                                   long long done, int chunk)
{
    extern __shared__ uint4 res_smem[];
    __shared__ uint32_t sthr[16];
    __shared__ int red[kResThreads / 32][5];
    __shared__ Geom sg;
    const long long left = n[blockIdx.x] - done;
    if (left <= 0) return;   // uniform over the CTA
    const int m = (int)(left < (long long)chunk ? left : (long long)chunk);
    if (threadIdx.x < sizeof(Geom) / 4)
        reinterpret_cast<uint32_t *>(&sg)[threadIdx.x] = reinterpret_cast<const uint32_t *>(&geoms[blockIdx.x])[threadIdx.x];
    __syncthreads();
    const bool narrow = (uint64_t)sg.L * (sg.half >> 2) <= (uint64_t)kResThreads;
    if (sg.model == LAT_NE) {
        if (narrow) resident_words<true, false>(sg, sg.ctrl->sweep, m, true, res_smem, sthr, red);
        else resident_body<true>(sg, sg.ctrl->sweep, m, true, res_smem, sthr, red);
    } else {
        if (narrow && sg.acc_sym) resident_words<false, true>(sg, sg.ctrl->sweep, m, true, res_smem, sthr, red);
        else if (narrow) resident_words<false, false>(sg, sg.ctrl->sweep, m, true, res_smem, sthr, red);
        else resident_body<false>(sg, sg.ctrl->sweep, m, true, res_smem, sthr, red);
    }
}

size_t resident_bytes(const Geom &g)
{
    return (size_t)g.N + (g.model == LAT_NE ? (size_t)2 * g.rows * g.G : 0);
}

}  // namespace

bool wide_supported(const Geom &g)
{
    if (!(g.dims == 2 && g.two_S == 1 && g.bits[0] == nullptr && (g.L % 32) == 0)) return false;
    if (g.model == LAT_POTTS) return false;
    for (int k = 0; k < 16; ++k) {
        if ((k & 7) > 4) continue;
        if (!((g.always16 >> k) & 1u) && g.thr16[k] == 0u) return false;
    }
    return true;
}

bool any_supported(const Geom &g)
{
    if (!(g.dims == 2 && g.two_S == 1 && g.bits[0] == nullptr && g.cpl == nullptr && (g.L % 2) == 0)) return false;
    if (g.model == LAT_POTTS) return false;
    for (int k = 0; k < 16; ++k) {
        if ((k & 7) > 4) continue;
        if (!((g.always16 >> k) & 1u) && g.thr16[k] == 0u) return false;
    }
    return true;
}

int any_items(const Geom &g, int passes)
{
    const AnyItemShape sh = any_item_shape(g.half, (uint32_t)passes);
    return (int)((((uint32_t)g.L + sh.br - 1u) / sh.br) * sh.nseg);
}

int batch_any_grid(bool ne)
{
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (ne) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_batch_any<true, false, 1>, kThreads, 0);
    else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_batch_any<false, false, 1>, kThreads, 0);
    if (per < 1) per = 1;
    return sms * per;
}

cudaError_t launch_batch_any(const Geom *geoms, const uint2 *items, int n_items, unsigned *next_item, int colour,
                             bool ne, bool aligned, int passes, int grid, cudaStream_t st)
{
    using K = void (*)(const Geom *, const uint2 *, int, unsigned *, uint32_t);
    // [Ising, North-East at T][aligned][colour]
    static const K kern[2][2][2] = {
        {{k_batch_any<false, false, 0>, k_batch_any<false, false, 1>},
         {k_batch_any<false, true, 0>, k_batch_any<false, true, 1>}},
        {{k_batch_any<true, false, 0>, k_batch_any<true, false, 1>},
         {k_batch_any<true, true, 0>, k_batch_any<true, true, 1>}}};
    return launch_pdl(kern[ne ? 1 : 0][aligned ? 1 : 0][colour ? 1 : 0], (unsigned)grid, kThreads, st, geoms, items,
                      n_items, next_item, (uint32_t)passes);
}

bool sweep_at_known(const Geom &g) { return g.model == LAT_ISING || ne_walk_supported(g); }

cudaError_t launch_sweep_wide(const Geom &g, bool fields, SweepAt at, cudaStream_t st)
{
    if (ne_walk_supported(g)) return launch_sweep_ne(g, at, st);
    const Geom k = tiled_geom(g);  // compact table in t' = thr - 1 form
    const int ref = k.ref != nullptr ? 1 : 0, al = g.L % 32 == 0 ? 1 : 0;
    const uint64_t blocks = ((uint64_t)g.L * ((g.half + 15u) >> 4) + kThreads - 1) / kThreads;
    if (g.model == LAT_NE) {   // North-East at temperature T
        using K = void (*)(Geom, int);
        static const K ne[2][2][2] = {
            {{k_any_pipe_ne<0, false>, k_any_pipe_ne<1, false>}, {k_any_pipe_ne<0, true>, k_any_pipe_ne<1, true>}},
            {{k_wide_pipe_ne<0, false>, k_wide_pipe_ne<1, false>}, {k_wide_pipe_ne<0, true>, k_wide_pipe_ne<1, true>}}};
        static const unsigned w[2] = {one_wave(reinterpret_cast<const void *>(ne[0][1][1])),
                                      one_wave(reinterpret_cast<const void *>(ne[1][1][1]))};
        const unsigned grid = (unsigned)std::min<uint64_t>(blocks, w[al]);
        cudaError_t e = launch_pdl(ne[al][ref][0], grid, kThreads, st, k, at.off);
        return e == cudaSuccess ? launch_pdl(ne[al][ref][1], grid, kThreads, st, k, at.off) : e;
    }
    using K = void (*)(Geom, SweepAt);
#define LAT_WALK(dis, acc, al, one)                                                          \
    {{k_ising_walk<0, false, dis, acc, al, one>, k_ising_walk<1, false, dis, acc, al, one>}, \
     {k_ising_walk<0, true, dis, acc, al, one>, k_ising_walk<1, true, dis, acc, al, one>}}
    // [uniform at any even L, then L % 32 == 0: uniform, bonds, fields][reference][colour]
    static const K one[4][2][2] = {LAT_WALK(kUniform, kLookUp, false, true), LAT_WALK(kUniform, kLookUp, true, true),
                                   LAT_WALK(kBonds, kLookUp, true, true), LAT_WALK(kFields, kLookUp, true, true)};
    static const K walk[4][2][2] = {LAT_WALK(kUniform, kLookUp, false, false), LAT_WALK(kUniform, kLookUp, true, false),
                                    LAT_WALK(kBonds, kLookUp, true, false), LAT_WALK(kFields, kLookUp, true, false)};
    static const K top[3][2][2] = {LAT_WALK(kUniform, kTopSym, false, false), LAT_WALK(kUniform, kTopSym, true, false),
                                   LAT_WALK(kBonds, kTopSym, true, false)};
    static const K few[2][2][2] = {LAT_WALK(kUniform, kTopGen, false, true), LAT_WALK(kUniform, kTopSym, false, true)};
#undef LAT_WALK
    static const unsigned wave = one_wave(reinterpret_cast<const void *>(walk[1][0][1]));   // all: kWalkMinB per SM
    const int m = g.cpl != nullptr ? (fields ? 3 : 2) : al, sym = k.acc_sym ? 1 : 0;
    // One chunk a thread up to two waves of them: up to there the row walk's
    // start-up costs more than its register reuse saves.  The 16-bit
    // acceptance of symmetric tables from 10 rows a thread on: its rows to be
    // done again are a chain of memory trips at the end of every thread's walk
    // (launches of a graph, 16-bit and look-ups: L = 3000, 3 rows, 20.0 and
    // 17.6 us a sweep; 4096, 7 rows, 20.5 and 19.9; 6000, 15 rows, 55.0 and
    // 56.2; 8192, 27 rows, 67.4 and 70.6).  And where rows of any alignment
    // give no more than a CTA an SM, whose undecided chunks are settled from
    // registers: L = 66 4.78 and 4.97, 1000 5.79 and 5.96 (2000: 10.8 and 10.2).
    const bool many = blocks > 2u * wave;
    const K *kern = many ? (sym && blocks >= 10u * wave ? top[m][ref] : walk[m][ref])
                         : (m == 0 && blocks <= wave / kWalkMinB ? few[sym][ref] : one[m][ref]);
    const unsigned grid = many ? wave : (unsigned)blocks;
    cudaError_t e = launch_pdl(kern[0], grid, kThreads, st, k, at);
    return e == cudaSuccess ? launch_pdl(kern[1], grid, kThreads, st, k, at) : e;
}

bool resident_supported(const Geom &g)
{
    return wide_supported(g) && g.cpl == nullptr && resident_bytes(g) <= kResMaxBytes;
}

cudaError_t launch_sweep_resident(const Geom &g, SweepAt at, int n_sweeps, cudaStream_t st)
{
    const Geom k = tiled_geom(g);
    const size_t smem = resident_bytes(g);
    const bool narrow = (uint64_t)g.L * (g.half >> 2) <= (uint64_t)kResThreads;
    using K = void (*)(Geom, SweepAt, int);
    const bool ne = g.model == LAT_NE;
    if (narrow) {   // L = 32, 64
        static const K pair[3] = {k_resident_pair<false, false>, k_resident_pair<false, true>, k_resident_pair<true, false>};
        pair[ne ? 2 : (k.acc_sym ? 1 : 0)]<<<1, (unsigned)(g.N / 4), 0, st>>>(k, at, n_sweeps);
        return cudaGetLastError();
    }
    static const K fn[2] = {k_resident_ising, k_resident_ne};
    static const cudaError_t attr = [] {
        cudaError_t e = cudaSuccess;
        for (K f : fn)
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kResMaxBytes);
        return e;
    }();
    if (attr != cudaSuccess) return attr;
    fn[ne ? 1 : 0]<<<1, kResThreads, smem, st>>>(k, at, n_sweeps);
    return cudaGetLastError();
}

}  // namespace lat

namespace lat {

cudaError_t launch_batch_resident(const Geom *geoms, const long long *n, int n_lat, long long done, int chunk,
                                  size_t smem, cudaStream_t st)
{
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k_batch_resident, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)kResMaxBytes);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    k_batch_resident<<<n_lat, kResThreads, smem, st>>>(geoms, n, done, chunk);
    return cudaGetLastError();
}

size_t resident_smem_bytes(const Geom &g) { return resident_bytes(g); }

}  // namespace lat
