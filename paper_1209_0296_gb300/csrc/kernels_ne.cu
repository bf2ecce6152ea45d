// kernels_ne.cu -- checkerboard sweeps of the North-East model in c-mode
// (§III.B: rates that depend on the move alone), two launches per sweep, any
// even L, int8 spins in the checkerboard-planar layout; solo and batched.
//
// A site moves only if its north and east neighbours are up; then one of the
// two moves is certain (c < 1/2: up -> down) and the other is accepted with
// one fixed probability.  So most sites need no random number: at c = 0.3
// one group of four in four needs its Philox call, at c = 0.05 one in a
// hundred.  A thread walks a column of 16-site chunks down consecutive
// rows.  The main pass does everything that needs no draw with a few logic
// operations per four sites: constraint, certain moves, store, counters (as
// byte dot products on the multiply pipe).  Groups with an undecided site
// are queued, and whenever a warp has 32 of them each lane makes one Philox
// call and applies the accepted moves as byte stores with counter
// corrections.  The queue is the warp's own, so calls fill whole warps
// whatever c is, and the main pass never waits for a draw.
//
// "Unflipped" is carried from the previous sweep's counter and reduced by
// the sites that change for the first time, so persistence bytes are read
// and written only where a site flips.
#include <algorithm>

#include "ne_walk.cuh"

namespace lat {

namespace {

constexpr int kNeMinB = 3;            // CTAs per SM, solo
constexpr int kNeBatchMinB = 2;       // batched (the lattice descriptor costs registers)
constexpr int kWarps = kThreads / 32;

// The planes of one colour's pass.
template <int kColour>
struct NeRows {
    const int8_t *pS, *pO;   // this colour's old sites, the other colour's current sites
    int8_t *dS;              // this colour's plane in the new buffer
    uint8_t *fl;             // this colour's persistence bytes
    const int8_t *r1, *r0;   // reference planes 1 and 0
    uint32_t half, L, G;
};

template <int kColour>
LAT_D NeRows<kColour> ne_rows(const SweepView &v, unsigned long long sweep)
{
    const int8_t *old = (sweep & 1) ? v.s1 : v.s0;
    int8_t *nw = (sweep & 1) ? v.s0 : v.s1;
    const size_t plane = (size_t)v.plane;
    NeRows<kColour> p;
    p.pS = old + kColour * plane;
    p.pO = (kColour == 0 ? old : nw) + (1 - kColour) * plane;
    p.dS = nw + kColour * plane;
    p.fl = v.flags + (size_t)kColour * v.rows * v.G;
    p.r1 = v.ref ? v.ref + plane : nullptr;
    p.r0 = v.ref;
    p.half = v.half;
    p.L = (uint32_t)v.L;
    p.G = v.G;
    return p;
}

// Rows [y, y1) of chunk column k by one thread (act: the thread has any).
// The warp's 32 threads call together.
template <int kColour, bool kRef, bool kAligned>
LAT_D void ne_walk(const NeRows<kColour> &p, const PhiloxPre &pp, const NeRate rate, uint32_t k, uint32_t y,
                   uint32_t y1, bool act, NeJob *queue, Counts &cnt)
{
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    const ChunkCol<kAligned> cc = chunk_col<kAligned>(k, p.half);
    const NePlanes where{reinterpret_cast<uint8_t *>(p.dS), p.fl, p.r1};
    int sites = 0;
    unsigned queued = 0;   // warp-uniform
    uint32_t R[4][4];      // rows of the other plane, row y - 1 + i in R[(s + i) & 3] at step s
    Row16<kAligned> nS, nD;
    uint32_t nb_next = 0;
    auto other_row = [&](uint32_t r) { return p.pO + (size_t)r * p.half + cc.j0; };
    auto fetch = [&](uint32_t r) {   // row r's own sites and neighbour byte, row r + 1 of the other plane
        row_load<kAligned>(p.pS + (size_t)r * p.half + cc.j0, cc.nv, nS);
        row_load<kAligned>(other_row(r + 1u == p.L ? 0u : r + 1u), cc.nv, nD);
        // x = 2j in even rows of colour 0: west is j - 1, east is j; else west is j, east is j + 1
        nb_next = (uint32_t)(uint8_t)p.pO[(size_t)r * p.half + (((kColour + r) & 1u) ? cc.jn : cc.jp)];
    };
    if (act) {
        Row16<kAligned> a, b;
        const int8_t *qa = other_row(y == 0u ? p.L - 1u : y - 1u), *qb = other_row(y);
        row_load<kAligned>(qa, cc.nv, a);
        row_load<kAligned>(qb, cc.nv, b);
        fetch(y);
        row_words<kAligned>(qa, a, R[0]);
        row_words<kAligned>(qb, b, R[1]);
    }
    auto drain = [&](bool all) {
        __syncwarp();
        while (queued >= 32u) {
            queued -= 32u;
            const NeJob j = queue[queued + lane];
            ne_job<kRef>(where, pp, rate, j, (uint32_t)kColour, cnt);
        }
        if (all && (unsigned)lane < queued) {
            const NeJob j = queue[lane];
            ne_job<kRef>(where, pp, rate, j, (uint32_t)kColour, cnt);
        }
        __syncwarp();
    };
    for (bool more = __any_sync(0xffffffffu, act); more;) {
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            uint32_t(&U)[4] = R[s], (&O)[4] = R[(s + 1) & 3], (&D)[4] = R[(s + 2) & 3];
            uint32_t S[4], cand[4], ws[4];
            const uint32_t nb = nb_next;
            const uint32_t at0 = y * p.half + cc.j0;
            if (act) {
                row_words<kAligned>(p.pS + (size_t)at0, nS, S);
                row_words<kAligned>(other_row(y + 1u == p.L ? 0u : y + 1u), nD, D);
            }
            const bool act1 = act && y + 1u < y1;
            if (act1) fetch(y + 1u);
            bool need[4] = {false, false, false, false};
            if (act) {
                const bool odd = ((kColour + y) & 1u) != 0u;
                uint32_t X[4], Sn[4], sure[4];
                if (odd) {   // east is the shifted row
                    shifted_row<kAligned>(cc, true, nb, O, X);
                    ne_moves<kAligned, true>(U, D, X, O, S, cc.vm, rate, cand, sure, ws, Sn, need);
                } else {
                    shifted_row<kAligned>(cc, false, nb, O, X);
                    ne_moves<kAligned, true>(U, D, O, X, S, cc.vm, rate, cand, sure, ws, Sn, need);
                }
                store16_any<kAligned>(p.dS + (size_t)at0, cc.nv, Sn);
                if constexpr (kColour == 1) {
                    ne_count(Sn, U, D, O, X, cc.vm, cnt);
                    sites += 2 * (int)cc.nv;
                    if constexpr (kRef) {
                        uint32_t R1[4], R0[4];
                        load16_any<kAligned>(p.r1 + (size_t)at0, cc.nv, R1);
                        load16_any<kAligned>(p.r0 + (size_t)at0, cc.nv, R0);
#pragma unroll
                        for (int w = 0; w < 4; ++w)
                            cnt.acf = dot4(Sn[w] & cc.vm[w], R1[w], dot4(O[w] & cc.vm[w], R0[w], cnt.acf));
                    }
                }
                if (((sure[0] | sure[1] | sure[2] | sure[3]) & kB1) != 0u) {
                    const uint32_t chg = ne_changed(sure);
                    uint8_t *fp = p.fl + (size_t)y * p.G + 4u * k;
                    const uint32_t was = ne_flags<kAligned>(fp, cc.nv);
                    cnt.unfl -= __popc(chg & ~was);
                    ne_set_flags<kAligned>(fp, was, was | chg);
                }
            }
            const uint32_t g0 = y * p.G + 4u * k;
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                const unsigned bal = __ballot_sync(0xffffffffu, need[w]);
                if (need[w])
                    queue[queued + __popc(bal & below)] = NeJob{g0 + (uint32_t)w, at0 + 4u * (uint32_t)w, cand[w], ws[w]};
                queued += __popc(bal);
            }
            if (queued >= 32u) drain(false);
            act = act1;
            ++y;
            more = __any_sync(0xffffffffu, act);
            if (!more) break;
        }
    }
    drain(true);
    if constexpr (kColour == 1) cnt.up += (cnt.mag + sites) / 2;
}

// The chunk of row y and column k alone (lattices with no more chunks than
// threads: nothing to keep in registers from row to row).  Such a pass is as
// long as its chain of memory trips, so everything it reads is asked for at
// once, and the thread draws for its own groups, all four, while that is on
// its way.  (L = 1024, c = 0.3, launches of a graph: 5.0 us a sweep; with
// persistence bits read once a move is known and the draws queued, 7.4.)
template <int kColour, bool kRef, bool kAligned>
LAT_D void ne_one(const NeRows<kColour> &p, const PhiloxPre &pp, const NeRate rate, uint32_t k, uint32_t y, Counts &cnt)
{
    const ChunkCol<kAligned> cc = chunk_col<kAligned>(k, p.half);
    const uint32_t at0 = y * p.half + cc.j0, g0 = y * p.G + 4u * k;
    auto other = [&](uint32_t r) { return p.pO + (size_t)r * p.half + cc.j0; };
    const bool odd = ((kColour + y) & 1u) != 0u;
    uint32_t U[4], O[4], D[4], S[4], X[4], E[4], W[4], Sn[4], cand[4], moved[4], ws[4], rej[4];
    bool need[4];
    uint8_t *fp = p.fl + g0;
    load16_any<kAligned>(other(y == 0u ? p.L - 1u : y - 1u), cc.nv, U);
    load16_any<kAligned>(other(y), cc.nv, O);
    load16_any<kAligned>(other(y + 1u == p.L ? 0u : y + 1u), cc.nv, D);
    load16_any<kAligned>(p.pS + (size_t)at0, cc.nv, S);
    const uint32_t nb = (uint32_t)(uint8_t)p.pO[(size_t)y * p.half + (odd ? cc.jn : cc.jp)];
    [[maybe_unused]] uint32_t R1[4], R0[4];
    if constexpr (kColour == 1 && kRef) {
        load16_any<kAligned>(p.r1 + (size_t)at0, cc.nv, R1);
        load16_any<kAligned>(p.r0 + (size_t)at0, cc.nv, R0);
    }
    const uint32_t was = ne_flags<kAligned>(fp, cc.nv);
#pragma unroll
    for (int w = 0; w < 4; ++w) rej[w] = ne_rejected(philox_item(pp, g0 + (uint32_t)w, (uint32_t)kColour), rate.K);
    shifted_row<kAligned>(cc, odd, nb, O, X);
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        E[w] = odd ? X[w] : O[w];
        W[w] = odd ? O[w] : X[w];
    }
    ne_moves<kAligned>(U, D, E, W, S, cc.vm, rate, cand, moved, ws, Sn, need);
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        moved[w] |= cand[w] & ~rej[w];
        Sn[w] = S[w] ^ (moved[w] & 0xFEFEFEFEu);
    }
    store16_any<kAligned>(p.dS + (size_t)at0, cc.nv, Sn);
    const uint32_t chg = ne_changed(moved), now = was | chg;
    cnt.unfl -= __popc(chg & ~was);
    ne_set_flags<kAligned>(fp, was, now);
    if constexpr (kColour == 1) {
        ne_count(Sn, U, D, O, X, cc.vm, cnt);
        cnt.up += (cnt.mag + 2 * (int)cc.nv) / 2;
        if constexpr (kRef) {
#pragma unroll
            for (int w = 0; w < 4; ++w)
                cnt.acf = dot4(Sn[w] & cc.vm[w], R1[w], dot4(O[w] & cc.vm[w], R0[w], cnt.acf));
        }
    }
}

// kOne: a thread per chunk (the launch has one for each); else a thread per
// (chunk column, band of consecutive rows), the launch having at least cpr.
template <int kColour, bool kRef, bool kAligned, bool kOne>
__global__ void __launch_bounds__(kThreads, kNeMinB) k_ne_walk(Geom g, SweepAt at)
{
    __shared__ int red[kWarps][5];
    __shared__ NeJob queue[kOne ? 1 : kWarps][kOne ? 1 : kNeQueue];
    dep_wait();
    const unsigned long long sweep = sweep_of(g.ctrl, at);
    const SweepView v = sweep_view(g);
    Counts cnt;
    const uint32_t L = (uint32_t)g.L, cpr = (g.half + 15u) >> 4;
    const uint32_t nb = kOne ? L : min((gridDim.x * blockDim.x) / cpr, L);
    const uint32_t gt = blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t band = gt / cpr;
    PhiloxPre pp;
    philox_prepare(pp, (uint32_t)sweep, (uint32_t)(sweep >> 32), g.key0, g.key1);
    const bool act = band < nb;
    const uint32_t k = act ? gt - band * cpr : 0u;
    const NeRows<kColour> p = ne_rows<kColour>(v, sweep);
    if constexpr (kOne) {
        if (act) ne_one<kColour, kRef, kAligned>(p, pp, ne_rate(g.thr16), k, band, cnt);
    } else {
        uint32_t y = 0, y1 = 0;
        if (act) walk_rows(band, nb, L, y, y1);
        ne_walk<kColour, kRef, kAligned>(p, pp, ne_rate(g.thr16), k, y, y1, act, queue[threadIdx.x >> 5], cnt);
    }
    dep_launch();   // main work done: the next kernel may be scheduled
    unsigned long long *slot = series_slot(g.ctrl, sweep);
    if constexpr (kColour == 1) {
        if (gt == 0u) {
            add_counter(slot + 3, ne_unflipped_before(g.ctrl, sweep));
            sweep_done(g.ctrl, at);
        }
        flush(v, sweep, cnt, true, red);
    } else {
        flush_one(slot + 3, cnt.unfl, red);
    }
}

// Batched form: items (lattice, band of rows x segment of 256 chunk columns)
// from an atomic counter; every lattice is a c-mode North-East one.
template <int kColour, bool kAligned>
__global__ void __launch_bounds__(kThreads, kNeBatchMinB) k_batch_ne(const Geom *geoms, const uint2 *items, int n_items,
                                                               unsigned *next_item, uint32_t passes)
{
    __shared__ int red[kWarps][5];
    __shared__ NeJob queue[kWarps][kNeQueue];
    __shared__ Geom sg;
    __shared__ int cur;
    int loaded = -1;
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
            loaded = (int)w.x;
            __syncthreads();
        }
        const SweepView v = sweep_view(sg);
        const unsigned long long sweep = v.ctrl->sweep;
        Counts cnt;
        PhiloxPre pp;
        philox_prepare(pp, (uint32_t)sweep, (uint32_t)(sweep >> 32), v.key0, v.key1);
        const AnyItemShape sh = any_item_shape(v.half, passes);
        const uint32_t band = w.y / sh.nseg, seg = w.y - band * sh.nseg;
        const bool narrow = sh.cpr <= (uint32_t)kThreads;
        const uint32_t k = narrow ? threadIdx.x % sh.cpr : seg * kThreads + threadIdx.x;
        const uint32_t r0 = narrow ? threadIdx.x / sh.cpr : 0u;
        const uint32_t y = band * sh.br + r0 * (sh.br / sh.rsb);
        const uint32_t y1 = min((uint32_t)v.L, y + sh.br / sh.rsb);
        const bool act = k < sh.cpr && r0 < sh.rsb && y < y1;
        const NeRows<kColour> p = ne_rows<kColour>(v, sweep);
        const NeRate rate = ne_rate(sg.thr16);
        if (v.ref)
            ne_walk<kColour, true, kAligned>(p, pp, rate, act ? k : 0u, y, y1, act, queue[threadIdx.x >> 5], cnt);
        else
            ne_walk<kColour, false, kAligned>(p, pp, rate, act ? k : 0u, y, y1, act, queue[threadIdx.x >> 5], cnt);
        unsigned long long *slot = series_slot(v.ctrl, sweep);
        if constexpr (kColour == 1) {
            if (w.y == 0u && threadIdx.x == 0u) add_counter(slot + 3, ne_unflipped_before(v.ctrl, sweep));
            flush(v, sweep, cnt, true, red);   // ends with __syncthreads()
        } else {
            flush_one(slot + 3, cnt.unfl, red);
        }
        __syncthreads();
    }
    dep_launch();   // no items left: the next kernel may be scheduled
}

}  // namespace

bool ne_walk_supported(const Geom &g)
{
    return g.model == LAT_NE && g.cmode != 0 && g.cpl == nullptr && any_supported(g);
}

cudaError_t launch_sweep_ne(const Geom &g, SweepAt at, cudaStream_t st)
{
    using K = void (*)(Geom, SweepAt);
    // [one chunk a thread][aligned][reference][colour]
#define LAT_NE_K(ref, al, one) {k_ne_walk<0, ref, al, one>, k_ne_walk<1, ref, al, one>}
    static const K kern[2][2][2][2] = {
        {{LAT_NE_K(false, false, false), LAT_NE_K(true, false, false)}, {LAT_NE_K(false, true, false), LAT_NE_K(true, true, false)}},
        {{LAT_NE_K(false, false, true), LAT_NE_K(true, false, true)}, {LAT_NE_K(false, true, true), LAT_NE_K(true, true, true)}}};
#undef LAT_NE_K
    static const unsigned wave[2] = {one_wave(reinterpret_cast<const void *>(kern[0][0][1][1])),
                                     one_wave(reinterpret_cast<const void *>(kern[0][1][1][1]))};
    const Geom k = tiled_geom(g);
    const int al = g.L % 32 == 0 ? 1 : 0, ref = g.ref != nullptr ? 1 : 0;
    const uint64_t blocks = ((uint64_t)g.L * ((g.half + 15u) >> 4) + kThreads - 1) / kThreads;
    // one chunk a thread up to two waves of them: up to there the row walk's
    // start-up costs more than its register reuse saves
    const int one = blocks <= 2u * wave[al] ? 1 : 0;
    const unsigned grid = one ? (unsigned)blocks : wave[al];
    cudaError_t e = launch_pdl(kern[one][al][ref][0], grid, kThreads, st, k, at);
    return e == cudaSuccess ? launch_pdl(kern[one][al][ref][1], grid, kThreads, st, k, at) : e;
}

int batch_ne_grid() { return (int)one_wave(reinterpret_cast<const void *>(k_batch_ne<1, false>)); }

cudaError_t launch_batch_ne(const Geom *geoms, const uint2 *items, int n_items, unsigned *next_item, int colour,
                            bool aligned, int passes, int grid, cudaStream_t st)
{
    using K = void (*)(const Geom *, const uint2 *, int, unsigned *, uint32_t);
    static const K kern[2][2] = {{k_batch_ne<0, false>, k_batch_ne<1, false>}, {k_batch_ne<0, true>, k_batch_ne<1, true>}};
    return launch_pdl(kern[aligned ? 1 : 0][colour ? 1 : 0], (unsigned)grid, kThreads, st, geoms, items, n_items,
                      next_item, (uint32_t)passes);
}

}  // namespace lat
