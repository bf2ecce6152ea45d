// band.cuh -- many sweeps in one launch for 2D spin-1/2 lattices that
// fit the chip's shared memory: every CTA keeps a band of rows resident and
// neighbouring bands exchange their boundary rows.
//
// With two launches per sweep a lattice of a million sites spends most of
// its time between kernels: a launch costs about 2.5 us of start-up, memory
// latency and drain, its work 0.6 us.  Here one cooperative launch runs all
// sweeps of a call.  CTA b holds rows [y0, y1) of both colour planes in
// shared memory, rows at 16-byte alignment whatever L is, and updates a
// colour in place.  The new values of its first and last row go to the two
// neighbouring bands as packets of 4 data bytes and a 4-byte half-sweep
// number in one 64-bit word; the reader polls the packets themselves, so a
// row costs one trip through L2 and no fence or flag.  Interior rows come
// first, so the neighbours' packets are usually there before they are asked
// for, and the next half-sweep's first draws are made before that.
// A packet is overwritten two half-sweeps later, after the reader's own
// packet of the half-sweep in between has arrived.
//
// A wait is bounded: when it gives up the launch ends normally and the host
// sees the error word (LAT_ETIMEOUT).  It also sets the launch's abort word,
// which ends the launch's other waits early; the host clears it with the packets
// before the next launch once it has seen the error.  (A word that holds the
// mark of the launch that gave up needs no clearing, but costs 1 to 2 % in the
// waits' code.)
#pragma once

#include <memory>
#include <type_traits>
#include <vector>

#include "ising_walk.cuh"
#include "ne_walk.cuh"

#if defined(__CUDACC__)
namespace lat {
namespace {

constexpr int kBandThreads = 512;
constexpr int kBandWarps = kBandThreads / 32;
constexpr int kBandNeThreads = 1024;        // North-East on bits, alone on the GPU, bands of more than 1024 words
constexpr int kBandMaxCtas = 160;           // a batched launch's parts are kernel parameters
constexpr uint32_t kAbortBytes = 128;       // the abort word's line, before the packets
constexpr size_t kBandMaxSmem = 224 * 1024;

// What a CTA runs: band `band` of `bands` of one lattice.  The key and the
// acceptance table are here (and not read from the lattice's descriptor) so
// that they are kernel parameters, which the sweep loop reads as such.
// (The order is measured: with four bytes more before the key and the table the
// batched kernel, which reads them at a run-time index, took 721 us for the 707
// of a served mix of 16 lattices; with the table first the bit-packed kernel
// took 1 % more.)
struct BandPart {
    uint32_t band, bands;        // batched (solo: the CTA and the grid)
    uint32_t lat, kind, ref;     // batched: descriptor index, BandKind, reference set
    uint32_t epoch;              // packets are marked epoch + 1 .. epoch + 2 n
    unsigned long long sweep0;   // sweeps done before the launch
    int *err;                    // host-visible error word of the lattice
    uint32_t mail;               // batched: packet rows start at this pair
    int n;                       // sweeps to run
    uint32_t key0, key1;
    uint32_t acc[8];
    uint32_t limit;              // polls after which a wait gives up
    int *err_all;                // batched: host-visible error word of the batch
};

struct BandShared {
    uint32_t sthr[16];
    int sum[2][5];   // a sweep's bond, mag, up, unflipped, overlap: two sweeps in turn
    int fld;
    int bad;         // a wait gave up
    int unfl;        // unflipped sites of the band
};

// The launch's view of a band.
struct Band {
    uint32_t y0, nr, half, pitch, cpr, L, G;
    bool al;                     // rows are 16-byte aligned in global memory
    size_t plane;
    const int8_t *src;           // spins before the launch
    uint32_t up, dn;             // rows above and below the band
    unsigned *abort;             // set when a wait of the launch gave up
    // packet rows of colour 0 (colour 1: + cpr packet pairs): this band's
    // first and last row, the last row of the band above, the first below
    ulonglong2 *first, *last;
    const ulonglong2 *above, *below;
};

LAT_D Band band_of(const Geom &g, const BandPart &p, uint32_t band, uint32_t bands, uint8_t *mail)
{
    Band b;
    uint32_t y1;
    b.L = (uint32_t)g.L;
    band_rows(band, bands, b.L, b.y0, y1);
    b.nr = y1 - b.y0;
    b.half = g.half;
    b.cpr = (g.half + 15u) >> 4;
    b.pitch = 16u * b.cpr;
    b.G = g.G;
    b.al = (g.half & 15u) == 0u;
    b.plane = (size_t)g.plane;
    b.src = (p.sweep0 & 1) ? g.s[1] : g.s[0];
    b.up = b.y0 == 0u ? b.L - 1u : b.y0 - 1u;
    b.dn = y1 == b.L ? 0u : y1;
    b.abort = reinterpret_cast<unsigned *>(mail);
    ulonglong2 *m = reinterpret_cast<ulonglong2 *>(mail + kAbortBytes) + p.mail;
    const size_t row = 4u * b.cpr;   // both colours, two packet pairs a chunk
    const uint32_t above = band == 0u ? bands - 1u : band - 1u, below = band + 1u == bands ? 0u : band + 1u;
    b.first = m + (size_t)band * 2u * row;
    b.last = b.first + row;
    b.above = m + (size_t)above * 2u * row + row;
    b.below = m + (size_t)below * 2u * row;
    return b;
}

LAT_D ulonglong2 ld_pair(const ulonglong2 *q)
{
    ulonglong2 v;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(q) : "memory");
    return v;
}

// Send 16 bytes as packets marked `tag`.
LAT_D void mail_put(ulonglong2 *q, uint32_t tag, const uint32_t (&v)[4])
{
    const unsigned long long t = (unsigned long long)tag << 32;
#pragma unroll
    for (int i = 0; i < 2; ++i)
        asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(q + i), "l"(t | v[2 * i]), "l"(t | v[2 * i + 1])
                     : "memory");
}

// After poll i: whether the wait gives up, at its limit or because another
// wait of the launch did.
LAT_D bool mail_over(unsigned i, const BandPart &p, unsigned *abort)
{
    if ((i & 1023u) != 1023u) return false;
    if (i < p.limit && *reinterpret_cast<volatile unsigned *>(abort) == 0u) return false;
    *reinterpret_cast<volatile unsigned *>(abort) = 1u;
    return true;
}

// Wait for the 16 bytes marked `tag`; false when the wait gave up.
LAT_D bool mail_take(const ulonglong2 *q, uint32_t tag, const BandPart &p, unsigned *abort, uint32_t (&v)[4])
{
    for (unsigned i = 0;; ++i) {
        const ulonglong2 a = ld_pair(q), b = ld_pair(q + 1);
        v[0] = (uint32_t)a.x;
        v[1] = (uint32_t)a.y;
        v[2] = (uint32_t)b.x;
        v[3] = (uint32_t)b.y;
        if ((uint32_t)(a.x >> 32) == tag && (uint32_t)(a.y >> 32) == tag && (uint32_t)(b.x >> 32) == tag &&
            (uint32_t)(b.y >> 32) == tag)
            return true;
        if (mail_over(i, p, abort)) return false;
    }
}

// The same for one word.
LAT_D void mail_put_word(unsigned long long *q, uint32_t tag, uint32_t v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(q), "l"((unsigned long long)tag << 32 | v) : "memory");
}

LAT_D bool mail_take_word(const unsigned long long *q, uint32_t tag, const BandPart &p, unsigned *abort, uint32_t &v)
{
    for (unsigned i = 0;; ++i) {
        unsigned long long a;
        asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(a) : "l"(q) : "memory");
        v = (uint32_t)a;
        if ((uint32_t)(a >> 32) == tag) return true;
        if (mail_over(i, p, abort)) return false;
    }
}

// nr rows of half bytes, global (row pitch half) -> shared (row pitch
// pitch, a multiple of 4), whole words at any alignment.
LAT_D void rows_in(const int8_t *from, uint32_t half, uint32_t nr, uint8_t *to, uint32_t pitch)
{
    if ((half & 15u) == 0u && pitch == half) {
        const uint4 *q = reinterpret_cast<const uint4 *>(from);
        for (uint32_t i = threadIdx.x; i < nr * (half >> 4); i += blockDim.x) reinterpret_cast<uint4 *>(to)[i] = q[i];
        return;
    }
    const uint32_t wpr = (half + 3u) >> 2;
    for (uint32_t i = threadIdx.x; i < nr * wpr; i += blockDim.x) {
        const uint32_t r = i / wpr, w = i - r * wpr;
        const uintptr_t a = reinterpret_cast<uintptr_t>(from + (size_t)r * half + 4u * w);
        const uint32_t sh = (uint32_t)(a & 3u), nv = min(4u, half - 4u * w);
        const uint32_t *q = reinterpret_cast<const uint32_t *>(a - sh);
        const uint32_t hi = nv + sh > 4u ? q[1] : 0u;
        *reinterpret_cast<uint32_t *>(to + (size_t)r * pitch + 4u * w) = __funnelshift_r(q[0], hi, 8u * sh);
    }
}

// The way back: only the rows' own bytes are written.
LAT_D void rows_out(const uint8_t *from, uint32_t pitch, uint32_t nr, int8_t *to, uint32_t half)
{
    if ((half & 15u) == 0u && pitch == half) {
        uint4 *q = reinterpret_cast<uint4 *>(to);
        for (uint32_t i = threadIdx.x; i < nr * (half >> 4); i += blockDim.x)
            q[i] = reinterpret_cast<const uint4 *>(from)[i];
    } else if ((half & 3u) == 0u && (reinterpret_cast<uintptr_t>(to) & 3u) == 0u) {
        const uint32_t wpr = half >> 2;
        for (uint32_t i = threadIdx.x; i < nr * wpr; i += blockDim.x) {
            const uint32_t r = i / wpr, w = i - r * wpr;
            *reinterpret_cast<uint32_t *>(to + (size_t)r * half + 4u * w) =
                *reinterpret_cast<const uint32_t *>(from + (size_t)r * pitch + 4u * w);
        }
    } else {
        for (uint32_t i = threadIdx.x; i < nr * half; i += blockDim.x) {
            const uint32_t r = i / half, x = i - r * half;
            to[i] = (int8_t)from[(size_t)r * pitch + x];
        }
    }
}

LAT_D void smem_words(const uint8_t *q, uint32_t (&v)[4]) { load_words<4>(reinterpret_cast<const int8_t *>(q), v); }

// The block's sweep counters: warp sums into sh.sum[par]; after the next
// barrier warp 1 adds them to the sweep's slots and clears them.
LAT_D void band_count(BandShared &sh, int par, const Counts &c, bool ne, bool ref)
{
    const int lane = threadIdx.x & 31;
    const int v[5] = {c.bond, c.mag, c.up, c.unfl, c.acf};
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        if ((i == 3 && !ne) || (i == 4 && !ref)) continue;
        const int s = __reduce_add_sync(0xffffffffu, v[i]);
        if (lane == 0) atomicAdd(&sh.sum[par][i], s);
    }
}

LAT_D void band_post(BandShared &sh, int par, const Geom &g, unsigned long long sweep, bool ne, bool ref)
{
    const int i = (int)threadIdx.x - 32;
    if (i < 0 || i >= 5 || (i == 3 && !ne) || (i == 4 && !ref)) return;
    long long v = sh.sum[par][i];
    if (i == 3) {
        sh.unfl += (int)v;   // newly flipped sites, negative
        v = sh.unfl;
    }
    sh.sum[par][i] = 0;
    add_counter(i < 4 ? series_slot(g.ctrl, sweep) + i : acf_slot(g.ctrl, sweep), v);
}

// Exact flips of one chunk from full 32-bit draws (rare; a call keeps it out
// of the sweep's registers).
struct Chunk16 {
    Nbr n[4];
    uint32_t S[4];
};
__device__ __noinline__ uint4 band_exact(const uint32_t *sthr, unsigned long long sweep, uint32_t key0, uint32_t key1,
                                         uint32_t g0, uint32_t colour, const Chunk16 c)
{
    PhiloxPre pp;
    philox_prepare(pp, (uint32_t)sweep, (uint32_t)(sweep >> 32), key0, key1);
    uint32_t F[4];
#pragma unroll 1
    for (int w = 0; w < 4; ++w)
        F[w] = ~reject4_exact(sthr, c.n[w], c.S[w], philox_item(pp, g0 + (uint32_t)w, colour)) & 0xFEFEFEFEu;
    return make_uint4(F[0], F[1], F[2], F[3]);
}

// The other plane's row shifted towards the side neighbour that is not at the
// same index (shifted_row), row and its wrap-around read from shared memory.
template <bool kFull>
LAT_D void band_shifted(const ChunkCol<kFull> &cc, bool odd, const uint8_t *row, const uint32_t (&O)[4], uint32_t (&X)[4])
{
    if constexpr (kFull) {   // whole words: the one after the chunk, or the one before it
        const uint32_t nb = *reinterpret_cast<const uint32_t *>(row + (odd ? cc.jn : cc.jp - 3u));
#pragma unroll
        for (int w = 0; w < 4; ++w)
            X[w] = odd ? __funnelshift_r(O[w], w == 3 ? nb : O[w + 1], 8)
                       : __funnelshift_l(w == 0 ? nb : O[w - 1], O[w], 8);
    } else {
        shifted_row<false>(cc, odd, row[odd ? cc.jn : cc.jp], O, X);
    }
}

// North and south neighbour words of local row r: from the band, or for its
// first and last row from the neighbours (before the launch's first
// half-sweep from the spins themselves).
struct BandWait {
    const int8_t *src;   // the other colour's plane before the launch
    uint32_t tag;        // of the packets to wait for (0: read src)
    uint32_t mail;       // packet index of the other colour's chunk in a packet row
};

LAT_D bool band_updown(const Band &b, const BandPart &part, const BandWait &wt, const uint8_t *other, uint32_t r,
                       uint32_t j0, uint32_t nv, uint32_t (&U)[4], uint32_t (&D)[4])
{
    bool ok = true;
    auto from = [&](const ulonglong2 *mail, uint32_t y, uint32_t (&v)[4]) {
        if (wt.tag != 0u) ok = mail_take(mail + wt.mail, wt.tag, part, b.abort, v) && ok;
        else if (b.al) load16_any<true>(wt.src + (size_t)y * b.half + j0, nv, v);
        else load16_any<false>(wt.src + (size_t)y * b.half + j0, nv, v);
    };
    const uint8_t *at = other + r * b.pitch + j0;
    if (r == 0u) from(b.above, b.up, U);
    else smem_words(at - b.pitch, U);
    if (r + 1u == b.nr) from(b.below, b.dn, D);
    else smem_words(at + b.pitch, D);
    return ok;
}

// Ising with a general table (uniform, bonds, fields), int8 on the chip.
template <bool kRef, int kDis, bool kSym, bool kFull>
LAT_D void band_ising(const Geom &g, const BandPart &part, uint32_t band, uint32_t bands, uint8_t *mail,
                     BandShared &sh, uint8_t *smem)
{
    const Band b = band_of(g, part, band, bands, mail);
    const uint32_t tid = threadIdx.x, pb = b.nr * b.pitch;
    uint8_t *dis = smem + 2u * pb;
    for (int c = 0; c < 2; ++c) {
        rows_in(b.src + c * b.plane + (size_t)b.y0 * b.half, b.half, b.nr, smem + c * pb, b.pitch);
        if constexpr (kDis != kUniform)
            rows_in(reinterpret_cast<const int8_t *>(g.cpl) + c * b.plane + (size_t)b.y0 * b.half, b.half, b.nr,
                    dis + c * pb, b.pitch);
    }
    if (tid < 16) sh.sthr[tid] = g.thr16[tid];
    if (tid < 10) (&sh.sum[0][0])[tid] = 0;
    if (tid == 10) sh.bad = 0;
    if (tid == 11) sh.fld = 0;
    __syncthreads();
    // Interior rows 1 .. nr - 2: thread (rr, k) takes chunk k of rows 1 + rr,
    // 1 + rr + rsb, ...  The two boundary rows' chunks are the last threads',
    // which have an interior row less where the rows do not divide.
    const uint32_t rsb = (uint32_t)kBandThreads / b.cpr, rr = tid / b.cpr, k = tid - rr * b.cpr;
    const uint32_t r0 = rr < rsb ? 1u + rr : b.nr, rend = b.nr - 1u;
    const uint32_t edge0 = (uint32_t)kBandThreads - 1u - tid, edges = 2u * b.cpr;   // (nr >= 2)
    const ChunkCol<kFull> cc = chunk_col<kFull>(k, b.half);
    const uint32_t at0 = r0 * b.pitch + cc.j0, at_step = rsb * b.pitch;
    const uint32_t g00 = (b.y0 + r0) * b.G + 4u * k, g_step = rsb * b.G;
    // The group a thread draws for first in a half-sweep.
    auto edge_row = [&](uint32_t e) { return e < b.cpr ? rend : 0u; };
    auto edge_col = [&](uint32_t e) { return e < b.cpr ? e : e - b.cpr; };
    auto edge_group = [&](uint32_t e) { return (b.y0 + edge_row(e)) * b.G + 4u * edge_col(e); };
    const bool has_in = r0 < rend, has_edge = edge0 < edges;
    const uint32_t g_first = has_in ? g00 : (has_edge ? edge_group(edge0) : 0u);
    const int last = 2 * part.n;
    uint32_t p01[4], p23[4];
    PhiloxPre pp;
    philox_prepare(pp, (uint32_t)part.sweep0, (uint32_t)(part.sweep0 >> 32), part.key0, part.key1);
    auto draw = [&](const PhiloxPre &q, uint32_t g0, uint32_t colour, uint32_t (&d01)[4], uint32_t (&d23)[4]) {
#pragma unroll
        for (int w = 0; w < 4; ++w) top_halves(philox_item(q, g0 + (uint32_t)w, colour), d01[w], d23[w]);
    };
    if (has_in || has_edge) draw(pp, g_first, 0u, p01, p23);
    Counts cnt;
    int bad = 0;   // a wait of this thread gave up
    for (int h = 0; h < last; ++h) {
        const uint32_t colour = (uint32_t)h & 1u;
        const unsigned long long sweep = part.sweep0 + (unsigned long long)(h >> 1);
        uint8_t *mine = smem + colour * pb;
        const uint8_t *other = smem + (1u - colour) * pb;
        PhiloxPre pn = pp;   // of the next half-sweep's draws
        if (colour == 1u)
            philox_prepare(pn, (uint32_t)(sweep + 1ull), (uint32_t)((sweep + 1ull) >> 32), part.key0, part.key1);
        // The draws of group gn, of the next half-sweep when `over`.
        auto draw_next = [&](uint32_t gn, bool over, uint32_t (&d01)[4], uint32_t (&d23)[4]) {
            PhiloxPre q = pp;
            q.A = over ? pn.A : pp.A;
            q.B = over ? pn.B : pp.B;
            q.H2 = over ? pn.H2 : pp.H2;
            q.L2 = over ? pn.L2 : pp.L2;
            draw(q, gn, over ? 1u - colour : colour, d01, d23);
        };
        // One chunk whose neighbour rows are loaded: group g0, shared offset
        // at.  Interior: the next chunk's draws share its instruction block;
        // boundary: they wait until the neighbour has been served.
        auto chunk = [&](auto interior, IsingChunk &c, const ChunkCol<kFull> &col, uint32_t at, uint32_t y, uint32_t g0,
                         uint32_t gn, bool over, uint32_t (&Sn)[4]) {
            uint32_t C[4] = {0, 0, 0, 0}, O[4], F[4], d01[4], d23[4];
            const bool odd = ((colour + y) & 1u) != 0u;
            smem_words(mine + at, c.S);
            smem_words(other + at, O);
            if constexpr (kDis != kUniform) smem_words(dis + colour * pb + at, C);
            band_shifted<kFull>(col, odd, other + (at - col.j0), O, c.X);
#pragma unroll
            for (int w = 0; w < 4; ++w) c.O[w] = O[w];
            if constexpr (interior.value) draw_next(gn, over, d01, d23);
            ising_neighbours<kDis>(c, C, odd);
            if (flips16<kSym>(part.acc, c.n, c.St, p01, p23, F)) {
                Chunk16 e;
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    e.n[w] = c.n[w];
                    e.S[w] = c.St[w];
                }
                const uint4 f = band_exact(sh.sthr, sweep, part.key0, part.key1, g0, colour, e);
                F[0] = f.x;
                F[1] = f.y;
                F[2] = f.z;
                F[3] = f.w;
            }
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                Sn[w] = c.S[w] ^ F[w];
                if constexpr (interior.value) {
                    p01[w] = d01[w];
                    p23[w] = d23[w];
                }
            }
            store_words<4>(reinterpret_cast<int8_t *>(mine) + at, Sn);
            if constexpr (!interior.value) {
                const uint32_t box = 2u * (colour * b.cpr + (col.j0 >> 4));
                mail_put((y == b.y0 ? b.first : b.last) + box, part.epoch + (uint32_t)h + 1u, Sn);
                draw_next(gn, over, p01, p23);
            }
            if (colour == 1u) {
                ising_count<1, kDis, kFull>(c, Sn, col.vm, cnt);
#pragma unroll
                for (int w = 0; w < 4; ++w) cnt.mag = dot4(O[w], 0x01010101u & col.vm[w], cnt.mag);
                if constexpr (kRef) {
                    uint32_t R1[4], R0[4];
                    const int8_t *rp = g.ref + (size_t)y * b.half + col.j0;
                    load16_any<kFull>(rp + b.plane, col.nv, R1);
                    load16_any<kFull>(rp, col.nv, R0);
#pragma unroll
                    for (int w = 0; w < 4; ++w)
                        cnt.acf = dot4(Sn[w] & col.vm[w], R1[w], dot4(O[w] & col.vm[w], R0[w], cnt.acf));
                }
                cnt.up += (int)col.nv;
            } else if constexpr (kDis == kFields) {
                ising_count<0, kDis, kFull>(c, Sn, col.vm, cnt);
            }
        };
        {
            uint32_t at = at0, g0 = g00;
#pragma unroll 1
            for (uint32_t r = r0; r < rend; r += rsb) {
                IsingChunk c;
                uint32_t Sn[4];
                smem_words(other + at - b.pitch, c.U);
                smem_words(other + at + b.pitch, c.D);
                const bool more = r + rsb < rend;
                const uint32_t gn = more ? g0 + g_step : (has_edge ? edge_group(edge0) : g_first);
                chunk(std::true_type(), c, cc, at, b.y0 + r, g0, gn, !more && !has_edge, Sn);
                at += at_step;
                g0 += g_step;
            }
        }
#pragma unroll 1
        for (uint32_t e = edge0; e < edges; e += (uint32_t)kBandThreads) {
            const uint32_t r = edge_row(e), q = edge_col(e), y = b.y0 + r;
            const ChunkCol<kFull> col = chunk_col<kFull>(q, b.half);
            const uint32_t at = r * b.pitch + col.j0;
            const BandWait wt{b.src + (1u - colour) * b.plane, h > 0 ? part.epoch + (uint32_t)h : 0u,
                              2u * ((1u - colour) * b.cpr + q)};
            IsingChunk c;
            uint32_t Sn[4];
            if (!band_updown(b, part, wt, other, r, col.j0, col.nv, c.U, c.D)) bad = 1;
            const bool more = e + (uint32_t)kBandThreads < edges;
            chunk(std::false_type(), c, col, at, y, edge_group(e),
                  more ? edge_group(e + (uint32_t)kBandThreads) : g_first, !more, Sn);
        }
        pp = pn;
        if (colour == 1u) {
            cnt.up += cnt.mag / 2;   // nv sites of each plane: up = nv + mag / 2
            band_count(sh, h >> 1 & 1, cnt, false, kRef);
            if constexpr (kDis == kFields) {
                const int f = __reduce_add_sync(0xffffffffu, cnt.fld);
                if ((tid & 31u) == 0u) atomicAdd(&sh.fld, f);
            }
            cnt = Counts();
        }
        const int stop = __syncthreads_or(bad);
        if (colour == 1u) {
            band_post(sh, h >> 1 & 1, g, sweep, false, kRef);
            if constexpr (kDis == kFields) {
                if (tid == 64u) {
                    add_counter(fld_slot(g.ctrl, sweep), (long long)sh.fld);
                    sh.fld = 0;   // next added to a barrier later
                }
            }
        }
        if (stop) {
            sh.bad = 1;
            break;
        }
    }
    int8_t *fin = ((part.sweep0 + (unsigned long long)part.n) & 1) ? g.s[1] : g.s[0];
    for (int c = 0; c < 2; ++c)
        rows_out(smem + c * pb, b.pitch, b.nr, fin + c * b.plane + (size_t)b.y0 * b.half, b.half);
}

// Lattices with no more than one chunk a thread and colour, Ising or c-mode
// North-East: a half-sweep is one pass whose length is the latency from a
// neighbour's packet to this band's own, so everything else is taken off
// that path.  A thread keeps its chunk of both colours (and disorder bytes,
// reference, persistence bits) in registers; its draws of the next half-sweep
// are made after its packet has left -- all of them for North-East too,
// reduced to rejection masks, since with most threads idle a draw that is
// not needed costs nothing.  A row is a warp's where it fits, so that the two
// boundary rows wait side by side.
LAT_HD bool band_is_small(uint32_t L, uint32_t half, uint32_t bands)
{
    const uint32_t nr = (L + bands - 1u) / bands, cpr = (half + 15u) >> 4;
    return cpr <= 32u ? nr <= (uint32_t)kBandWarps : nr * cpr <= (uint32_t)kBandThreads;
}

template <bool kNe, bool kRef, int kDis, bool kSym, bool kFull>
LAT_D void band_small(const Geom &g, const BandPart &part, uint32_t band, uint32_t bands, uint8_t *mail,
                      BandShared &sh, uint8_t *smem)
{
    const Band b = band_of(g, part, band, bands, mail);
    const uint32_t tid = threadIdx.x, pb = b.nr * b.pitch;
    for (int c = 0; c < 2; ++c)
        rows_in(b.src + c * b.plane + (size_t)b.y0 * b.half, b.half, b.nr, smem + c * pb, b.pitch);
    if (tid < 16) sh.sthr[tid] = g.thr16[tid];
    if (tid < 10) (&sh.sum[0][0])[tid] = 0;
    if (tid == 10) sh.bad = 0;
    if (tid == 11) sh.fld = 0;
    if (tid == 12) sh.unfl = (int)(2u * b.nr * b.half);
    __syncthreads();
    const uint32_t r = b.cpr <= 32u ? tid >> 5 : tid / b.cpr, k = b.cpr <= 32u ? tid & 31u : tid - r * b.cpr;
    const bool mine = r < b.nr && k < b.cpr, top = r == 0u, bottom = r + 1u == b.nr;
    const ChunkCol<kFull> cc = chunk_col<kFull>(mine ? k : 0u, b.half);
    const uint32_t at = r * b.pitch + cc.j0, y = b.y0 + r, g0 = y * b.G + 4u * k;
    const NeRate rate = ne_rate(g.thr16);
    uint32_t S[2][4], C[2][4] = {}, Rf[2][4] = {}, was[2] = {0u, 0u};
    if (mine) {
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            smem_words(smem + c * pb + at, S[c]);
            const size_t ga = c * b.plane + (size_t)y * b.half + cc.j0;
            if constexpr (kDis != kUniform) load_words<4>(reinterpret_cast<const int8_t *>(g.cpl) + ga, C[c]);
            if constexpr (kRef) load16_any<kFull>(g.ref + ga, cc.nv, Rf[c]);
            if constexpr (kNe)
                for (uint32_t w = 0; w < 4u && 4u * k + w < b.G; ++w)
                    was[c] |= (uint32_t)g.flags[((size_t)c * g.rows + y) * b.G + 4u * k + w] << (8u * w);
        }
    }
    if constexpr (kNe) {
        const int n = __reduce_add_sync(0xffffffffu, __popc(was[0]) + __popc(was[1]));
        if ((tid & 31u) == 0u) atomicSub(&sh.unfl, n);
        __syncthreads();
    }
    uint32_t p01[4], p23[4];   // draws of the next half-sweep (North-East: p01 = rejections)
    auto draw = [&](unsigned long long sweep, uint32_t colour) {
        PhiloxPre pp;
        philox_prepare(pp, (uint32_t)sweep, (uint32_t)(sweep >> 32), part.key0, part.key1);
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const U4 u = philox_item(pp, g0 + (uint32_t)w, colour);
            if constexpr (kNe) p01[w] = ne_rejected(u, rate.K);
            else top_halves(u, p01[w], p23[w]);
        }
    };
    if (mine) draw(part.sweep0, 0u);
    Counts cnt;
    int bad = 0;   // a wait of this thread gave up
    auto half_sweep = [&](auto which, int h, unsigned long long sweep) {
        constexpr uint32_t colour = decltype(which)::value;
        uint8_t *own = smem + colour * pb;
        const uint8_t *other = smem + (1u - colour) * pb;
        if (mine) {
            const bool odd = ((colour + y) & 1u) != 0u;
            IsingChunk c;
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                c.S[w] = S[colour][w];
                c.O[w] = S[1u - colour][w];
            }
            band_shifted<kFull>(cc, odd, other + (at - cc.j0), S[1u - colour], c.X);
            const BandWait wt{b.src + (1u - colour) * b.plane, h > 0 ? part.epoch + (uint32_t)h : 0u,
                              2u * ((1u - colour) * b.cpr + k)};
            if (!band_updown(b, part, wt, other, r, cc.j0, cc.nv, c.U, c.D)) bad = 1;
            uint32_t F[4], Sn[4];
            [[maybe_unused]] uint32_t moved[4];
            if constexpr (kNe) {
                uint32_t cand[4], sure[4], ws[4], Sm[4];
                bool need[4];
                if (odd) ne_moves<kFull>(c.U, c.D, c.X, c.O, c.S, cc.vm, rate, cand, sure, ws, Sm, need);
                else ne_moves<kFull>(c.U, c.D, c.O, c.X, c.S, cc.vm, rate, cand, sure, ws, Sm, need);
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    moved[w] = sure[w] | (cand[w] & ~p01[w]);
                    F[w] = moved[w] & 0xFEFEFEFEu;
                }
            } else {
                ising_neighbours<kDis>(c, C[colour], odd);
                if (flips16<kSym>(part.acc, c.n, c.St, p01, p23, F)) {
                    Chunk16 e;
#pragma unroll
                    for (int w = 0; w < 4; ++w) {
                        e.n[w] = c.n[w];
                        e.S[w] = c.St[w];
                    }
                    const uint4 f = band_exact(sh.sthr, sweep, part.key0, part.key1, g0, colour, e);
                    F[0] = f.x;
                    F[1] = f.y;
                    F[2] = f.z;
                    F[3] = f.w;
                }
            }
#pragma unroll
            for (int w = 0; w < 4; ++w) Sn[w] = c.S[w] ^ F[w];
            const uint32_t box = 2u * (colour * b.cpr + k), tag = part.epoch + (uint32_t)h + 1u;
            if (top) mail_put(b.first + box, tag, Sn);
            if (bottom) mail_put(b.last + box, tag, Sn);
            store_words<4>(reinterpret_cast<int8_t *>(own) + at, Sn);
            draw(sweep + (colour == 1u ? 1ull : 0ull), 1u - colour);
            if constexpr (kNe) {
                const uint32_t chg = ne_changed(moved);
                cnt.unfl -= __popc(chg & ~was[colour]);
                was[colour] |= chg;
            }
            if constexpr (colour == 1u) {
                ising_count<1, kDis, kFull>(c, Sn, cc.vm, cnt);
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    cnt.mag = dot4(S[0][w], 0x01010101u & cc.vm[w], cnt.mag);
                    if constexpr (kRef)
                        cnt.acf = dot4(Sn[w] & cc.vm[w], Rf[1][w], dot4(S[0][w] & cc.vm[w], Rf[0][w], cnt.acf));
                }
                cnt.up = (int)cc.nv + cnt.mag / 2;   // nv sites of each plane
            } else if constexpr (kDis == kFields) {
                ising_count<0, kDis, kFull>(c, Sn, cc.vm, cnt);
            }
#pragma unroll
            for (int w = 0; w < 4; ++w) S[colour][w] = Sn[w];
        }
        if constexpr (colour == 1u) {
            band_count(sh, h >> 1 & 1, cnt, kNe, kRef);
            if constexpr (kDis == kFields) {
                const int f = __reduce_add_sync(0xffffffffu, cnt.fld);
                if ((tid & 31u) == 0u) atomicAdd(&sh.fld, f);
            }
            cnt = Counts();
        }
        const int stop = __syncthreads_or(bad);
        if constexpr (colour == 1u) {
            band_post(sh, h >> 1 & 1, g, sweep, kNe, kRef);
            if constexpr (kDis == kFields) {
                if (tid == 0u) {
                    add_counter(fld_slot(g.ctrl, sweep), (long long)sh.fld);
                    sh.fld = 0;   // next added to a barrier later
                }
            }
        }
        return stop;
    };
    for (int n = 0; n < part.n; ++n) {
        const unsigned long long sweep = part.sweep0 + (unsigned long long)n;
        int stop = half_sweep(std::integral_constant<uint32_t, 0>(), 2 * n, sweep);
        if (!stop) stop = half_sweep(std::integral_constant<uint32_t, 1>(), 2 * n + 1, sweep);
        if (stop) {
            sh.bad = 1;
            break;
        }
    }
    int8_t *fin = ((part.sweep0 + (unsigned long long)part.n) & 1) ? g.s[1] : g.s[0];
    for (int c = 0; c < 2; ++c)
        rows_out(smem + c * pb, b.pitch, b.nr, fin + c * b.plane + (size_t)b.y0 * b.half, b.half);
    if constexpr (kNe) {
        if (mine)
            for (int c = 0; c < 2; ++c)
                for (uint32_t w = 0; w < 4u && 4u * k + w < b.G; ++w)
                    g.flags[((size_t)c * g.rows + y) * b.G + 4u * k + w] = (uint8_t)(was[c] >> (8u * w));
    }
}

}  // namespace
}  // namespace lat
#endif
