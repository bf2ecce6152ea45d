// band_potts.cuh -- band-resident sweeps (band.cuh) of the 2D 3-state Potts
// model without field (J >= 0), two bit planes of 32 sites a word on the chip.
//
// Label k is held as the planes a = [k = 1], b = [k = 2]; the proposal
// k + 1 + p (mod 3), the unlike neighbours of both labels and their
// difference m are a few dozen logic operations for 32 sites (the byte-wise
// equality masks of the streaming kernel cost 20 instructions a site). A
// move is certain unless it makes m = 1 .. 4 more neighbours unlike; the four
// thresholds' bytes are picked by m's two low bits as permute selectors, eight
// sites a word, and compared on the top 16 bits (accept16.cuh). The draws are
// what bounds it: two sites a Philox call, about 1400 of a word's 1900 issue
// cycles. L = 2048: 15.7 us a sweep in two launches of the streaming kernel,
// 9.7 here. Tried and slower: a pair of lanes per word (10.9, the logic done
// twice), the boundary words' draws before their packets (9.9).
#pragma once

#include "band_bits.cuh"

#if defined(__CUDACC__)
namespace lat {
namespace {

// Number of set planes among four, bit-sliced.
struct Count4 {
    uint32_t b0, b1, b2;
};

LAT_D Count4 count4(uint32_t w, uint32_t x, uint32_t y, uint32_t z)
{
    const uint32_t s = w ^ x ^ y, c = (w & x) | (w & y) | (x & y);
    return Count4{s ^ z, c ^ (s & z), c & s & z};
}

// A word of labels, and its unlike sites against another.
struct Lab {
    uint32_t a, b;
};

LAT_D uint32_t unlike(const Lab &s, const Lab &t) { return (s.a ^ t.a) | (s.b ^ t.b); }

// Rejections by full 32-bit draws (rare; by value, out of line).
__device__ __noinline__ uint32_t potts_rejected_exact(uint4 K, unsigned long long sweep, uint32_t key0, uint32_t key1,
                                                      uint32_t g0, uint32_t colour, uint32_t m0, uint32_t m1, uint32_t m2)
{
    PhiloxPre pp;
    philox_prepare(pp, (uint32_t)sweep, (uint32_t)(sweep >> 32), key0, key1);
    uint32_t rej = 0;
#pragma unroll 1
    for (uint32_t c = 0; c < 16u; ++c) {
        const U4 u = philox_item(pp, g0 + c, colour);
#pragma unroll
        for (uint32_t w = 0; w < 2u; ++w) {
            const uint32_t i = 2u * c + w;
            const uint32_t t = (m2 >> i) & 1u ? K.w : (m1 >> i) & 1u ? ((m0 >> i) & 1u ? K.z : K.y) : K.x;
            if ((w ? u.z : u.x) > t) rej |= 1u << i;
        }
    }
    return rej;
}

template <bool kRef>
LAT_D void band_potts(const Geom &g, const BandPart &part, uint32_t band, uint32_t bands, uint8_t *mail,
                      BandShared &sh, uint8_t *smem)
{
    const uint32_t tid = threadIdx.x, L = (uint32_t)g.L, half = g.half, bw = (half + 31u) >> 5;
    const uint32_t nvl = half - 32u * (bw - 1u);
    uint32_t y0, y1;
    band_rows(band, bands, L, y0, y1);
    const uint32_t nr = y1 - y0, rend = nr - 1u, pw = nr * bw;
    // planes [colour][a, b], reference planes [colour][a, b]
    uint32_t *sm = reinterpret_cast<uint32_t *>(smem), *rf = sm + 4u * pw;
    const size_t plane = (size_t)g.plane;
    const int8_t *src = (part.sweep0 & 1) ? g.s[1] : g.s[0];
    const bool al = (half & 15u) == 0u;
    auto valid = [&](uint32_t k) { return k + 1u == bw ? nvl : 32u; };
    auto mask = [&](uint32_t k) { return 0xFFFFFFFFu >> (32u - valid(k)); };
    auto packed = [&](const int8_t *q, uint32_t c, uint32_t y, uint32_t k) {
        uint32_t w[8];
        load32(q + c * plane + (size_t)y * half + 32u * k, valid(k), al && valid(k) == 32u, w);
        return Lab{gather32(w, 0) & mask(k), gather32(w, 1) & mask(k)};
    };
    if (tid < 10) (&sh.sum[0][0])[tid] = 0;
    if (tid == 10) sh.bad = 0;
    for (uint32_t c = 0; c < 2u; ++c)
        for (uint32_t i = tid; i < pw; i += kBandThreads) {
            const uint32_t r = i / bw, k = i - r * bw;
            const Lab v = packed(src, c, y0 + r, k);
            sm[2u * c * pw + i] = v.a;
            sm[(2u * c + 1u) * pw + i] = v.b;
            if constexpr (kRef) {
                const Lab q = packed(g.ref, c, y0 + r, k);
                rf[2u * c * pw + i] = q.a;
                rf[(2u * c + 1u) * pw + i] = q.b;
            }
        }
    __syncthreads();
    // packet pairs: [band][first, last row][colour][word], one plane a packet
    unsigned *abort = reinterpret_cast<unsigned *>(mail);
    ulonglong2 *m = reinterpret_cast<ulonglong2 *>(mail + kAbortBytes);
    ulonglong2 *first = m + (size_t)band * 4u * bw, *last_row = first + 2u * bw;
    const ulonglong2 *above = m + (size_t)(band == 0u ? bands - 1u : band - 1u) * 4u * bw + 2u * bw;
    const ulonglong2 *below = m + (size_t)(band + 1u == bands ? 0u : band + 1u) * 4u * bw;
    const uint32_t up = y0 == 0u ? L - 1u : y0 - 1u, dn = y1 == L ? 0u : y1;
    const uint4 K = make_uint4(part.acc[0], part.acc[1], part.acc[2], part.acc[3]);   // t' for m = 1 .. 4
    // bytes 2 and 3 of the thresholds, in the order of m & 3: m = 4, 1, 2, 3
    const uint32_t lo4 = prmt(prmt(K.w, K.x, 0x0062u), prmt(K.y, K.z, 0x0062u), 0x5410u);
    const uint32_t hi4 = prmt(prmt(K.w, K.x, 0x0073u), prmt(K.y, K.z, 0x0073u), 0x5410u);
    const uint32_t rsb = (uint32_t)kBandThreads / bw, rr = tid / bw, kc = tid - rr * bw;
    const uint32_t r0 = rr < rsb ? 1u + rr : nr, edge0 = (uint32_t)kBandThreads - 1u - tid, edges = 2u * bw;
    Counts cnt;   // mag: sites in state 0
    int bad = 0, sites = 0;
    for (int h = 0; h < 2 * part.n; ++h) {
        const uint32_t colour = (uint32_t)h & 1u;
        const unsigned long long sweep = part.sweep0 + (unsigned long long)(h >> 1);
        PhiloxPre pp;
        philox_prepare(pp, (uint32_t)sweep, (uint32_t)(sweep >> 32), part.key0, part.key1);
        uint32_t *mine = sm + 2u * colour * pw;
        const uint32_t *other = sm + 2u * (1u - colour) * pw;
        auto word = [&](uint32_t r, uint32_t k, const Lab &U, const Lab &D) {
            const uint32_t at = r * bw + k, y = y0 + r, vm = mask(k), g0 = y * g.G + 16u * k;
            const Lab O{other[at], other[pw + at]}, S{mine[at], mine[pw + at]};
            const bool odd = ((colour + y) & 1u) != 0u;
            const Lab X{bit_side(other + r * bw, k, bw, nvl, odd, O.a), bit_side(other + pw + r * bw, k, bw, nvl, odd, O.b)};
            // draws: top halves of the acceptance words of sites t, t + 8, t + 16,
            // t + 24 (t = 0..7), and the proposal bits
            uint32_t p01[8], p23[8], p = 0;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                U4 u[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) u[c] = philox_item(pp, g0 + (uint32_t)(j + 4 * c), colour);
#pragma unroll
                for (int w = 0; w < 2; ++w) {
                    const int t = 2 * j + w;
                    p01[t] = prmt(word_of(u[0], 2 * w), word_of(u[1], 2 * w), 0x7632u);
                    p23[t] = prmt(word_of(u[2], 2 * w), word_of(u[3], 2 * w), 0x7632u);
                    // floor(u * 2 / 2^32): the top bit, spread over a byte each
                    const uint32_t lo = prmt(word_of(u[0], 2 * w + 1), word_of(u[1], 2 * w + 1), 0xFBFBu);
                    const uint32_t hi = prmt(word_of(u[2], 2 * w + 1), word_of(u[3], 2 * w + 1), 0xFBFBu);
                    p |= (lo & (0x00000101u << t)) | (hi & (0x01010000u << t));
                }
            }
            const uint32_t z = ~(S.a | S.b);
            const Lab T{(z & ~p) | (S.b & p), (z & p) | (S.a & ~p)};
            const Count4 o = count4(unlike(S, U), unlike(S, D), unlike(S, O), unlike(S, X));
            const Count4 n = count4(unlike(T, U), unlike(T, D), unlike(T, O), unlike(T, X));
            // m = n - o, two's complement in three bits and the borrow
            const uint32_t m0 = n.b0 ^ o.b0, w0 = ~n.b0 & o.b0;
            const uint32_t m1 = n.b1 ^ o.b1 ^ w0, w1 = (~n.b1 & o.b1) | (~n.b1 & w0) | (o.b1 & w0);
            const uint32_t m2 = n.b2 ^ o.b2 ^ w1, neg = (~n.b2 & o.b2) | (~n.b2 & w1) | (o.b2 & w1);
            uint32_t rej = 0, tie = kNoTie;
#pragma unroll
            for (int t = 0; t < 4; ++t) {   // sites t + 4 n: a selector nibble each
                const uint32_t sel = ((m0 >> t) & 0x11111111u) | ((t ? m1 >> (t - 1) : m1 << 1) & 0x22222222u);
                const uint32_t la = prmt(lo4, lo4, sel), ha = prmt(hi4, hi4, sel);
                const uint32_t lb = prmt(lo4, lo4, sel >> 16), hb = prmt(hi4, hi4, sel >> 16);
                rej |= reject4(prmt(la, ha, 0x6240u), prmt(lb, hb, 0x6240u), p01[t], p23[t], tie) & (0x01010101u << t);
                rej |= reject4(prmt(la, ha, 0x7351u), prmt(lb, hb, 0x7351u), p01[t + 4], p23[t + 4], tie) &
                       (0x10101010u << t);
            }
            if (tie_hit(tie))
                rej = potts_rejected_exact(K, sweep, part.key0, part.key1, g0, colour, m0, m1, m2);
            const uint32_t mv = ~rej | neg | ~(m0 | m1 | m2);
            const Lab N{((T.a & mv) | (S.a & ~mv)) & vm, ((T.b & mv) | (S.b & ~mv)) & vm};
            mine[at] = N.a;
            mine[pw + at] = N.b;
            if (colour == 1u) {
                const uint32_t f0 = (n.b0 & mv) | (o.b0 & ~mv), f1 = (n.b1 & mv) | (o.b1 & ~mv),
                               f2 = (n.b2 & mv) | (o.b2 & ~mv);
                cnt.bond -= __popc(f0 & vm) + 2 * __popc(f1 & vm) + 4 * __popc(f2 & vm);   // unlike bonds
                cnt.mag += __popc(~(N.a | N.b) & vm) + __popc(~(O.a | O.b) & vm);
                if constexpr (kRef) {
                    const Lab R1{rf[2u * pw + at], rf[3u * pw + at]}, R0{rf[at], rf[pw + at]};
                    cnt.acf += __popc(~unlike(N, R1) & vm) + __popc(~unlike(O, R0) & vm);
                }
                sites += (int)valid(k);
            }
            return N;
        };
        auto row_lab = [&](uint32_t r, uint32_t k) { return Lab{other[r * bw + k], other[pw + r * bw + k]}; };
#pragma unroll 1
        for (uint32_t r = r0; r < rend; r += rsb) word(r, kc, row_lab(r - 1u, kc), row_lab(r + 1u, kc));
#pragma unroll 1
        for (uint32_t e = edge0; e < edges; e += (uint32_t)kBandThreads) {
            const bool lo = e < bw;   // the last row's words, then the first row's
            const uint32_t k = lo ? e : e - bw, r = lo ? rend : 0u;
            Lab far{0u, 0u};
            if (h == 0) {
                far = packed(src, 1u - colour, lo ? dn : up, k);
            } else {
                const unsigned long long *box =
                    reinterpret_cast<const unsigned long long *>((lo ? below : above) + (1u - colour) * bw + k);
                if (!mail_take_word(box, part.epoch + (uint32_t)h, part, abort, far.a) ||
                    !mail_take_word(box + 1, part.epoch + (uint32_t)h, part, abort, far.b))
                    bad = 1;
            }
            const Lab near = row_lab(lo ? rend - 1u : 1u, k);
            const Lab N = word(r, k, lo ? near : far, lo ? far : near);
            unsigned long long *out =
                reinterpret_cast<unsigned long long *>((lo ? last_row : first) + colour * bw + k);
            mail_put_word(out, part.epoch + (uint32_t)h + 1u, N.a);
            mail_put_word(out + 1, part.epoch + (uint32_t)h + 1u, N.b);
        }
        if (colour == 1u) {
            cnt.bond += 4 * sites;
            cnt.up = 2 * sites - cnt.mag;
            band_count(sh, h >> 1 & 1, cnt, false, kRef);
            cnt = Counts();
            sites = 0;
        }
        const int stop = __syncthreads_or(bad);
        if (colour == 1u) band_post(sh, h >> 1 & 1, g, sweep, false, kRef);
        if (stop) {
            sh.bad = 1;
            break;
        }
    }
    int8_t *fin = ((part.sweep0 + (unsigned long long)part.n) & 1) ? g.s[1] : g.s[0];
    for (uint32_t c = 0; c < 2u; ++c)
        for (uint32_t i = tid; i < pw; i += kBandThreads) {
            const uint32_t r = i / bw, k = i - r * bw;
            const uint32_t a = sm[2u * c * pw + i], b = sm[(2u * c + 1u) * pw + i];
            uint32_t w[8];
#pragma unroll
            for (int j = 0; j < 8; ++j)
                w[j] = (((a >> (4 * j)) & 0xFu) * 0x00204081u & 0x01010101u) +
                       2u * (((b >> (4 * j)) & 0xFu) * 0x00204081u & 0x01010101u);
            store32(w, fin + c * plane + (size_t)(y0 + r) * half + 32u * k, valid(k), al && valid(k) == 32u);
        }
}

}  // namespace
}  // namespace lat
#endif
