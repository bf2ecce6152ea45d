// band_bits.cuh -- band-resident sweeps (band.cuh) with one bit per site on
// the chip, whatever the lattice's layout in memory.
//
// Spin-1/2 sites are bits: 32 sites share every logic operation of the
// neighbour count, an Ising word costs little more than its Philox draws
// (bits_step.cuh), and a North-East word about 40 instructions plus its
// undecided groups' draws.  int8 lattices are packed as they are loaded and
// unpacked as they are written back, once per call.  One bit a site also
// puts lattices up to L = 16384 (Ising) and about 11000 (North-East with its
// persistence bits) into shared memory.  Used for Ising with a symmetric
// table (J >= 0, h = 0), uniform or with bond signs, and c-mode North-East;
// bands of at most one 16-site chunk a thread stay on the int8 form
// (band_small), whose half-sweep is shorter.
#pragma once

#include "band.cuh"
#include "bits_step.cuh"

#if defined(__CUDACC__)
namespace lat {
namespace {

constexpr uint32_t kBitQueue = 32 + 8 * 32;   // jobs per warp: under 32 left over, 8 groups per lane new

// 32 bytes from q, of which nv exist (al: q is 16-byte aligned and nv = 32).
LAT_D void load32(const int8_t *q, uint32_t nv, bool al, uint32_t (&w)[8])
{
    if (al) {
        const uint4 a = reinterpret_cast<const uint4 *>(q)[0], b = reinterpret_cast<const uint4 *>(q)[1];
        w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w;
        w[4] = b.x; w[5] = b.y; w[6] = b.z; w[7] = b.w;
        return;
    }
    const uintptr_t a = reinterpret_cast<uintptr_t>(q);
    const uint32_t sh = (uint32_t)(a & 3u);
    const uint32_t *p = reinterpret_cast<const uint32_t *>(a - sh);
    uint32_t x[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) x[i] = 4u * (uint32_t)i < nv + sh ? p[i] : 0u;
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = __funnelshift_r(x[i], x[i + 1], 8u * sh);
}

// Bit i = bit `bit` of byte i.
LAT_D uint32_t gather32(const uint32_t (&w)[8], int bit)
{
    uint32_t v = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) v |= (uint32_t)dot4((w[i] >> bit) & 0x01010101u, 0x08040201u, 0) << (4 * i);
    return v;
}

// Up bits of 32 spins.
LAT_D uint32_t pack32(const int8_t *q, uint32_t nv, bool al, uint32_t vm)
{
    uint32_t w[8];
    load32(q, nv, al, w);
    return ~gather32(w, 7) & vm;
}

// The way back: 32 bytes to q, only the nv that exist.
LAT_D void store32(const uint32_t (&w)[8], int8_t *q, uint32_t nv, bool al)
{
    if (al) {
        reinterpret_cast<uint4 *>(q)[0] = make_uint4(w[0], w[1], w[2], w[3]);
        reinterpret_cast<uint4 *>(q)[1] = make_uint4(w[4], w[5], w[6], w[7]);
    } else if ((reinterpret_cast<uintptr_t>(q) & 3u) == 0u && (nv & 3u) == 0u) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (4u * (uint32_t)i < nv) reinterpret_cast<uint32_t *>(q)[i] = w[i];
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int b = 0; b < 4; ++b)
                if (4u * (uint32_t)i + (uint32_t)b < nv) q[4 * i + b] = (int8_t)(w[i] >> (8 * b));
    }
}

LAT_D void unpack32(uint32_t v, int8_t *q, uint32_t nv, bool al)
{
    uint32_t w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = ~((((v >> (4 * i)) & 0xFu) * 0x00204081u & 0x01010101u) * 0xFEu);
    store32(w, q, nv, al);
}

// One row of the other plane as words: its word k shifted towards the side
// neighbours (odd: east), the row taken round; nvl = valid bits of its last
// word (bits past them are 0).
LAT_D uint32_t bit_side(const uint32_t *row, uint32_t k, uint32_t bw, uint32_t nvl, bool odd, uint32_t O)
{
    if (odd) {
        const bool end = k + 1u == bw;
        const uint32_t next = row[end ? 0u : k + 1u];
        const uint32_t o = end && nvl < 32u ? O | (next & 1u) << nvl : O;
        return __funnelshift_r(o, next, 1);
    }
    const uint32_t prev = k == 0u ? row[bw - 1u] << (32u - nvl) : row[k - 1u];
    return __funnelshift_l(prev, O, 1);
}

// kT: threads of the CTA.
template <bool kNe, bool kRef, bool kBonds, bool kPacked, int kT>
LAT_D void band_bits(const Geom &g, const BandPart &part, uint32_t band, uint32_t bands, uint8_t *mail,
                     BandShared &sh, uint8_t *smem)
{
    const uint32_t tid = threadIdx.x, L = (uint32_t)g.L, half = g.half, bw = (half + 31u) >> 5;
    const uint32_t nvl = half - 32u * (bw - 1u);   // valid bits of a row's last word
    uint32_t y0, y1;
    band_rows(band, bands, L, y0, y1);
    const uint32_t nr = y1 - y0, rend = nr - 1u, pw = (nr + 2u) * bw, fw = nr * bw;
    // planes with a halo row either side; then disorder planes [colour][bond],
    // persistence planes, reference planes, job queues
    uint32_t *sm = reinterpret_cast<uint32_t *>(smem);
    uint32_t *dis = sm + 2u * pw, *fl = dis + (kBonds ? 8u * fw : 0u), *rf = fl + (kNe ? 2u * fw : 0u);
    uint32_t *queue = rf + (kRef ? 2u * fw : 0u) + (tid >> 5) * kBitQueue;
    const size_t plane = (size_t)g.plane;
    const bool odd_buf = (part.sweep0 & 1) != 0;
    const int8_t *src = odd_buf ? g.s[1] : g.s[0];
    const uint32_t *bsrc = odd_buf ? g.bits[1] : g.bits[0];
    auto valid = [&](uint32_t k) { return k + 1u == bw ? nvl : 32u; };
    auto mask = [&](uint32_t k) { return 0xFFFFFFFFu >> (32u - valid(k)); };
    const bool al = (half & 15u) == 0u;
    auto spins_at = [&](uint32_t c, uint32_t y, uint32_t k) {   // before the launch
        if constexpr (kPacked) return bsrc[((size_t)c * L + y) * bw + k];
        else return pack32(src + c * plane + (size_t)y * half + 32u * k, valid(k), al && valid(k) == 32u, mask(k));
    };
    if (tid < 10) (&sh.sum[0][0])[tid] = 0;
    if (tid == 10) sh.bad = 0;
    if (tid == 12) sh.unfl = (int)(2u * nr * half);
    __syncthreads();
    int changed = 0;
    for (uint32_t c = 0; c < 2u; ++c)
        for (uint32_t i = tid; i < fw; i += kT) {
            const uint32_t r = i / bw, k = i - r * bw, y = y0 + r;
            sm[c * pw + bw + i] = spins_at(c, y, k);
            if constexpr (kRef) {
                if constexpr (kPacked) rf[c * fw + i] = g.ref_bits[((size_t)c * L + y) * bw + k];
                else rf[c * fw + i] = pack32(g.ref + c * plane + (size_t)y * half + 32u * k, valid(k),
                                             al && valid(k) == 32u, mask(k));
            }
            if constexpr (kBonds) {
                uint32_t w[8];
                load32(reinterpret_cast<const int8_t *>(g.cpl) + c * plane + (size_t)y * half + 32u * k, valid(k),
                       al && valid(k) == 32u, w);
#pragma unroll
                for (int d = 0; d < 4; ++d) dis[(4u * c + (uint32_t)d) * fw + i] = gather32(w, d);
            }
            if constexpr (kNe) {
                const uint8_t *q = g.flags + ((size_t)c * g.rows + y) * g.G + 8u * k;   // a byte's low nibble per group
                uint32_t f = 0;
                if ((g.G & 7u) == 0u) {
                    const uint2 v = *reinterpret_cast<const uint2 *>(q);
                    const uint32_t a = (v.x | v.x >> 4) & 0x00FF00FFu, e = (v.y | v.y >> 4) & 0x00FF00FFu;
                    f = ((a | a >> 8) & 0xFFFFu) | (e | e >> 8) << 16;
                } else {
                    for (uint32_t m = 0; m < 8u && 8u * k + m < g.G; ++m) f |= (uint32_t)q[m] << (4u * m);
                }
                fl[c * fw + i] = f;
                changed += __popc(f);
            }
        }
    if constexpr (kNe) {
        changed = __reduce_add_sync(0xffffffffu, changed);
        if ((tid & 31u) == 0u) atomicSub(&sh.unfl, changed);
    }
    __syncthreads();
    // packets: [band][first, last row][colour][word]
    unsigned *abort = reinterpret_cast<unsigned *>(mail);
    unsigned long long *m = reinterpret_cast<unsigned long long *>(mail + kAbortBytes) + 2u * (size_t)part.mail;
    unsigned long long *first = m + (size_t)band * 4u * bw, *last_row = first + 2u * bw;
    const unsigned long long *above = m + (size_t)(band == 0u ? bands - 1u : band - 1u) * 4u * bw + 2u * bw;
    const unsigned long long *below = m + (size_t)(band + 1u == bands ? 0u : band + 1u) * 4u * bw;
    const uint32_t up = y0 == 0u ? L - 1u : y0 - 1u, dn = y1 == L ? 0u : y1;
    const SymK sk = bits_sym(g.thr16);
    const NeRate rate = ne_rate(g.thr16);
    const uint32_t lane = tid & 31u;
    // interior rows 1 .. nr - 2: thread (rr, k); the boundary rows' words are
    // the last threads'
    const uint32_t rsb = (uint32_t)kT / bw, rr = tid / bw, kc = tid - rr * bw;
    const uint32_t r0 = rr < rsb ? 1u + rr : nr, edge0 = (uint32_t)kT - 1u - tid, edges = 2u * bw;
    Counts cnt;   // mag counts up spins
    int bad = 0, sites = 0;
    for (int h = 0; h < 2 * part.n; ++h) {
        const uint32_t colour = (uint32_t)h & 1u;
        const unsigned long long sweep = part.sweep0 + (unsigned long long)(h >> 1);
        PhiloxPre pp;
        philox_prepare(pp, (uint32_t)sweep, (uint32_t)(sweep >> 32), part.key0, part.key1);
        uint32_t *mine = sm + colour * pw, *other = sm + (1u - colour) * pw;
        unsigned queued = 0;   // warp-uniform
        // A queued group: draw, accept, apply.
        auto job = [&](uint32_t e) {
            const uint32_t k = e & 511u, r = (e >> 9) & 2047u, q = (e >> 20) & 7u, y = y0 + r;
            const uint32_t rej = ne_rejected(philox_item(pp, y * g.G + 8u * k + q, colour), rate.K);
            const uint32_t acc = (e >> 24) & ~((uint32_t)dot4(rej & 0x01010101u, 0x08040201u, 0));
            if (acc == 0u) return;
            const uint32_t mv = acc << (4u * q), at = (r + 1u) * bw + k;
            atomicXor(&mine[at], mv);
            const uint32_t was = atomicOr(&fl[colour * fw + r * bw + k], mv);
            cnt.unfl -= __popc(mv & ~was);
            if (colour == 1u) {
                // north and east are up, so a site's neighbour sum is 4 - 2 (west down + south down)
                const bool odd = ((colour + y) & 1u) != 0u;
                const uint32_t O = other[at], W = odd ? O : bit_side(other + (r + 1u) * bw, k, bw, nvl, false, O);
                const int n = __popc(acc), side = __popc(mv & ~W) + __popc(mv & ~other[at + bw]);
                const int sg = rate.inv ? -1 : 1;
                cnt.mag += sg * n;
                cnt.bond += sg * (8 * n - 4 * side);
                if constexpr (kRef) cnt.acf += sg * (4 * __popc(mv & rf[fw + r * bw + k]) - 2 * n);
            }
        };
        auto drain = [&](bool all) {
            __syncwarp();
            while (queued >= 32u) {
                queued -= 32u;
                job(queue[queued + lane]);
            }
            if (all && lane < queued) job(queue[lane]);
            __syncwarp();
        };
        // Word k of row r between U and D; returns its new spins (North-East:
        // after the certain moves; the undecided sites' flags go to cand).
        auto word = [&](uint32_t r, uint32_t k, uint32_t U, uint32_t D, uint32_t &cand) {
            const uint32_t at = (r + 1u) * bw + k, y = y0 + r, O = other[at], S = mine[at];
            const bool odd = ((colour + y) & 1u) != 0u;
            const uint32_t X = bit_side(other + (r + 1u) * bw, k, bw, nvl, odd, O);
            const uint32_t vm = mask(k);
            uint32_t a = U, d = D, o = O, x = X;
            if constexpr (kBonds) {   // a negative bond enters as a flipped neighbour
                const uint32_t *b = dis + 4u * colour * fw + r * bw + k;
                x ^= b[(odd ? 1u : 0u) * fw];
                o ^= b[(odd ? 0u : 1u) * fw];
                a ^= b[2u * fw];
                d ^= b[3u * fw];
            }
            const Nbr n = nbr_sum(a, d, o, x);
            uint32_t Sn;
            if constexpr (kNe) {
                const uint32_t open = U & (odd ? X : O) & vm, draws = ~(S ^ rate.inv);
                const uint32_t sure = open & ~draws;
                cand = open & draws;
                Sn = S ^ sure;
                if (sure != 0u) {
                    uint32_t *f = &fl[colour * fw + r * bw + k];
                    const uint32_t was = *f;
                    *f = was | sure;
                    cnt.unfl -= __popc(sure & ~was);
                }
            } else {
                Sn = bits_step(sk, g.thr16, pp, sweep, part.key0, part.key1, y * g.G + 8u * k, colour, n, S) & vm;
            }
            mine[at] = Sn;
            if (colour == 1u) {
                cnt.bond -= 2 * (__popc((n.s1 ^ Sn) & vm) + 2 * __popc((n.c1 ^ Sn) & vm) + __popc((n.R ^ Sn) & vm));
                cnt.mag += __popc(Sn) + __popc(O);
                if constexpr (kRef)
                    cnt.acf -= 2 * (__popc(Sn ^ rf[fw + r * bw + k]) + __popc(O ^ rf[r * bw + k]));
                sites += (int)valid(k);
            }
            return Sn;
        };
        // Queue the groups of cand.
        auto push = [&](uint32_t r, uint32_t k, uint32_t cand) {
            if (!__any_sync(0xffffffffu, cand != 0u)) return;
            uint32_t z = cand | cand >> 1;
            z = (z | z >> 2) & 0x11111111u;
            const uint32_t n = (uint32_t)__popc(z);
            uint32_t incl = n;
#pragma unroll
            for (int s = 1; s < 32; s *= 2) {
                const uint32_t t = __shfl_up_sync(0xffffffffu, incl, s);
                if (lane >= (uint32_t)s) incl += t;
            }
            uint32_t at = queued + incl - n;
            while (z != 0u) {
                const uint32_t b = (uint32_t)__ffs((int)z) - 1u;
                z &= z - 1u;
                queue[at++] = k | r << 9 | b << 18 | ((cand >> b) & 0xFu) << 24;   // b = 4 q
            }
            queued += __shfl_sync(0xffffffffu, incl, 31);
            if (queued >= 32u) drain(false);
        };
        if constexpr (kNe) {   // the warp's lanes stay in step
            for (uint32_t r = r0;; r += rsb) {
                const bool act = r < rend;
                if (!__any_sync(0xffffffffu, act)) break;
                uint32_t cand = 0;
                if (act) word(r, kc, other[r * bw + kc], other[(r + 2u) * bw + kc], cand);
                push(r, kc, cand);
            }
        } else {
            uint32_t none;
#pragma unroll 1
            for (uint32_t r = r0; r < rend; r += rsb) word(r, kc, other[r * bw + kc], other[(r + 2u) * bw + kc], none);
        }
        for (uint32_t e = edge0;; e += (uint32_t)kT) {
            const bool act = e < edges;
            if (!__any_sync(0xffffffffu, act)) break;
            uint32_t cand = 0, k = 0, r = 0;
            if (act) {
                const bool lo = e < bw;   // the last row's words, then the first row's
                k = lo ? e : e - bw;
                r = lo ? rend : 0u;
                uint32_t far = 0;
                if (h == 0) far = spins_at(1u - colour, lo ? dn : up, k);
                else if (!mail_take_word((lo ? below : above) + (1u - colour) * bw + k, part.epoch + (uint32_t)h, part, abort, far))
                    bad = 1;
                const uint32_t near = other[(lo ? rend : 2u) * bw + k];   // row rend - 1, row 1
                if constexpr (kNe) {
                    if (lo) other[(nr + 1u) * bw + k] = far;   // queued moves look south
                }
                const uint32_t Sn = word(r, k, lo ? near : far, lo ? far : near, cand);
                if constexpr (!kNe)
                    mail_put_word((lo ? last_row : first) + colour * bw + k, part.epoch + (uint32_t)h + 1u, Sn);
            }
            if constexpr (kNe) push(r, k, cand);
        }
        if constexpr (kNe) drain(true);
        if (colour == 1u) {
            cnt.bond += 4 * sites;
            cnt.up = cnt.mag;
            cnt.mag = 2 * cnt.mag - 2 * sites;
            if constexpr (kRef) cnt.acf += 2 * sites;
            band_count(sh, h >> 1 & 1, cnt, kNe, kRef);
            cnt = Counts();
            sites = 0;
        }
        const int stop = __syncthreads_or(bad);
        if constexpr (kNe) {   // boundary rows out, their queued moves done
            for (uint32_t i = tid; i < edges; i += kT) {
                const bool lo = i < bw;
                const uint32_t k = lo ? i : i - bw;
                mail_put_word((lo ? last_row : first) + colour * bw + k, part.epoch + (uint32_t)h + 1u,
                              mine[(lo ? nr : 1u) * bw + k]);
            }
        }
        if (colour == 1u) band_post(sh, h >> 1 & 1, g, sweep, kNe, kRef);
        if (stop) {
            sh.bad = 1;
            break;
        }
    }
    const bool fin_odd = ((part.sweep0 + (unsigned long long)part.n) & 1) != 0;
    int8_t *fin = fin_odd ? g.s[1] : g.s[0];
    uint32_t *bfin = fin_odd ? g.bits[1] : g.bits[0];
    for (uint32_t c = 0; c < 2u; ++c)
        for (uint32_t i = tid; i < fw; i += kT) {
            const uint32_t r = i / bw, k = i - r * bw, y = y0 + r;
            const uint32_t v = sm[c * pw + bw + i];
            if constexpr (kPacked) bfin[((size_t)c * L + y) * bw + k] = v;
            else unpack32(v, fin + c * plane + (size_t)y * half + 32u * k, valid(k), al && valid(k) == 32u);
            if constexpr (kNe) {
                uint8_t *q = g.flags + ((size_t)c * g.rows + y) * g.G + 8u * k;
                const uint32_t f = fl[c * fw + i];
                if ((g.G & 7u) == 0u) {
                    auto spread = [](uint32_t x) {   // four nibbles to four bytes
                        x = (x | x << 8) & 0x00FF00FFu;
                        return (x | x << 4) & 0x0F0F0F0Fu;
                    };
                    *reinterpret_cast<uint2 *>(q) = make_uint2(spread(f & 0xFFFFu), spread(f >> 16));
                } else {
                    for (uint32_t mm = 0; mm < 8u && 8u * k + mm < g.G; ++mm) q[mm] = (uint8_t)((f >> (4u * mm)) & 0xFu);
                }
            }
        }
}

}  // namespace
}  // namespace lat
#endif
