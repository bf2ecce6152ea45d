// band_kinds.cuh -- which form of the band-resident sweep a lattice takes, and
// the memory it needs: shared by the solo and the batched launches.
#pragma once

#include "band_bits.cuh"
#include "band_potts.cuh"

#if defined(__CUDACC__)
namespace lat {
namespace {

// End of a CTA's run: tell the host if a wait gave up; band 0 moves the
// lattice's sweep counter on.
LAT_D void band_end(const Geom &g, const BandPart &p, uint32_t band, const BandShared &sh)
{
    if (threadIdx.x != 0) return;
    if (sh.bad) {
        *reinterpret_cast<volatile int *>(p.err) = 1;
        if (p.err_all != nullptr) *reinterpret_cast<volatile int *>(p.err_all) = 1;
    }
    if (band == 0u) g.ctrl->sweep = p.sweep0 + (unsigned long long)p.n;
}

// Kinds: Ising with a general or a symmetric table and North-East, each with
// a partial last chunk or without; without: bonds (either table), fields;
// bit-packed layout: Ising (symmetric table), North-East; 3-state Potts.
enum BandKind { kBandGen = 0, kBandSym, kBandNe, kBandGenFull, kBandSymFull, kBandNeFull, kBandBondGen, kBandBondSym,
                kBandFields, kBandPacked, kBandPackedNe, kBandPotts3, kBandKinds };

// Kinds that have one bit a site on the chip unless the bands are small.
LAT_HD bool band_kind_bits(int kind)
{
    return kind == kBandSym || kind == kBandSymFull || kind == kBandNe || kind == kBandNeFull || kind == kBandBondSym ||
           kind >= kBandPacked;
}

// kT: threads of the CTA; kForm: small bands (0), the others (1), either (2).
template <int kKind, bool kRef, int kT, int kForm>
LAT_D void band_body(const Geom &g, const BandPart &part, uint32_t band, uint32_t bands, uint8_t *mail,
                     BandShared &sh, uint8_t *smem)
{
    constexpr bool kNe = kKind == kBandNe || kKind == kBandNeFull || kKind == kBandPackedNe;
    constexpr bool kFull = kKind != kBandGen && kKind != kBandSym && kKind != kBandNe;
    constexpr bool kSym = kKind == kBandSym || kKind == kBandSymFull || kKind == kBandBondSym;
    constexpr int kDis = kKind == kBandBondGen || kKind == kBandBondSym ? kBonds : (kKind == kBandFields ? kFields : kUniform);
    constexpr bool kPacked = kKind == kBandPacked || kKind == kBandPackedNe;
    if constexpr (kKind == kBandPotts3) {
        band_potts<kRef>(g, part, band, bands, mail, sh, smem);
    } else if constexpr (kPacked) {
        band_bits<kNe, kRef, false, true, kT>(g, part, band, bands, mail, sh, smem);
    } else {
        if (kForm == 0 || (kForm == 2 && band_is_small((uint32_t)g.L, g.half, bands))) {
            band_small<kNe, kRef, kDis, kSym, kFull>(g, part, band, bands, mail, sh, smem);
        } else if constexpr (kForm != 0) {
            if constexpr (kNe || kSym) band_bits<kNe, kRef, kDis == kBonds, false, kT>(g, part, band, bands, mail, sh, smem);
            else band_ising<kRef, kDis, kSym, kFull>(g, part, band, bands, mail, sh, smem);
        }
    }
}

inline int band_kind(const Geom &k, bool fields)
{
    if (k.bits[0] != nullptr) return k.model == LAT_NE ? kBandPackedNe : kBandPacked;
    if (k.model == LAT_POTTS) return kBandPotts3;
    const int full = k.half % 16 == 0 ? kBandGenFull : kBandGen;
    if (k.model == LAT_NE) return full + kBandNe;
    if (k.cpl == nullptr) return full + (k.acc_sym ? kBandSym : kBandGen);
    return fields ? kBandFields : (k.acc_sym ? kBandBondSym : kBandBondGen);
}

inline bool band_on_bits(const Geom &k, int kind, int bands)
{
    return kind >= kBandPacked || (band_kind_bits(kind) && !band_is_small((uint32_t)k.L, k.half, (uint32_t)bands));
}

// k: a tiled_geom descriptor.  Rows per band are at least 2, so a lattice has
// at most L / 2 bands.
inline size_t band_smem_bytes(const Geom &k, int kind, int bands, int threads = kBandThreads)
{
    const size_t nr = ((size_t)k.L + bands - 1) / bands, ref = k.ref != nullptr || k.ref_bits != nullptr ? 1 : 0;
    if (band_on_bits(k, kind, bands)) {
        const size_t bw = ((size_t)k.half + 31) / 32;
        if (kind == kBandPotts3) return 4 * nr * bw * (1 + ref) * 4;
        size_t words = 2 * (nr + 2) * bw + 2 * nr * bw * ref;
        if (kind == kBandBondSym) words += 8 * nr * bw;
        if (k.model == LAT_NE) words += 2 * nr * bw + (size_t)threads / 32 * kBitQueue;
        return words * 4;
    }
    const size_t pitch = ((size_t)k.half + 15) & ~(size_t)15;
    return 2 * nr * pitch * (k.cpl != nullptr ? 2 : 1);
}

// Packet pairs of a lattice.
inline size_t band_mail_pairs(const Geom &k, int kind, int bands)
{
    if (band_on_bits(k, kind, bands)) return (size_t)bands * (kind == kBandPotts3 ? 4 : 2) * ((k.half + 31) / 32);
    return (size_t)bands * 2 * 4 * ((k.half + 15) / 16);
}

// Threads and words or chunks of a row fit the kernels' indices.
inline bool band_fits(const Geom &k, int kind, int bands)
{
    const size_t nr = ((size_t)k.L + bands - 1) / bands;
    const size_t cols = band_on_bits(k, kind, bands) ? (k.half + 31) / 32 : (k.half + 15) / 16;
    return cols <= (size_t)kBandThreads && nr < 2048 && band_smem_bytes(k, kind, bands) <= kBandMaxSmem;
}

// Whether a lattice can run in bands at all (fields: its field signs are set).
inline bool band_kind_ok(const Geom &g, int kind)
{
    if (kind == kBandPacked) return bitpacked_supported(g) && tiled_geom(g).acc_sym != 0;
    if (kind == kBandPackedNe) return bitpacked_supported(g) && g.cmode != 0;
    if (kind == kBandPotts3) return g.potts3_ok != 0 && g.cpl == nullptr;
    if (g.model == LAT_NE) return ne_walk_supported(g);
    if (g.model != LAT_ISING) return false;
    return g.cpl == nullptr ? any_supported(g) : wide_supported(g);
}

inline BandPart band_part(const Geom &k, unsigned long long sweep0, int n, unsigned epoch, int *err)
{
    BandPart p = {};
    p.epoch = epoch;
    p.sweep0 = sweep0;
    p.err = err;
    p.limit = band_test().limit;
    p.n = n;
    p.key0 = k.key0;
    p.key1 = k.key1;
    for (int i = 0; i < 8; ++i) p.acc[i] = k.model == LAT_POTTS ? (i < 4 ? k.potts3[i] : 0u) : k.acc[i];
    return p;
}

}  // namespace
}  // namespace lat
#endif
