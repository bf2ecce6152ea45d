// kernels_band_batch.cu -- the band-resident kernel (band.cuh) for a batch:
// the SMs are shared out over uneven 2D lattices, each a ring of bands, and
// every lattice runs all its sweeps in the one cooperative launch.
#include <algorithm>
#include <cmath>

#include "band_host.h"
#include "band_kinds.cuh"

namespace lat {

namespace {

// A CTA's part is a kernel parameter (uniform loads), the lattice's
// descriptor is read from memory once.
struct BandParts {
    BandPart p[kBandMaxCtas];
};

template <bool kRef>
LAT_D void band_any(const Geom &g, const BandPart &part, uint8_t *mail, BandShared &sh, uint8_t *smem)
{
    switch (part.kind) {
    case kBandGen: band_body<kBandGen, kRef, kBandThreads, 2>(g, part, part.band, part.bands, mail, sh, smem); break;
    case kBandSym: band_body<kBandSym, kRef, kBandThreads, 2>(g, part, part.band, part.bands, mail, sh, smem); break;
    case kBandNe: band_body<kBandNe, kRef, kBandThreads, 2>(g, part, part.band, part.bands, mail, sh, smem); break;
    case kBandGenFull: band_body<kBandGenFull, kRef, kBandThreads, 2>(g, part, part.band, part.bands, mail, sh, smem); break;
    case kBandSymFull: band_body<kBandSymFull, kRef, kBandThreads, 2>(g, part, part.band, part.bands, mail, sh, smem); break;
    default: band_body<kBandNeFull, kRef, kBandThreads, 2>(g, part, part.band, part.bands, mail, sh, smem); break;
    }
}

// kRefs: some lattice of the launch has a reference state.
template <bool kRefs>
__global__ void __launch_bounds__(kBandThreads, 1) k_band_batch(const Geom *geoms, const __grid_constant__ BandParts parts,
                                                                uint8_t *mail)
{
    extern __shared__ __align__(16) uint8_t band_smem[];
    __shared__ BandShared sh;
    __shared__ Geom sg;
    const BandPart &part = parts.p[blockIdx.x];
    if (threadIdx.x < sizeof(Geom) / 4)
        reinterpret_cast<uint32_t *>(&sg)[threadIdx.x] =
            reinterpret_cast<const uint32_t *>(&geoms[part.lat])[threadIdx.x];
    __syncthreads();
    if (kRefs && part.ref) band_any<kRefs>(sg, part, mail, sh, band_smem);
    else band_any<false>(sg, part, mail, sh, band_smem);
    band_end(sg, part, part.band, sh);
}

// Estimated us of n sweeps of a lattice on c CTAs: a half-sweep's exchange
// with the neighbours and its sites at an SM's rate (from L = 1024 .. 4096 on
// 152 SMs).
double band_time(const Geom &k, int kind, long long n, int c)
{
    // sites per us and SM: int8, bits
    double rate = 5.8e3;
    if (band_on_bits(k, kind, c)) rate = k.model == LAT_NE ? 20e3 : 8.5e3;
    return (double)n * 2.0 * (0.5 * (double)k.N / c / rate + 0.7);
}

}  // namespace

// The fewest CTAs that hold the lattice, 0 when it cannot run here.
int band_min_ctas(const Geom &g)
{
    const Geom k = tiled_geom(g);
    const int kind = band_kind(k, false);
    if (g.cpl != nullptr || kind >= kBandPacked || !band_kind_ok(g, kind)) return 0;
    const int most = std::min(band_sms(), g.L / 2);
    int lo = 1, hi = most;
    if (hi < 1 || !band_fits(k, kind, hi)) return 0;
    while (lo < hi) {   // fewer bands need more memory each
        const int mid = (lo + hi) / 2;
        if (band_fits(k, kind, mid)) hi = mid;
        else lo = mid + 1;
    }
    return lo;
}

// CTAs for each of the lattices so that the slowest finishes soonest;
// returns its estimated us (infinite: they do not fit together).
double band_share(const std::vector<std::pair<const Geom *, long long>> &lats, std::vector<int> &ctas)
{
    const int sms = band_sms();
    ctas.assign(lats.size(), 0);
    int used = 0;
    std::vector<Geom> k;
    std::vector<int> kind;
    for (size_t i = 0; i < lats.size(); ++i) {
        k.push_back(tiled_geom(*lats[i].first));
        kind.push_back(band_kind(k.back(), false));
        ctas[i] = band_min_ctas(*lats[i].first);
        if (ctas[i] == 0) return INFINITY;
        used += ctas[i];
    }
    if (used > sms) return INFINITY;
    for (;;) {   // a CTA more for the slowest while there is one and it helps
        size_t worst = 0;
        double t = -1.0;
        for (size_t i = 0; i < lats.size(); ++i) {
            const double ti = band_time(k[i], kind[i], lats[i].second, ctas[i]);
            if (ti > t) {
                t = ti;
                worst = i;
            }
        }
        if (used >= sms || ctas[worst] >= lats[worst].first->L / 2) return t;
        ++ctas[worst];
        ++used;
    }
}

size_t band_batch_mail_bytes(const std::vector<std::pair<const Geom *, long long>> &lats, const std::vector<int> &ctas)
{
    size_t pairs = 0;
    for (size_t i = 0; i < lats.size(); ++i) {
        const Geom k = tiled_geom(*lats[i].first);
        pairs += band_mail_pairs(k, band_kind(k, false), ctas[i]);
    }
    return kAbortBytes + pairs * sizeof(ulonglong2);
}

cudaError_t launch_batch_band(const Geom *d_geoms, const std::vector<std::pair<const Geom *, long long>> &lats,
                              const std::vector<unsigned long long> &sweep0, const std::vector<int *> &err,
                              int *err_all, const std::vector<int> &ctas, void *mail, unsigned epoch, cudaStream_t st)
{
    static PerDevice<cudaError_t> attrs;
    int dev = 0;
    cudaError_t attr = cudaGetDevice(&dev);
    if (attr != cudaSuccess) return attr;
    attr = attrs.get(dev, [] {
        cudaError_t bad = cudaSuccess;
        for (auto f : {k_band_batch<false>, k_band_batch<true>})
            if (bad == cudaSuccess)
                bad = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBandMaxSmem);
        return bad;
    });
    if (attr != cudaSuccess) return attr;
    if (band_test().launch()) return cudaErrorCooperativeLaunchTooLarge;
    auto parts = std::make_unique<BandParts>();
    const int mute = (int)band_test().mute.exchange(0) - 1;
    size_t smem = 0, pairs = 0;
    int cta = 0;
    for (size_t i = 0; i < lats.size(); ++i) {
        const Geom k = tiled_geom(*lats[i].first);
        BandPart p = band_part(k, sweep0[i], (int)lats[i].second, epoch, err[i]);
        p.err_all = err_all;
        p.bands = (uint32_t)ctas[i];
        p.lat = (uint32_t)i;
        p.kind = (uint32_t)band_kind(k, false);
        p.ref = k.ref != nullptr ? 1u : 0u;
        p.mail = (uint32_t)pairs;
        pairs += band_mail_pairs(k, (int)p.kind, ctas[i]);
        smem = std::max(smem, band_smem_bytes(k, (int)p.kind, ctas[i]));
        for (int b = 0; b < ctas[i]; ++b) {
            p.band = (uint32_t)b;
            parts->p[cta] = p;
            if (cta == mute) parts->p[cta].n = 0;   // it leaves its rows alone and sends nothing
            ++cta;
        }
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)cta);
    cfg.blockDim = dim3(kBandThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute a[1];
    a[0].id = cudaLaunchAttributeCooperative;
    a[0].val.cooperative = 1;
    cfg.attrs = a;
    cfg.numAttrs = 1;
    bool refs = false;
    for (const auto &l : lats) refs = refs || l.first->ref != nullptr;
    return cudaLaunchKernelEx(&cfg, refs ? k_band_batch<true> : k_band_batch<false>, d_geoms, *parts, (uint8_t *)mail);
}

}  // namespace lat
