// kernels_band.cu -- the band-resident kernel (band.cuh) of one lattice: a
// grid of one CTA per SM, all sweeps of a call in one cooperative launch.
#include <algorithm>

#include "band_host.h"
#include "band_kinds.cuh"

namespace lat {

namespace {

// One lattice over the whole grid. kForm as in band_body.
template <int kKind, bool kRef, int kT, int kForm>
__global__ void __launch_bounds__(kT, 1) k_band(const __grid_constant__ Geom g, const __grid_constant__ BandPart part,
                                                uint8_t *mail)
{
    extern __shared__ __align__(16) uint8_t band_smem[];
    __shared__ BandShared sh;
    band_body<kKind, kRef, kT, kForm>(g, part, blockIdx.x, gridDim.x, mail, sh, band_smem);
    band_end(g, part, blockIdx.x, sh);
}

using BandKernel = void (*)(Geom, BandPart, uint8_t *);

// Kernels of a kind by reference set and form: small bands, the others, and
// for North-East the others with more threads.
template <int kKind, bool kRef, int kVar>
constexpr BandKernel band_kernel()
{
    constexpr bool kNe = kKind == kBandNe || kKind == kBandNeFull || kKind == kBandPackedNe;
    // on bits a partial last chunk makes no difference
    constexpr int kBits = kKind == kBandSym ? kBandSymFull : kKind == kBandNe ? kBandNeFull : kKind;
    if constexpr (kVar == 0) {
        if constexpr (kKind >= kBandPacked) return nullptr;
        else return k_band<kKind, kRef, kBandThreads, 0>;
    } else if constexpr (kVar == 1) {
        return k_band<kBits, kRef, kBandThreads, 1>;
    } else {
        if constexpr (kNe) return k_band<kBits, kRef, kBandNeThreads, 1>;
        else return nullptr;
    }
}

}  // namespace

BandTest &band_test()
{
    static BandTest t;
    return t;
}

int band_sms()
{
    static PerDevice<int> sms;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    return sms.get(dev, [dev] {
        int n = 0, coop = 0;
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
        return coop ? std::min(n, kBandMaxCtas) : 0;
    });
}

int band_count_for(const Geom &g, bool fields)
{
    const Geom k = tiled_geom(g);
    const int kind = band_kind(k, fields), bands = std::min(band_sms(), g.L / 2);
    return bands >= 2 && band_kind_ok(g, kind) && band_fits(k, kind, bands) ? bands : 0;
}

int band_chunk_load(const Geom &g, bool fields)
{
    const Geom k = tiled_geom(g);
    const int kind = band_kind(k, fields), bands = std::min(band_sms(), g.L / 2);
    if (bands < 2 || band_on_bits(k, kind, bands) || band_is_small((uint32_t)k.L, k.half, (uint32_t)bands)) return 0;
    return (int)((uint64_t)((k.L + bands - 1) / bands) * ((k.half + 15) / 16) * 100 / kBandThreads);
}

size_t band_mail_bytes(const Geom &g, bool fields, int bands)
{
    const Geom k = tiled_geom(g);
    return kAbortBytes + band_mail_pairs(k, band_kind(k, fields), bands) * sizeof(ulonglong2);
}

cudaError_t launch_sweep_band(const Geom &g, bool fields, int bands, unsigned long long sweep0, int n, void *mail,
                              unsigned epoch, int *err, cudaStream_t st)
{
#define LAT_VAR(k, ref) {band_kernel<k, ref, 0>(), band_kernel<k, ref, 1>(), band_kernel<k, ref, 2>()}
#define LAT_BAND(k) {LAT_VAR(k, false), LAT_VAR(k, true)}
    static const BandKernel kern[kBandKinds][2][3] = {
        LAT_BAND(kBandGen),     LAT_BAND(kBandSym),     LAT_BAND(kBandNe),     LAT_BAND(kBandGenFull),
        LAT_BAND(kBandSymFull), LAT_BAND(kBandNeFull),  LAT_BAND(kBandBondGen), LAT_BAND(kBandBondSym),
        LAT_BAND(kBandFields),  LAT_BAND(kBandPacked),  LAT_BAND(kBandPackedNe), LAT_BAND(kBandPotts3)};
#undef LAT_BAND
#undef LAT_VAR
    static PerDevice<cudaError_t> attrs;
    int dev = 0;
    cudaError_t attr = cudaGetDevice(&dev);
    if (attr != cudaSuccess) return attr;
    attr = attrs.get(dev, [] {
        cudaError_t bad = cudaSuccess;
        for (const auto &kind : kern)
            for (const auto &ref : kind)
                for (BandKernel f : ref) {
                    const cudaError_t e = f == nullptr ? cudaSuccess
                                                       : cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                                              (int)kBandMaxSmem);
                    if (e != cudaSuccess) bad = e;
                }
        return bad;
    });
    if (attr != cudaSuccess) return attr;
    if (band_test().launch()) return cudaErrorCooperativeLaunchTooLarge;
    const Geom k = tiled_geom(g);
    const BandPart part = band_part(k, sweep0, n, epoch, err);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)bands);
    // one chunk a thread: just the warps that have one (a row is a warp's when it fits)
    const int kind = band_kind(k, fields);
    const uint32_t nr = ((uint32_t)k.L + bands - 1) / bands, cpr = (k.half + 15) / 16;
    const bool small = kind < kBandPacked && band_is_small((uint32_t)k.L, k.half, (uint32_t)bands);
    // North-East waits on shared memory and warp scans more than on a pipe: bands
    // of several words a thread run with twice the threads, where their queues
    // fit (L = 8192, c = 0.3: 38.7 us a sweep with 512 threads, 32.0 with 768,
    // 31.5 with 1024; 4096: 12.1, 11.3, 10.0; at L = 2048 the idle warps cost: 4.6,
    // 4.9, 5.0)
    const bool more = !small && nr * ((k.half + 31u) / 32u) > 1024u && (kind == kBandNe || kind == kBandNeFull || kind == kBandPackedNe) &&
                      band_smem_bytes(k, kind, bands, kBandNeThreads) <= kBandMaxSmem;
    const int threads = more ? kBandNeThreads : kBandThreads;
    cfg.blockDim = dim3(!small ? (uint32_t)threads
                               : std::max(64u, cpr <= 32 ? 32u * nr : (nr * cpr + 31u) / 32u * 32u));
    cfg.dynamicSmemBytes = band_smem_bytes(k, kind, bands, threads);
    cfg.stream = st;
    cudaLaunchAttribute a[1];
    a[0].id = cudaLaunchAttributeCooperative;
    a[0].val.cooperative = 1;
    cfg.attrs = a;
    cfg.numAttrs = 1;
    const int ref = k.ref != nullptr || k.ref_bits != nullptr ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern[kind][ref][small ? 0 : more ? 2 : 1], k, part, (uint8_t *)mail);
}

}  // namespace lat
