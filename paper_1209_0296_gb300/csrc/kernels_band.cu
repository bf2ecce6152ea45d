// kernels_band.cu -- the band-resident kernel (band.cuh) of one lattice: a
// grid of one CTA per SM, all sweeps of a call in one cooperative launch.
#include <algorithm>
#include <mutex>

#include "band_kinds.cuh"

namespace lat {

namespace {

// One lattice over the whole grid.
template <int kKind, bool kRef>
__global__ void __launch_bounds__(kBandThreads, 1) k_band(const __grid_constant__ Geom g,
                                                          const __grid_constant__ BandPart part, uint8_t *mail)
{
    extern __shared__ __align__(16) uint8_t band_smem[];
    __shared__ BandShared sh;
    band_body<kKind, kRef>(g, part, blockIdx.x, gridDim.x, mail, sh, band_smem);
    band_end(g, part, blockIdx.x, sh);
}

}  // namespace

int band_sms()
{
    static const int sms = [] {
        int dev = 0, n = 0, coop = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
        return coop ? std::min(n, kBandMaxCtas) : 0;
    }();
    return sms;
}

int band_count_for(const Geom &g, bool fields)
{
    const Geom k = tiled_geom(g);
    const int kind = band_kind(k, fields), bands = std::min(band_sms(), g.L / 2);
    return bands >= 2 && band_kind_ok(g, kind) && band_fits(k, kind, bands) ? bands : 0;
}

size_t band_mail_bytes(const Geom &g, bool fields, int bands)
{
    const Geom k = tiled_geom(g);
    return kAbortBytes + band_mail_pairs(k, band_kind(k, fields), bands) * sizeof(ulonglong2);
}

cudaError_t launch_sweep_band(const Geom &g, bool fields, int bands, unsigned long long sweep0, int n, void *mail,
                              unsigned epoch, int *err, cudaStream_t st)
{
    using K = void (*)(Geom, BandPart, uint8_t *);
#define LAT_BAND(k) {k_band<k, false>, k_band<k, true>}
    static const K kern[kBandKinds][2] = {LAT_BAND(kBandGen),      LAT_BAND(kBandSym),     LAT_BAND(kBandNe),
                                          LAT_BAND(kBandGenFull),  LAT_BAND(kBandSymFull), LAT_BAND(kBandNeFull),
                                          LAT_BAND(kBandBondGen),  LAT_BAND(kBandBondSym), LAT_BAND(kBandFields),
                                          LAT_BAND(kBandPacked),   LAT_BAND(kBandPackedNe), LAT_BAND(kBandPotts3)};
#undef LAT_BAND
    static std::once_flag once;
    static cudaError_t attr = cudaSuccess;
    std::call_once(once, [] {
        for (const auto &row : kern)
            for (K f : row) {
                const cudaError_t e =
                    cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBandMaxSmem);
                if (e != cudaSuccess) attr = e;
            }
    });
    if (attr != cudaSuccess) return attr;
    const Geom k = tiled_geom(g);
    const BandPart part = band_part(k, sweep0, n, epoch, err);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)bands);
    // one chunk a thread: just the warps that have one (a row is a warp's when it fits)
    const int kind = band_kind(k, fields);
    const uint32_t nr = ((uint32_t)k.L + bands - 1) / bands, cpr = (k.half + 15) / 16;
    const bool small = kind < kBandPacked && band_is_small((uint32_t)k.L, k.half, (uint32_t)bands);
    cfg.blockDim = dim3(!small ? (uint32_t)kBandThreads
                               : std::max(64u, cpr <= 32 ? 32u * nr : (nr * cpr + 31u) / 32u * 32u));
    cfg.dynamicSmemBytes = band_smem_bytes(k, kind, bands);
    cfg.stream = st;
    cudaLaunchAttribute a[1];
    a[0].id = cudaLaunchAttributeCooperative;
    a[0].val.cooperative = 1;
    cfg.attrs = a;
    cfg.numAttrs = 1;
    const int ref = k.ref != nullptr || k.ref_bits != nullptr ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern[kind][ref], k, part, (uint8_t *)mail);
}

}  // namespace lat
