// kernels_band.cu -- the band-resident kernel (band.cuh) of one lattice: a
// grid of one CTA per SM, all sweeps of a call in one cooperative launch.
#include <algorithm>
#include <mutex>

#include "band.cuh"
#include "bits_step.cuh"

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

// Bit-packed Ising with a symmetric table: the same bands and packets (one
// 64-bit packet a word) on words of 32 sites.
template <bool kRef>
__global__ void __launch_bounds__(kBandThreads, 1) k_band_bits(const __grid_constant__ Geom g,
                                                               const __grid_constant__ BandPart part, uint8_t *mail)
{
    extern __shared__ __align__(16) uint8_t band_smem[];
    __shared__ BandShared sh;
    const uint32_t tid = threadIdx.x, L = (uint32_t)g.L, bw = g.bw, band = blockIdx.x, bands = gridDim.x;
    uint32_t y0, y1;
    band_rows(band, bands, L, y0, y1);
    const uint32_t nr = y1 - y0, pw = nr * bw, rend = nr - 1u;
    uint32_t *sm = reinterpret_cast<uint32_t *>(band_smem);
    const uint32_t *src = g.bits[part.sweep0 & 1];
    for (uint32_t c = 0; c < 2u; ++c)
        for (uint32_t i = tid; i < pw; i += kBandThreads) sm[c * pw + i] = src[((size_t)c * L + y0) * bw + i];
    if (tid < 10) (&sh.sum[0][0])[tid] = 0;
    if (tid == 10) sh.bad = 0;
    __syncthreads();
    // packets: [band][first, last row][colour][word]
    unsigned *abort = reinterpret_cast<unsigned *>(mail);
    unsigned long long *m = reinterpret_cast<unsigned long long *>(mail + kAbortBytes);
    unsigned long long *first = m + (size_t)band * 4u * bw, *last_row = first + 2u * bw;
    const unsigned long long *above = m + (size_t)(band == 0u ? bands - 1u : band - 1u) * 4u * bw + 2u * bw;
    const unsigned long long *below = m + (size_t)(band + 1u == bands ? 0u : band + 1u) * 4u * bw;
    const uint32_t up = y0 == 0u ? L - 1u : y0 - 1u, dn = y1 == L ? 0u : y1;
    const SymK sk = bits_sym(g.thr16);
    const uint32_t rsb = (uint32_t)kBandThreads / bw, rr = tid / bw, k = tid - rr * bw;
    const uint32_t r0 = rr < rsb ? 1u + rr : nr, edge0 = (uint32_t)kBandThreads - 1u - tid, edges = 2u * bw;
    Counts cnt;
    int bad = 0, words = 0;
    for (int h = 0; h < 2 * part.n; ++h) {
        const uint32_t colour = (uint32_t)h & 1u;
        const unsigned long long sweep = part.sweep0 + (unsigned long long)(h >> 1);
        PhiloxPre pp;
        philox_prepare(pp, (uint32_t)sweep, (uint32_t)(sweep >> 32), part.key0, part.key1);
        uint32_t *mine = sm + colour * pw;
        const uint32_t *other = sm + (1u - colour) * pw;
        auto word = [&](uint32_t r, uint32_t c, uint32_t U, uint32_t D) {
            const uint32_t at = r * bw + c, y = y0 + r, O = other[at], S = mine[at];
            const bool odd = ((colour + y) & 1u) != 0u;
            const uint32_t cn = odd ? (c + 1u == bw ? 0u : c + 1u) : (c == 0u ? bw - 1u : c - 1u);
            const Nbr n = nbr_sum(U, D, O, bits_shifted(odd, O, other[r * bw + cn]));
            const uint32_t Sn = bits_step(sk, g.thr16, pp, sweep, part.key0, part.key1, y * g.G + 8u * c, colour, n, S);
            mine[at] = Sn;
            if (colour == 1u) {
                cnt.bond -= 2 * bits_unlike(n, Sn);
                cnt.mag += __popc(Sn) + __popc(O);   // up spins
                if constexpr (kRef)
                    cnt.acf -= 2 * (__popc(Sn ^ g.ref_bits[((size_t)L + y) * bw + c]) +
                                    __popc(O ^ g.ref_bits[(size_t)y * bw + c]));
                ++words;
            }
            return Sn;
        };
#pragma unroll 1
        for (uint32_t r = r0; r < rend; r += rsb) word(r, k, other[(r - 1u) * bw + k], other[(r + 1u) * bw + k]);
#pragma unroll 1
        for (uint32_t e = edge0; e < edges; e += (uint32_t)kBandThreads) {
            const bool lo = e < bw;   // the last row's words, then the first row's
            const uint32_t c = lo ? e : e - bw, r = lo ? rend : 0u;
            const unsigned long long *box = (lo ? below : above) + (1u - colour) * bw + c;
            uint32_t far;
            if (h == 0) far = src[((size_t)(1u - colour) * L + (lo ? dn : up)) * bw + c];
            else if (!mail_take_word(box, part.epoch + (uint32_t)h, abort, far)) bad = 1;
            const uint32_t near = other[(lo ? r - 1u : 1u) * bw + c];
            const uint32_t Sn = word(r, c, lo ? near : far, lo ? far : near);
            mail_put_word((lo ? last_row : first) + colour * bw + c, part.epoch + (uint32_t)h + 1u, Sn);
        }
        if (colour == 1u) {
            const int ups = cnt.mag;
            cnt.bond += 128 * words;
            cnt.acf += 64 * words;
            cnt.up = ups;
            cnt.mag = 2 * ups - 64 * words;
            band_count(sh, h >> 1 & 1, cnt, false, kRef);
            cnt = Counts();
            words = 0;
        }
        const int stop = __syncthreads_or(bad);
        if (colour == 1u) band_post(sh, h >> 1 & 1, g, sweep, false, kRef);
        if (stop) {
            sh.bad = 1;
            break;
        }
    }
    uint32_t *fin = g.bits[(part.sweep0 + (unsigned long long)part.n) & 1];
    for (uint32_t c = 0; c < 2u; ++c)
        for (uint32_t i = tid; i < pw; i += kBandThreads) fin[((size_t)c * L + y0) * bw + i] = sm[c * pw + i];
    band_end(g, part, band, sh);
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

static int band_count_bits(const Geom &g);

int band_count_for(const Geom &g)
{
    if (g.bits[0] != nullptr) return band_count_bits(g);
    const bool kind_ok = g.model == LAT_NE ? ne_walk_supported(g) : (g.cpl == nullptr ? any_supported(g) : wide_supported(g));
    if (!kind_ok || (g.half + 15) / 16 > (uint32_t)kBandThreads) return 0;
    const int bands = std::min(band_sms(), g.L / 2);
    return bands >= 2 && band_smem_bytes(g, bands) <= kBandMaxSmem ? bands : 0;
}

// The same for bit-packed lattices.
static int band_count_bits(const Geom &g)
{
    if (g.model != LAT_ISING || !bitpacked_supported(g) || !tiled_geom(g).acc_sym || g.bw > (uint32_t)kBandThreads) return 0;
    const int bands = std::min(band_sms(), g.L / 2);
    const size_t smem = (size_t)2 * ((g.L + bands - 1) / bands) * g.bw * 4;
    return bands >= 2 && smem <= kBandMaxSmem ? bands : 0;
}

size_t band_mail_bytes(const Geom &g, int bands)
{
    if (g.bits[0] != nullptr) return kAbortBytes + (size_t)bands * 4 * g.bw * sizeof(unsigned long long);
    return kAbortBytes + band_mail_pairs(g, bands) * sizeof(ulonglong2);
}

cudaError_t launch_sweep_band(const Geom &g, bool fields, int bands, unsigned long long sweep0, int n, void *mail,
                              unsigned epoch, int *err, cudaStream_t st)
{
    using K = void (*)(Geom, BandPart, uint8_t *);
#define LAT_BAND(k) {k_band<k, false>, k_band<k, true>}
    static const K kern[kBandKinds][2] = {LAT_BAND(kBandGen),     LAT_BAND(kBandSym),     LAT_BAND(kBandNe),
                                          LAT_BAND(kBandGenFull), LAT_BAND(kBandSymFull), LAT_BAND(kBandNeFull),
                                          LAT_BAND(kBandBondGen), LAT_BAND(kBandBondSym), LAT_BAND(kBandFields)};
#undef LAT_BAND
    static const K bits[2] = {k_band_bits<false>, k_band_bits<true>};
    static std::once_flag once;
    static cudaError_t attr = cudaSuccess;
    std::call_once(once, [] {
        for (K f : bits) {
            const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBandMaxSmem);
            if (e != cudaSuccess) attr = e;
        }
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
    const uint32_t nr = ((uint32_t)k.L + bands - 1) / bands, cpr = (k.half + 15) / 16;
    const bool small = band_is_small((uint32_t)k.L, k.half, (uint32_t)bands);
    cfg.blockDim = dim3(!small ? (uint32_t)kBandThreads
                               : std::max(64u, cpr <= 32 ? 32u * nr : (nr * cpr + 31u) / 32u * 32u));
    const bool packed = k.bits[0] != nullptr;
    if (packed) cfg.blockDim = dim3(kBandThreads);
    cfg.dynamicSmemBytes = packed ? (size_t)2 * nr * k.bw * 4 : band_smem_bytes(k, bands);
    cfg.stream = st;
    cudaLaunchAttribute a[1];
    a[0].id = cudaLaunchAttributeCooperative;
    a[0].val.cooperative = 1;
    cfg.attrs = a;
    cfg.numAttrs = 1;
    if (packed) return cudaLaunchKernelEx(&cfg, bits[k.ref_bits != nullptr ? 1 : 0], k, part, (uint8_t *)mail);
    return cudaLaunchKernelEx(&cfg, kern[band_kind(k, fields)][k.ref != nullptr ? 1 : 0], k, part, (uint8_t *)mail);
}

}  // namespace lat
