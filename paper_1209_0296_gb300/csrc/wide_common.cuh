// wide_common.cuh -- pieces shared by the 2D spin-1/2 kernels that give a
// thread 16 consecutive sites of a plane row (kernels_wide.cu,
// kernels_ne.cu): 16-site loads and stores at any alignment, counter
// reduction, the split of rows into bands.
#pragma once

#include <algorithm>

#include "lattice_internal.cuh"

#if defined(__CUDACC__)
namespace lat {
namespace {

constexpr int kThreads = 256;

struct Counts {
    int bond = 0, mag = 0, up = 0, unfl = 0, acf = 0, fld = 0;
};

// W consecutive 4-byte words (4W same-colour sites) from p.
template <int W>
LAT_D void load_words(const int8_t *p, uint32_t (&v)[W])
{
    if constexpr (W == 4) {
        const uint4 q = *reinterpret_cast<const uint4 *>(p);
        v[0] = q.x;
        v[1] = q.y;
        v[2] = q.z;
        v[3] = q.w;
    } else if constexpr (W == 2) {
        const uint2 q = *reinterpret_cast<const uint2 *>(p);
        v[0] = q.x;
        v[1] = q.y;
    } else {
        v[0] = *reinterpret_cast<const uint32_t *>(p);
    }
}

template <int W>
LAT_D void store_words(int8_t *p, const uint32_t (&v)[W])
{
    if constexpr (W == 4) *reinterpret_cast<uint4 *>(p) = make_uint4(v[0], v[1], v[2], v[3]);
    else if constexpr (W == 2) *reinterpret_cast<uint2 *>(p) = make_uint2(v[0], v[1]);
    else *reinterpret_cast<uint32_t *>(p) = v[0];
}

// Add the block's counters to the sweep's slot (bond, mag, up[, unflipped]).
// Warp sums go to shared memory and warp 0 adds them up.  32-bit partial
// sums are enough: a block's |bond| is at most 2 per site it updated, and a
// block never updates 2^30 sites in one call.
// acf: the sweep's autocorrelation slot, or null when no reference is set.
LAT_D void flush_slot(unsigned long long *slot, unsigned long long *acf, const Counts &c, bool ne,
                      int (*red)[5])
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rb = __reduce_add_sync(0xffffffffu, c.bond);
    const int rm = __reduce_add_sync(0xffffffffu, c.mag);
    const int ru = __reduce_add_sync(0xffffffffu, c.up);
    const int rf = __reduce_add_sync(0xffffffffu, c.unfl);
    const int ra = acf ? __reduce_add_sync(0xffffffffu, c.acf) : 0;
    if (lane == 0) {
        red[warp][0] = rb;
        red[warp][1] = rm;
        red[warp][2] = ru;
        red[warp][3] = rf;
        red[warp][4] = ra;
    }
    __syncthreads();
    if (warp == 0) {
        const bool in = lane < (int)(blockDim.x >> 5);
        const int b = __reduce_add_sync(0xffffffffu, in ? red[lane][0] : 0);
        const int m = __reduce_add_sync(0xffffffffu, in ? red[lane][1] : 0);
        const int u = __reduce_add_sync(0xffffffffu, in ? red[lane][2] : 0);
        const int f = __reduce_add_sync(0xffffffffu, in ? red[lane][3] : 0);
        if (lane < (ne ? 4 : 3)) add_counter(slot + lane, (long long)(lane == 0 ? b : lane == 1 ? m : lane == 2 ? u : f));
        if (acf) {
            const int a = __reduce_add_sync(0xffffffffu, in ? red[lane][4] : 0);
            if (lane == 0) add_counter(acf, (long long)a);
        }
    }
    __syncthreads();
}

LAT_D void flush(const SweepView &g, unsigned long long sweep, const Counts &c, bool ne, int (*red)[5])
{
    flush_slot(series_slot(g.ctrl, sweep), g.ref ? acf_slot(g.ctrl, sweep) : nullptr, c, ne, red);
}

// Add one int per thread, summed over the block, to *dst (all threads call).
LAT_D void flush_one(unsigned long long *dst, int v, int (*red)[5])
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int r = __reduce_add_sync(0xffffffffu, v);
    if (lane == 0) red[warp][0] = r;
    __syncthreads();
    if (warp == 0) {
        const int t = __reduce_add_sync(0xffffffffu, lane < (int)(blockDim.x >> 5) ? red[lane][0] : 0);
        if (lane == 0) add_counter(dst, (long long)t);
    }
    __syncthreads();
}

// Rows [y0, y1) of band b of nb bands of L rows: their lengths differ by at
// most one, long and short ones in turn.
LAT_D void band_rows(uint32_t b, uint32_t nb, uint32_t L, uint32_t &y0, uint32_t &y1)
{
    y0 = (uint32_t)((uint64_t)b * L / nb);
    y1 = (uint32_t)((uint64_t)(b + 1u) * L / nb);
}

// The same for the threads of a streaming launch: where bands are short the
// long ones come first.  (In turn with the others every warp takes the longer
// time: L = 2400, two rows or three, 10.7 us a sweep for 9.2.  Many rows apart,
// equal lengths make bands meet in the same memory channels: bit-packed L =
// 32768, 143 rows or 144, 834 us for 810.)
LAT_D void walk_rows(uint32_t b, uint32_t nb, uint32_t L, uint32_t &y0, uint32_t &y1)
{
    const uint32_t q = L / nb, r = L - q * nb;
    if (q >= 32u) {
        band_rows(b, nb, L, y0, y1);
        return;
    }
    y0 = b * q + min(b, r);
    y1 = y0 + q + (b < r ? 1u : 0u);
}

// Bytes p[0 .. nv) (1 <= nv <= 16) as four words, byte b = p[b], the bytes
// from nv on unspecified; an aligned word that holds none of them is not
// read (the spin buffers are multiples of 4 bytes, so every word read is in
// bounds).  kAligned: p is 16-byte aligned and nv = 16 (every chunk of a
// lattice with L % 32 == 0), one 16-byte load.
template <bool kAligned = false>
LAT_D void load16_any(const int8_t *p, uint32_t nv, uint32_t (&v)[4])
{
    if constexpr (kAligned) {
        load_words<4>(p, v);
        return;
    }
    const uintptr_t a = reinterpret_cast<uintptr_t>(p);
    const uint32_t sh = (uint32_t)(a & 3u);
    const uint32_t *w = reinterpret_cast<const uint32_t *>(a - sh);
    uint32_t x[5];
    x[0] = w[0];
#pragma unroll
    for (int i = 1; i < 5; ++i) x[i] = (4u * (uint32_t)i < nv + sh) ? w[i] : 0u;
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = __funnelshift_r(x[i], x[i + 1], 8u * sh);
}

// Write bytes [0, nv) of v to p (any alignment) and no other byte: whole
// aligned words where the chunk covers them, single bytes at its ends.
template <bool kAligned = false>
LAT_D void store16_any(int8_t *p, uint32_t nv, const uint32_t (&v)[4])
{
    if constexpr (kAligned) {
        store_words<4>(p, v);
        return;
    }
    const uintptr_t a = reinterpret_cast<uintptr_t>(p);
    const uint32_t sh = (uint32_t)(a & 3u);
    uint32_t *w = reinterpret_cast<uint32_t *>(a - sh);
    uint32_t o[5];   // o[i]: the chunk's bytes that fall in aligned word i
    o[0] = __funnelshift_l(0u, v[0], 8u * sh);
#pragma unroll
    for (int i = 1; i < 4; ++i) o[i] = __funnelshift_l(v[i - 1], v[i], 8u * sh);
    o[4] = __funnelshift_l(v[3], 0u, 8u * sh);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const int lo = i == 0 ? (int)sh : 0;
        const int hi = min(4, (int)(nv + sh) - 4 * i);
        if (hi <= lo) continue;
        if (lo == 0 && hi == 4) {
            w[i] = o[i];
        } else {
            int8_t *pb = reinterpret_cast<int8_t *>(w + i);
            for (int j = lo; j < hi; ++j) pb[j] = (int8_t)(o[i] >> (8 * j));
        }
    }
}

struct AnyItemShape {
    uint32_t cpr, nseg, rsb, br;   // chunks per row, column segments, rows per pass, rows per band
};

// Rows a thread visits per item (passes): given by the batch (its tuner),
// or 0 for the default: 8 on large lattices (few items, long pipelines), 2
// on small ones (enough items to spread a batch of small lattices over the
// SMs).
LAT_HD AnyItemShape any_item_shape(uint32_t half, uint32_t passes)
{
    AnyItemShape sh;
    sh.cpr = (half + 15u) >> 4;
    sh.nseg = (sh.cpr + kThreads - 1u) / kThreads;
    sh.rsb = sh.cpr <= (uint32_t)kThreads ? (uint32_t)kThreads / sh.cpr : 1u;
    if (passes == 0u) passes = half >= 512u ? 8u : 2u;
    sh.br = passes * sh.rsb;
    return sh;
}

// A chunk's 16 bytes at any alignment: its aligned words as loaded, shifted
// into place when they are used.
template <bool kAligned>
struct Row16 {
    uint32_t x[kAligned ? 4 : 5];
};

template <bool kAligned>
LAT_D void row_load(const int8_t *q, uint32_t nv, Row16<kAligned> &r)
{
    if constexpr (kAligned) {
        load_words<4>(q, r.x);
    } else {
        const uintptr_t a = reinterpret_cast<uintptr_t>(q);
        const uint32_t sh = (uint32_t)(a & 3u);
        const uint32_t *w = reinterpret_cast<const uint32_t *>(a - sh);
        r.x[0] = w[0];
#pragma unroll
        for (int i = 1; i < 5; ++i) r.x[i] = (4u * (uint32_t)i < nv + sh) ? w[i] : 0u;
    }
}

template <bool kAligned>
LAT_D void row_words(const int8_t *q, const Row16<kAligned> &r, uint32_t (&v)[4])
{
    if constexpr (kAligned) {
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = r.x[i];
    } else {
        const uint32_t sh = 8u * (uint32_t)(reinterpret_cast<uintptr_t>(q) & 3u);
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = __funnelshift_r(r.x[i], r.x[i + 1], sh);
    }
}

// The chunk column's share of a row: valid sites, masks of the valid bytes,
// and the row index of the other plane's site before the chunk and after it.
template <bool kAligned>
struct ChunkCol {
    uint32_t j0, nv, vm[4], jp, jn;
};

template <bool kAligned>
LAT_D ChunkCol<kAligned> chunk_col(uint32_t k, uint32_t half)
{
    ChunkCol<kAligned> c;
    c.j0 = 16u * k;
    c.nv = kAligned ? 16u : min(16u, half - c.j0);
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        const int n = (int)c.nv - 4 * w;
        c.vm[w] = kAligned || n >= 4 ? 0xFFFFFFFFu : (n <= 0 ? 0u : (1u << (8 * n)) - 1u);
    }
    c.jp = c.j0 == 0u ? half - 1u : c.j0 - 1u;
    c.jn = c.j0 + c.nv == half ? 0u : c.j0 + c.nv;
    return c;
}

// The side neighbour that is not at the same index: the other plane's row
// shifted one site west (odd: x = 2j + 1, towards j + 1) or east, nb being
// the byte past the chunk's end on that side.
template <bool kAligned>
LAT_D void shifted_row(const ChunkCol<kAligned> &c, bool odd, uint32_t nb, const uint32_t (&O)[4], uint32_t (&X)[4])
{
    if (odd) {
        uint32_t T[4];
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            T[w] = O[w];
            if constexpr (!kAligned) {   // the byte after a partial chunk's last site
                const uint32_t d = c.nv - 4u * (uint32_t)w, m = d < 4u ? 0xFFu << (8u * d) : 0u;
                T[w] = (T[w] & ~m) | ((nb * 0x01010101u) & m);
            }
        }
#pragma unroll
        for (int w = 0; w < 4; ++w) X[w] = __funnelshift_r(T[w], w == 3 ? nb : T[w + 1], 8);
    } else {
#pragma unroll
        for (int w = 0; w < 4; ++w) X[w] = __funnelshift_l(w == 0 ? nb << 24 : O[w - 1], O[w], 8);
    }
}

// SMs x resident CTAs of a kernel on the current device.
unsigned one_wave(const void *fn)
{
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, kThreads, 0);
    return (unsigned)(sms * (per > 0 ? per : 1));
}

}  // namespace
}  // namespace lat
#endif
