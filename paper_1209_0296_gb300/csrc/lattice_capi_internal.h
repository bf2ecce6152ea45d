// lattice_capi_internal.h -- host-side handle of one lattice and helpers
// shared by the C-ABI, batch and server translation units.
#pragma once

#include <atomic>
#include <string>
#include <vector>

#include "lattice_internal.cuh"

namespace lat {

struct Params {
    int dims, L, two_S, model, cmode, init, layout;
    double J, h, T, c;
    uint64_t seed;
    uint64_t N;
};

int cuda_fail(cudaError_t e, const char *what);
cudaError_t dev_alloc(void **p, size_t bytes, cudaStream_t st);
void dev_free(void *p, cudaStream_t st);
int validate(int dims, int L, int two_S, int model, double J, double h, double T_or_c, int init,
             int layout, Params &P);
void build_table(const Params &P, std::vector<TabEntry> &tab, int &dsmax, int &nmax, int &nn);
size_t footprint_bytes(const Params &P);
int create_impl(struct ::lattice **out, int dims, int L, int two_S, int model, double J, double h,
                double T_or_c, uint64_t seed, int init, int layout, void *cuda_stream);
int sweep_impl(struct ::lattice *lt, int64_t n);
int choose_kernel(const struct ::lattice *lt);
// While one lives, this thread's allocations and queries break no capture that
// the caller has going on another stream (in the global mode they would).
class BesideCapture {
public:
    BesideCapture() { cudaThreadExchangeStreamCaptureMode(&mode_); }
    ~BesideCapture() { cudaThreadExchangeStreamCaptureMode(&mode_); }
    BesideCapture(const BesideCapture &) = delete;
    BesideCapture &operator=(const BesideCapture &) = delete;

private:
    cudaStreamCaptureMode mode_ = cudaStreamCaptureModeRelaxed;
};
// A host-visible error word for band launches, zeroed (null: no memory), the
// owner's until it is given back; busy: launches on st may still write it.
int *band_error_word();
void band_error_word_back(int *w, cudaStream_t st, bool busy);
// Whether a bounded wait of an earlier launch gave up, as far as the host has
// seen (after a synchronise: all of them).
int band_status(const struct ::lattice *lt);
// Band launches of several streams.  A band launch takes every SM, so two of
// them must not wait for each other's, and work that would have run beside it
// waits.  A launch on one stream therefore never waits for another stream's
// band launch that may itself wait for something (it is refused, and its
// caller queues the two-launch sweeps, which run beside whatever there is); it
// does wait where that one was queued on an idle stream of its own and both
// lattices are large (or, less large, only two of them meet), which is sooner
// done than their launches side by side.  Otherwise both owners leave the
// bands alone for their next kBandYield calls: small lattices on streams of
// their own overlap their launches.  Launches side by side and bands in turn,
// ms: 16 x L = 256, 100 sweeps 1.0 and 3.7; 2 x L = 512 0.42 and 0.47; 2, 4, 8 x
// L = 1000 0.76 and 0.52, 0.98 and 1.02, 1.70 and 2.02; 4 x L = 2048, 20 sweeps
// 0.49 and 0.43.
struct BandShare {
    int yield = 0;   // calls that still do without bands
};
constexpr int kBandYield = 32;
constexpr uint64_t kBandLarge = 2000000, kBandTwo = 800000;   // sites from which bands in turn win, for any number and for two
// At the start of a call that could use bands on st: whether it may.
bool band_may(cudaStream_t st, BandShare *me);
// Whether work queued on st now would start when the GPU has room: st is idle,
// and no other stream's work is implicitly ordered before it (as a blocking
// stream's or the legacy stream's is).
bool idle_stream(cudaStream_t st);
// Before *me is freed.
void band_forget(BandShare *me);

// Lives while one band launch is queued on st.  No lock is held meanwhile (a
// launch waits on the host when the stream's queue is full): other threads'
// band launches are refused until it is.
class BandTurn {
public:
    // clear: the launch waits for no other work than this call's and bands like it.
    BandTurn(cudaStream_t st, BandShare *me, uint64_t sites, bool clear);
    ~BandTurn();
    bool go = false;      // launch (else: refused)
    cudaError_t status = cudaSuccess;

private:
    cudaStream_t st_;
    BandShare *me_;
    int dev_ = 0;
    unsigned long long id_ = 0;
    bool clear_;
    int depth_ = 0;
    uint64_t sites_;
};
int ensure_series(struct ::lattice *lt, unsigned long long need);
bool tile_shape_ok(int tile_w, int tile_h);
int default_tile_h();
void compact_table(Geom &g, const TabEntry *host_tab);

// Sweeps per captured CUDA graph: small lattices are launch-bound, so they
// replay long graphs; large ones need only a few sweeps per graph.
inline int default_graph_sweeps(const Params &P)
{
    if (P.N <= (1u << 16)) return 64;
    if (P.N <= (1u << 22)) return 16;
    return 8;
}

}  // namespace lat

struct lattice {
    lat::Params P;
    lat::Geom geom;
    cudaStream_t stream = nullptr;
    cudaStream_t cap_stream = nullptr;
    int8_t *spins[2] = {nullptr, nullptr};   // int8 layout: double buffer; bit-packed: [0] = staging
    uint8_t *flags = nullptr;      // North-East persistence bytes (see Geom)
    uint32_t *bits[2] = {nullptr, nullptr};
    lat::TabEntry *tab = nullptr;
    lat::Ctrl *ctrl = nullptr;
    // [series_cap][4] counters, then [series_cap] overlaps, then [series_cap] field sums
    unsigned long long *series = nullptr;
    unsigned long long series_cap = 0;   // sweeps the buffer can hold (from series_first)
    int8_t *ref = nullptr;               // reference state s(0), int8 planar layout
    uint32_t *ref_bits = nullptr;        // reference state s(0), bit-packed layout
    int64_t ref_sweep = -1;              // sweeps done when the reference was taken (-1: none)
    int dynamics = 0;                    // LAT_DYNAMICS_*
    int rs_tile = 0, rs_lambda = 0;      // random-site sub-lattice side and picks per round
    int8_t *rs_scratch = nullptr;        // random-site: output of the first launch of a sweep
    uint8_t *cpl = nullptr;              // per-site disorder bytes (see Geom::cpl); null when all zero
    std::vector<uint8_t> dis_host;       // host copy of the disorder bytes (empty: none set)
    bool has_bonds = false;              // coupling signs set
    bool has_fields = false;             // field signs set (the table then has a -h half)
    bool fields_wide_ok = false;         // the -h half suits the 2D wide kernel
    int64_t disorder_from = 0;           // sweeps done when the couplings or field signs last changed
    int64_t fields_from = 0;             // sweeps done when the field signs were last set
    unsigned long long *scratch4 = nullptr;
    std::vector<lat::TabEntry> host_tab;
    int64_t sweeps = 0;        // sweeps done (global index of the next sweep)
    bool captured = false;     // a caller captured sweeps of it: replays move the device's count alone
    int64_t series_first = 0;  // first sweep index recorded in the series buffer
    int64_t unfl_base = 0;     // unflipped sites before that sweep (North-East)
    int kernel = 0, tile_w = 0, tile_h = 0, graph_sweeps = 0;
    int tuned_kernel = 0;      // autotuner's choice for LAT_KERNEL_AUTO (0 = not tuned)
    bool graph_pinned = false; // sweeps per graph set by lattice_set_kernel (the tuner keeps it)
    cudaGraphExec_t graph_exec = nullptr;
    bool graph_valid = false;
    // band-resident sweeps (kernels_band.cu)
    void *band_mail = nullptr;           // boundary-row packets
    size_t band_mail_cap = 0;            // its bytes: the kinds of a lattice's life differ (disorder set or dropped)
    unsigned band_epoch = 0;             // at least every packet mark sent so far
    int *band_err = nullptr;             // host-visible word: a bounded wait gave up
    lat::BandShare band_share;
};
