// Cell binning (the (cell, id) particle sort) for callers that cannot
// allocate device memory.
//
// Some callers must not allocate GPU memory while they run: code that is
// being recorded into a CUDA graph (cudaMalloc is not a stream operation and
// cannot be captured), real-time loops where cudaMalloc/cudaFree would
// introduce an implicit device synchronisation, and hosts that own a fixed
// device-memory budget and hand libraries only the buffers they asked for.
// lbdps_bin_sort_noalloc serves them: the caller passes the positions and the
// two output buffers, and every temporary this sort needs lives in one
// file-scope device array of fixed size that is created when the library is
// loaded on a GPU and kept until the process exits.
#include "lbdps.h"
#include "lbdps_internal.cuh"

#include <algorithm>
#include <cstdio>
#include <mutex>

namespace lbdpsk {
void set_last_error(const char *msg);
}

namespace {

constexpr int kMaxCells = 1 << 20;       // lattice cells per call
constexpr int kMaxParticles = 1 << 20;   // particles per call
// Stable radix sort of the cell keys.  Digits of up to 10 bits: every key of
// up to 2^20 cells takes at most two passes (three of 8 bits before).  A tile
// is one block of 1,024 threads, a particle each; the histograms are
// digit-major (entry d tiles + tile).
constexpr int kRadixBits = 10;
constexpr int kBins = 1 << kRadixBits;
constexpr int kTile = 1024;
constexpr int kTileWarps = kTile / 32;
constexpr int kMaxHist = kBins * (kMaxParticles / kTile);
// prefix sums: tiles of 4,096 entries and the sums of the tiles before
constexpr int kScanLog2 = 12;
constexpr int kScanTile = 1 << kScanLog2;
constexpr int kMaxScanTiles = kMaxCells / kScanTile + 1;   // of ncell + 1 counts
static_assert(kMaxHist <= kMaxCells && kMaxScanTiles <= kTile, "one block adds up the tiles");
constexpr size_t kCountInts = (size_t)kMaxCells + 4 + kMaxHist;   // counts, then the second digit's histogram
constexpr size_t kScratchInts = kCountInts + (size_t)kMaxHist      // first digit's histogram
                                + 3 * (size_t)kMaxParticles        // keys; keys and ids after a pass
                                + 4 * (size_t)kMaxScanTiles + 64;
constexpr int kMaxDevices = 64;

}  // namespace

// counts and second histogram | first histogram | keys | keys A | ids A | tile sums | tickets
static __device__ __align__(256) int g_bin_scratch[kScratchInts];

namespace {

std::mutex g_setup_mutex;
int *g_scratch_ptr[kMaxDevices] = {};

// An array of n counts, replaced by its exclusive prefix inside each tile of
// kScanTile entries, and the exclusive prefix of the tile sums: the prefix at e
// is data[e] + base[e >> kScanLog2].
struct Prefix {
    int *data;
    int n;
    int *tile_sum, *base;
    unsigned *ticket;   // zero between launches
    __host__ __device__ int tiles() const { return (n + kScanTile - 1) >> kScanLog2; }
    __device__ int at(int e) const { return __ldg(data + e) + __ldg(base + (e >> kScanLog2)); }
};

// Block-wide exclusive scan of one value per thread (kTile threads).
__device__ __forceinline__ int block_scan(int v, int *warp_tot, int *total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) warp_tot[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        const int w = warp_tot[lane];
        int wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += t;
        }
        warp_tot[lane] = wi - w;
        if (lane == 31) *total = wi;
    }
    __syncthreads();
    return warp_tot[warp] + inc - v;
}

// Prefix sums of one or two arrays in one launch: a block per tile, a's tiles
// first; the block of an array that finishes last (ticket, nothing waits) adds
// up its tile sums.
__global__ void __launch_bounds__(kTile) k_na_prefix(Prefix a, Prefix b)
{
    __shared__ int warp_tot[32];
    __shared__ int total;
    __shared__ bool last;
    const int nta = a.tiles();
    const bool first = (int)blockIdx.x < nta;
    const Prefix &s = first ? a : b;
    const int tile = first ? blockIdx.x : blockIdx.x - nta, nt = s.tiles();
    const int e = tile * kScanTile + 4 * (int)threadIdx.x;
    int4 c = make_int4(0, 0, 0, 0);
    if (e + 4 <= s.n) c = *reinterpret_cast<const int4 *>(s.data + e);
    else {
        if (e < s.n) c.x = s.data[e];
        if (e + 1 < s.n) c.y = s.data[e + 1];
        if (e + 2 < s.n) c.z = s.data[e + 2];
    }
    const int run = block_scan(c.x + c.y + c.z + c.w, warp_tot, &total);
    const int4 r = make_int4(run, run + c.x, run + c.x + c.y, run + c.x + c.y + c.z);
    if (e + 4 <= s.n) *reinterpret_cast<int4 *>(s.data + e) = r;
    else {
        if (e < s.n) s.data[e] = r.x;
        if (e + 1 < s.n) s.data[e + 1] = r.y;
        if (e + 2 < s.n) s.data[e + 2] = r.z;
    }
    if (threadIdx.x == 0) {
        s.tile_sum[tile] = total;
        __threadfence();
        last = atomicAdd(s.ticket, 1u) == (unsigned)nt - 1u;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int v = (int)threadIdx.x < nt ? __ldcg(s.tile_sum + threadIdx.x) : 0;
    const int ex = block_scan(v, warp_tot, &total);
    if ((int)threadIdx.x < nt) s.base[threadIdx.x] = ex;
    if (threadIdx.x == 0) *s.ticket = 0u;
}

// Cell key of each particle, the per-cell counts and the first digit's tile
// histogram.  Each coordinate is clamped in FP64 before any conversion: below 0
// (or NaN) to the first cell, at or above n[a] to the last, so the integer cast
// only sees [0, n[a]).
__global__ void __launch_bounds__(kTile)
k_na_keys(int dim, int n0, int n1, int n2, const double *P0, const double *P1, const double *P2, int np,
          int *key, int *counts, int bins, int tiles, int *hist)
{
    __shared__ int cnt[kBins];
    cnt[threadIdx.x] = 0;
    __syncthreads();
    const int k = blockIdx.x * kTile + threadIdx.x;
    int d = kBins, c = -1;
    if (k < np) {
        const int n[3] = {n0, n1, n2};
        const double *P[3] = {P0, P1, P2};
        int q[3] = {0, 0, 0};
        for (int a = 0; a < dim; ++a) {
            const double x = P[a][k];
            int v = 0;
            if (x >= 0.0) v = x < (double)n[a] ? (int)x : n[a] - 1;
            q[a] = v;
        }
        c = q[0] + n0 * (q[1] + n1 * q[2]);
        key[k] = c;
        d = c & (bins - 1);
    }
    // one atomic per warp and cell (digit): a crowded cell costs a warp one
    const unsigned mates = __match_any_sync(0xffffffffu, c);
    if (c >= 0 && (int)(threadIdx.x & 31) == __ffs(mates) - 1) atomicAdd(&counts[c], __popc(mates));
    const unsigned same = __match_any_sync(0xffffffffu, d);
    if (d < kBins && (int)(threadIdx.x & 31) == __ffs(same) - 1) atomicAdd(&cnt[d], __popc(same));
    __syncthreads();
    if ((int)threadIdx.x < bins) hist[threadIdx.x * tiles + blockIdx.x] = cnt[threadIdx.x];
}

// Stable placement by digit: a particle goes to the prefix of (its digit, its
// tile) plus the number of particles before it in the tile with the same digit.
//   ids_in null    the id is the particle's index (first pass)
//   keys_out null  last pass: only ids are written
//   hist           else: counts of the next digit per tile of the output (zero on entry)
// The blocks past the tiles (first pass) write the cell list from its prefix.
__global__ void __launch_bounds__(kTile)
k_na_scatter(const int *keys, const int *ids_in, int np, int shift, int bins, int tiles, Prefix offs,
             int *keys_out, int *ids_out, int next_shift, int next_bins, int *hist, Prefix cells,
             int *cell_start)
{
    __shared__ __align__(16) unsigned char cnt[kTileWarps][kBins];   // a warp's particles of a digit (at most 32)
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    if ((int)blockIdx.x >= tiles) {
        const int e = (blockIdx.x - tiles) * kTile + t;
        if (e < cells.n) cell_start[e] = cells.at(e);
        return;
    }
    unsigned *zero = reinterpret_cast<unsigned *>(&cnt[0][0]);
#pragma unroll
    for (int k = 0; k < kTileWarps * kBins / 4; k += kTile) zero[k + t] = 0u;
    __syncthreads();
    const int item = blockIdx.x * kTile + t;
    const int c = item < np ? keys[item] : 0;
    const int d = item < np ? (c >> shift) & (bins - 1) : kBins;
    const unsigned same = __match_any_sync(0xffffffffu, d);
    if (d < kBins && lane == __ffs(same) - 1) cnt[warp][d] = (unsigned char)__popc(same);
    __syncthreads();
    int next = -1;
    if (item < np) {
        int pos = offs.at(d * tiles + blockIdx.x) + __popc(same & ((1u << lane) - 1u));
        for (int w = 0; w < warp; ++w) pos += cnt[w][d];
        ids_out[pos] = ids_in ? ids_in[item] : item;
        if (keys_out) {
            keys_out[pos] = c;
            next = ((c >> next_shift) & (next_bins - 1)) * tiles + pos / kTile;
        }
    }
    if (!keys_out) return;   // the whole block
    const unsigned mates = __match_any_sync(0xffffffffu, next);
    if (next >= 0 && lane == __ffs(mates) - 1) atomicAdd(&hist[next], __popc(mates));
}

int na_fail(int code, const char *msg)
{
    lbdpsk::set_last_error(msg);
    return code;
}

}  // namespace

extern "C" int lbdps_bin_sort_noalloc(int dim, const int n[3], int64_t np, const double *const pos[3],
                                      int *cell_start, int *order, void *stream)
{
    if ((dim != 2 && dim != 3) || !n || !pos || !cell_start || np < 0 || (np > 0 && !order))
        return na_fail(LBDPS_ERR_INVALID, "lbdps_bin_sort_noalloc: bad arguments");
    long long ncell = 1;
    int nn[3] = {1, 1, 1};
    for (int a = 0; a < dim; ++a) {
        if (n[a] < 1) return na_fail(LBDPS_ERR_INVALID, "lbdps_bin_sort_noalloc: n[a] must be positive");
        if (np > 0 && !pos[a]) return na_fail(LBDPS_ERR_INVALID, "lbdps_bin_sort_noalloc: NULL position array");
        nn[a] = n[a];
        ncell *= n[a];
        if (ncell > kMaxCells) break;
    }
    if (ncell > kMaxCells || np > kMaxParticles) {
        char buf[200];
        snprintf(buf, sizeof(buf),
                 "lbdps_bin_sort_noalloc: %lld%s cells / %lld particles exceed the fixed scratch "
                 "(at most %d cells and %d particles)",
                 ncell, ncell > kMaxCells ? "+" : "", (long long)np, kMaxCells, kMaxParticles);
        return na_fail(LBDPS_ERR_CAPACITY, buf);
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        cudaGetLastError();
        return na_fail(LBDPS_ERR_CUDA, "lbdps_bin_sort_noalloc: no current CUDA device");
    }
    int *base = nullptr;
    {
        // one-time set-up per device, with that device current: the device
        // address of the scratch array (the host-side symbol is only a stand-in)
        std::lock_guard<std::mutex> lock(g_setup_mutex);
        if (!g_scratch_ptr[dev]) {
            void *p = nullptr;
            cudaError_t e = cudaGetSymbolAddress(&p, g_bin_scratch);
            if (e != cudaSuccess || !p) {
                cudaGetLastError();
                char buf[160];
                snprintf(buf, sizeof(buf), "lbdps_bin_sort_noalloc: cudaGetSymbolAddress failed: %s",
                         cudaGetErrorString(e));
                return na_fail(LBDPS_ERR_CUDA, buf);
            }
            g_scratch_ptr[dev] = (int *)p;
        }
        base = g_scratch_ptr[dev];
    }
    cudaStream_t st = (cudaStream_t)stream;
    const int npi = (int)np, nc = (int)ncell;
    const int tiles = (npi + kTile - 1) / kTile;
    // digits of equal width, as few as the largest key needs
    int bits = 0;
    while ((1ll << bits) < ncell) ++bits;
    const int passes = bits > kRadixBits ? 2 : 1;
    const int width = passes == 2 ? (bits + 1) / 2 : std::max(bits, 1);
    const int bins = 1 << width, bins2 = 1 << std::max(bits - width, 0);
    int *counts = base;                                  // nc + 1, then the second histogram
    int *hist2 = counts + ((nc + 1 + 3) & ~3);
    int *hist = base + kCountInts;
    int *keys = hist + kMaxHist;
    int *keys_a = keys + kMaxParticles;
    int *ids_a = keys_a + kMaxParticles;
    int *sums = ids_a + kMaxParticles;                   // sums and bases of two prefixes
    unsigned *tickets = reinterpret_cast<unsigned *>(sums + 4 * kMaxScanTiles);
    const Prefix cells{counts, nc + 1, sums, sums + kMaxScanTiles, tickets};
    const Prefix digit1{hist, bins * tiles, sums + 2 * kMaxScanTiles, sums + 3 * kMaxScanTiles, tickets + 1};
    const Prefix digit2{hist2, bins2 * tiles, digit1.tile_sum, digit1.base, tickets + 1};

    // counts (and the second histogram) start at zero; the array keeps
    // whatever the last call left
    const size_t clear = passes == 2 ? (size_t)(hist2 - counts) + (size_t)digit2.n : (size_t)nc + 1;
    cudaError_t e = cudaMemsetAsync(counts, 0, sizeof(int) * clear, st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return na_fail(LBDPS_ERR_CUDA, "lbdps_bin_sort_noalloc: clearing the counts failed");
    }
    // Launches bound this at ordinary sizes: one each for keys with counts and
    // the first histogram, both prefixes, the first placement with the cell
    // list and the second histogram, then its prefix and the second placement.
    // 200,000 particles in 256 x 2048 cells: 107 us with 20 launches (8-bit
    // digits, three launches per prefix), now 46 us; 2^20 particles 244 -> 176 us spread
    // evenly and 853 -> 108 us all in one cell (GB300).
    if (npi > 0)
        k_na_keys<<<tiles, kTile, 0, st>>>(dim, nn[0], nn[1], nn[2], pos[0], pos[1],
                                           dim > 2 ? pos[2] : nullptr, npi, keys, counts, bins, tiles, hist);
    k_na_prefix<<<cells.tiles() + digit1.tiles(), kTile, 0, st>>>(cells, digit1);
    const bool two = passes == 2 && npi > 0;
    k_na_scatter<<<tiles + (nc + kTile) / kTile, kTile, 0, st>>>(
        keys, nullptr, npi, 0, bins, tiles, digit1, two ? keys_a : nullptr, two ? ids_a : order, width,
        bins2, hist2, cells, cell_start);
    if (two) {
        k_na_prefix<<<digit2.tiles(), kTile, 0, st>>>(digit2, Prefix{});
        k_na_scatter<<<tiles, kTile, 0, st>>>(keys_a, ids_a, npi, width, bins2, tiles, digit2, nullptr, order,
                                              0, 0, nullptr, Prefix{}, nullptr);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) {
        char buf[160];
        snprintf(buf, sizeof(buf), "lbdps_bin_sort_noalloc: launch failed: %s", cudaGetErrorString(e));
        return na_fail(LBDPS_ERR_CUDA, buf);
    }
    return LBDPS_OK;
}
