// Peano-Hilbert keys, the stable device radix sort of (key, index) and a device
// exclusive scan (Sec. 1.2: Gadget3 orders its particles along the Hilbert curve).
#include <algorithm>
#include <utility>

#include "sph_internal.cuh"

namespace sphgrp {

// ---------------------------------------------------------------------------------
// Keys
// ---------------------------------------------------------------------------------

// Spreads the low 21 bits of v so that bit b lands on bit 3b.
__device__ __forceinline__ uint64_t spread3(uint32_t v) {
    uint64_t x = v & 0x1fffffu;
    x = (x | (x << 32)) & 0x001f00000000ffffull;
    x = (x | (x << 16)) & 0x001f0000ff0000ffull;
    x = (x | (x << 8)) & 0x100f00f00f00f00full;
    x = (x | (x << 4)) & 0x10c30c30c30c30c3ull;
    x = (x | (x << 2)) & 0x1249249249249249ull;
    return x;
}

// Hilbert index of a cell of the 2^21 grid by Skilling's transpose construction:
// from the coarsest level down, every axis either reflects (bit set) or swaps its
// lower bits with axis 0 (bit clear); then a Gray code across the axes and a common
// correction; the index interleaves the transposed words, axis 0 most significant.
__device__ __forceinline__ uint64_t hilbert_key(uint32_t a0, uint32_t a1, uint32_t a2) {
#pragma unroll
    for (uint32_t q = 1u << (kKeyLevels - 1); q > 1u; q >>= 1) {
        const uint32_t lowmask = q - 1u;
        if (a0 & q) a0 ^= lowmask;
        if (a1 & q) {
            a0 ^= lowmask;
        } else {
            uint32_t t = (a0 ^ a1) & lowmask;
            a0 ^= t;
            a1 ^= t;
        }
        if (a2 & q) {
            a0 ^= lowmask;
        } else {
            uint32_t t = (a0 ^ a2) & lowmask;
            a0 ^= t;
            a2 ^= t;
        }
    }
    a1 ^= a0;
    a2 ^= a1;
    uint32_t corr = 0;
#pragma unroll
    for (uint32_t q = 1u << (kKeyLevels - 1); q > 1u; q >>= 1)
        if (a2 & q) corr ^= q - 1u;
    a0 ^= corr;
    a1 ^= corr;
    a2 ^= corr;
    return (spread3(a0) << 2) | (spread3(a1) << 1) | spread3(a2);
}

// The cell of the 2^21 grid, floor(x 2^21) clamped to [0, 2^21 - 1] (a NaN to 0), taken
// from the bits of x with integer operations: x = (2^52 + f) 2^(e - 1075), so
// floor(x 2^21) = (2^52 + f) >> (1054 - e) for 0 < x < 1; FP64 arithmetic is a slow
// pipe on this part, and this form is exact.
__device__ __forceinline__ uint32_t grid21(uint64_t b) {
    if (b >> 63) return 0u;                                     // x <= -0 (or a negative NaN)
    const int e = (int)(b >> 52);                               // biased exponent
    if (e >= 1023) return (e == 2047 && (b << 12)) ? 0u : 2097151u;   // x >= 1, inf; NaN
    const int sh = 1054 - e;                                    // >= 32
    if (sh > 52) return 0u;                                     // x 2^21 < 1 (zero, subnormal)
    return (uint32_t)(((b & 0xfffffffffffffull) | (1ull << 52)) >> sh);
}

// 0 <= x < 1 from the bits (-0 included, NaN excluded)
__device__ __forceinline__ bool unit_bits(uint64_t b) {
    return b < 0x3ff0000000000000ull || b == 0x8000000000000000ull;
}

// Radix digits: 9 bits, 7 passes for the 63-bit keys.
constexpr int kDigitBits = 9;
constexpr int kBins = 1 << kDigitBits;
constexpr int kKeyPasses = 7;
static_assert(kDigitBits * kKeyPasses >= 3 * kKeyLevels, "the passes cover the key");
// counts of every pass's digits, then counters (the tickets of the passes, the blocks done)
constexpr int kSortTickets = 16;
constexpr int kHistWords = kKeyPasses * kBins + kSortTickets;
static_assert(kHistWords <= kSortHeadWords, "sort scratch head");

// The last block to finish turns the digit counts of `passes` passes into each digit's first
// position (exclusive scan over the bins), so that no launch of its own is needed.
__device__ __forceinline__ void scan_digit_counts(uint32_t* hist, int passes, uint32_t* done) {
    __shared__ uint32_t wsum[kKeyPasses][8];
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t c0[kKeyPasses], c1[kKeyPasses], v[kKeyPasses];
#pragma unroll
    for (int p = 0; p < kKeyPasses; ++p) {   // all loads in flight together
        c0[p] = p < passes ? __ldcg(hist + p * kBins + 2 * threadIdx.x) : 0u;
        c1[p] = p < passes ? __ldcg(hist + p * kBins + 2 * threadIdx.x + 1) : 0u;
        v[p] = c0[p] + c1[p];
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
        for (int p = 0; p < kKeyPasses; ++p) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, v[p], o);
            if (lane >= o) v[p] += t;
        }
    }
    if (lane == 31) {
#pragma unroll
        for (int p = 0; p < kKeyPasses; ++p) wsum[p][w] = v[p];
    }
    __syncthreads();
#pragma unroll
    for (int p = 0; p < kKeyPasses; ++p) {
        if (p >= passes) break;
        uint32_t off = v[p] - c0[p] - c1[p];
        for (int k = 0; k < w; ++k) off += wsum[p][k];
        hist[p * kBins + 2 * threadIdx.x] = off;
        hist[p * kBins + 2 * threadIdx.x + 1] = off + c0[p];
    }
}

// Keys of the particles and the digit counts of all passes.
__global__ void __launch_bounds__(256) k_keys(int64_t n, const double* __restrict__ pos, uint64_t* __restrict__ keys,
                                              uint32_t* hist, unsigned* err) {
    __shared__ uint32_t h[kKeyPasses * kBins];
    for (int k = threadIdx.x; k < kKeyPasses * kBins; k += 256) h[k] = 0u;
    __syncthreads();
    const uint64_t* pb = reinterpret_cast<const uint64_t*>(pos);
    for (int64_t i = blockIdx.x * 256ll + threadIdx.x; i < n; i += gridDim.x * 256ll) {
        const uint64_t x = pb[3 * i], y = pb[3 * i + 1], z = pb[3 * i + 2];
        if (!(unit_bits(x) && unit_bits(y) && unit_bits(z))) atomicOr(err, kErrRange);
        const uint64_t key = hilbert_key(grid21(x), grid21(y), grid21(z));
        keys[i] = key;
#pragma unroll
        for (int p = 0; p < kKeyPasses; ++p)
            atomicAdd(&h[p * kBins + (int)((key >> (p * kDigitBits)) & (kBins - 1))], 1u);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < kKeyPasses * kBins; k += 256)
        if (h[k]) atomicAdd(&hist[k], h[k]);
    scan_digit_counts(hist, kKeyPasses, hist + kKeyPasses * kBins + kSortTickets - 1);
}

// ---------------------------------------------------------------------------------
// Exclusive scan (int32 / int64), three phases: tile sums, scan of the sums
// (recursive), tile scan with carry.  Tiles of 4096 = 1024 threads x 4 items.
// ---------------------------------------------------------------------------------

constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;

template <typename T>
__device__ __forceinline__ T block_exclusive(T v, T* warp_tot, T& block_total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    T inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) warp_tot[w] = inc;
    __syncthreads();
    if (w == 0) {
        T s = (lane < (int)(blockDim.x >> 5)) ? warp_tot[lane] : T(0);
        T si = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            T t = __shfl_up_sync(0xffffffffu, si, o);
            if (lane >= o) si += t;
        }
        warp_tot[lane] = si - s;  // exclusive prefix of warp totals
        if (lane == 31) warp_tot[32] = si;
    }
    __syncthreads();
    block_total = warp_tot[32];
    T r = warp_tot[w] + inc - v;
    __syncthreads();
    return r;
}

template <typename T>
__global__ void k_scan_reduce(const T* __restrict__ in, int64_t n, T* __restrict__ sums) {
    __shared__ T wt[33];
    int64_t base = blockIdx.x * (int64_t)kScanTile + threadIdx.x * kScanItems;
    T s = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k)
        if (base + k < n) s += in[base + k];
    T tot;
    block_exclusive<T>(s, wt, tot);
    if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

template <typename T>
__global__ void k_scan_down(const T* in, T* out, int64_t n, const T* __restrict__ carry,
                            T* total) {
    __shared__ T wt[33];
    int64_t base = blockIdx.x * (int64_t)kScanTile + threadIdx.x * kScanItems;
    T v[kScanItems];
    T s = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        v[k] = (base + k < n) ? in[base + k] : T(0);
        s += v[k];
    }
    T tot;
    T ex = block_exclusive<T>(s, wt, tot);
    T c = carry ? carry[blockIdx.x] : T(0);
    T run = c + ex;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        if (base + k < n) out[base + k] = run;
        run += v[k];
    }
    if (total && blockIdx.x == gridDim.x - 1 && threadIdx.x == blockDim.x - 1) *total = c + tot;
}

template <typename T>
static void scan_rec(const T* in, T* out, int64_t n, T* aux, T* total, cudaStream_t s) {
    int64_t nb = (n + kScanTile - 1) / kScanTile;
    if (nb <= 1) {
        k_scan_down<T><<<1, kScanThreads, 0, s>>>(in, out, n, nullptr, total);
        note_launch();
        return;
    }
    k_scan_reduce<T><<<(unsigned)nb, kScanThreads, 0, s>>>(in, n, aux);
    note_launch();
    scan_rec<T>(aux, aux, nb, aux + nb, nullptr, s);
    k_scan_down<T><<<(unsigned)nb, kScanThreads, 0, s>>>(in, out, n, aux, total);
    note_launch();
}

static int64_t scan_aux_need(int64_t n) {
    int64_t need = 0;
    while (n > kScanTile) {
        n = (n + kScanTile - 1) / kScanTile;
        need += n;
    }
    return need + 8;
}

int exclusive_scan_i32(Ctx* c, const int32_t* in, int32_t* out, int64_t n, int32_t* total_dev,
                       cudaStream_t s) {
    if (n <= 0) return SPHGRP_OK;
    if (scan_aux_need(n) > c->scan_aux_cap) return set_error(SPHGRP_EOVERFLOW, "scan scratch too small");
    scan_rec<int32_t>(in, out, n, c->scan_aux, total_dev, s);
    return check_cuda(cudaGetLastError(), "scan");
}

int exclusive_scan_i64(Ctx* c, const int64_t* in, int64_t* out, int64_t n, int64_t* total_dev,
                       cudaStream_t s) {
    if (n <= 0) return SPHGRP_OK;
    if (2 * scan_aux_need(n) > c->scan_aux_cap) return set_error(SPHGRP_EOVERFLOW, "scan scratch too small");
    scan_rec<int64_t>(in, out, n, reinterpret_cast<int64_t*>(c->scan_aux), total_dev, s);
    return check_cuda(cudaGetLastError(), "scan");
}

// ---------------------------------------------------------------------------------
// LSD radix sort, 9-bit digits, stable, one kernel per pass.  The digit counts of all
// passes come from the kernel that makes the keys.  A pass's block takes the next tile
// (in ticket order), ranks its keys by ballots of their digits' bits -- warp w owns a
// contiguous part of the tile and goes through it 32 keys at a time, so ranks follow the
// input order --
// publishes the tile's digit counts, sorts the tile by digit in shared memory, and finds
// for every digit how many such keys the earlier tiles hold by looking back through their
// published counts until one has its total (decoupled look-back).  Then every digit's
// run goes out with consecutive threads on consecutive addresses.
//
// Every key and value is read and written once per pass.  On large sets a pass is bound by
// the dependent steps of a block, of which 60 KB of shared memory leave three on an SM: a
// pass over 4.0M keys takes about 70 us (97 the last), where its 96 MB take 14 at the measured
// 6791 GB/s.  On small ones it is bound by the launches (8 where counting, scanning and
// scattering 8-bit digits took 25): 20k particles by the allocation-free call 182 -> 101 us.
//
// A tile's word of a digit: 0 = not there yet, v + 1 = the tile's own count v, bit 31 set =
// the count of all tiles up to it.  The earlier tiles were taken by blocks that run
// already, so a wait ends.  It is bounded all the same, and a thread at the limit counts its
// digit in the earlier tile's keys itself: the order is right whatever happens, so that the
// kernels that follow in a step that reads nothing back never index by a part of it.
// ---------------------------------------------------------------------------------

constexpr uint32_t kTotalBit = 0x80000000u;
constexpr uint32_t kSpinLimit = 1u << 16;   // reads of a word, some 50 ms

struct SweepArgs {
    const uint64_t* kin;
    const int32_t* vin;    // null: the value is the position
    uint64_t* kout;
    int32_t* vout;
    uint64_t* kout2;       // second copies of the output, or null (last pass)
    int32_t* vout2;
    int32_t* rank_of;      // inverse of the values, or null (last pass)
    int64_t n;
    int shift;
    const uint32_t* start; // first position of every digit
    uint32_t* counts;      // published words, kBins per tile (zero)
    uint32_t* counts_next; // those of the next pass, zeroed here
    uint32_t* ticket;
};

// lanes with the same digit (kDigitBits bits and the one above them)
__device__ __forceinline__ uint32_t same_digit(uint32_t d) {
    uint32_t peers = 0xffffffffu;
#pragma unroll
    for (int b = 0; b <= kDigitBits; ++b) {
        const bool set = d >> b & 1u;
        const uint32_t vote = __ballot_sync(0xffffffffu, set);
        peers &= set ? vote : ~vote;
    }
    return peers;
}

// keys of tile t (a whole one: a later tile exists) with digit d
__device__ __noinline__ uint32_t count_in_tile(const SweepArgs& a, int t, int tile_keys, uint32_t d) {
    const uint64_t* k = a.kin + (int64_t)t * tile_keys;
    uint32_t n = 0;
    for (int e = 0; e < tile_keys; ++e) n += ((uint32_t)(k[e] >> a.shift) & (kBins - 1)) == d ? 1u : 0u;
    return n;
}

template <int ITEMS>
constexpr size_t sweep_smem() {
    return (size_t)256 * ITEMS * 12;
}

template <int ITEMS>
__global__ void __launch_bounds__(256) k_radix_pass(SweepArgs a) {
    constexpr int kTileKeys = 256 * ITEMS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint64_t* sk = reinterpret_cast<uint64_t*>(smem_raw);        // the tile, sorted by digit
    int32_t* sv = reinterpret_cast<int32_t*>(sk + kTileKeys);
    __shared__ uint16_t wh[8][kBins];
    __shared__ uint32_t lbase[kBins];    // tile-local position of the digit's run
    __shared__ uint32_t gbase[kBins];    // global position of the digit's run, less lbase
    __shared__ uint32_t wsum[8];
    __shared__ int tile_s;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (threadIdx.x == 0) tile_s = (int)atomicAdd(a.ticket, 1u);
    for (int d = threadIdx.x; d < 8 * kBins / 2; d += 256) reinterpret_cast<uint32_t*>(&wh[0][0])[d] = 0u;
    __syncthreads();
    const int tile = tile_s;
    const int64_t tile0 = (int64_t)tile * kTileKeys;
    uint32_t* mine = a.counts + (int64_t)tile * kBins;
    {
        uint32_t* clear = a.counts_next + (int64_t)tile * kBins;
        clear[threadIdx.x] = 0u;
        clear[threadIdx.x + 256] = 0u;
    }
    const int64_t base = tile0 + w * 32 * ITEMS;
    const uint32_t lt = (1u << lane) - 1u;
    uint64_t kk[ITEMS];
    int32_t vv[ITEMS];
    uint32_t rk[ITEMS];
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const int64_t i = base + r * 32 + lane;
        kk[r] = i < a.n ? a.kin[i] : 0ull;
        vv[r] = i < a.n ? (a.vin ? a.vin[i] : (int32_t)i) : 0;
    }
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const bool valid = base + r * 32 + lane < a.n;
        const uint32_t d = valid ? (uint32_t)(kk[r] >> a.shift) & (kBins - 1) : (uint32_t)kBins;
        const uint32_t peers = same_digit(d);
        const uint32_t prev = valid ? wh[w][d] : 0u;
        __syncwarp();
        if (valid && lane == __ffs(peers) - 1) wh[w][d] = (uint16_t)(prev + __popc(peers));
        __syncwarp();
        rk[r] = prev + __popc(peers & lt);
    }
    __syncthreads();
    // thread t owns the digits 2t and 2t + 1: prefix over the warps, the tile's count
    // published, and the tile-local starts (exclusive scan of the counts)
    uint32_t tot[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int d = 2 * threadIdx.x + q;
        uint32_t run = 0;
#pragma unroll
        for (int ww = 0; ww < 8; ++ww) {
            const uint32_t c = wh[ww][d];
            wh[ww][d] = (uint16_t)run;
            run += c;
        }
        tot[q] = run;
    }
    volatile uint32_t* pub = mine;
#pragma unroll
    for (int q = 0; q < 2; ++q) pub[2 * threadIdx.x + q] = tile == 0 ? (kTotalBit | tot[q]) : tot[q] + 1u;
    uint32_t v = tot[0] + tot[1];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    if (lane == 31) wsum[w] = v;
    __syncthreads();
    uint32_t off = v - tot[0] - tot[1];
    for (int ww = 0; ww < w; ++ww) off += wsum[ww];
    lbase[2 * threadIdx.x] = off;
    lbase[2 * threadIdx.x + 1] = off + tot[0];
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        if (base + r * 32 + lane < a.n) {
            const uint32_t d = (uint32_t)(kk[r] >> a.shift) & (kBins - 1);
            const uint32_t q = lbase[d] + wh[w][d] + rk[r];
            sk[q] = kk[r];
            sv[q] = vv[r];
        }
    }
    // look back
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int d = 2 * threadIdx.x + q;
        uint32_t before = 0;
        uint32_t spins = 0;
        for (int t = tile - 1; t >= 0;) {
            const uint32_t word = *reinterpret_cast<volatile uint32_t*>(a.counts + (int64_t)t * kBins + d);
            if (word & kTotalBit) {
                before += word & ~kTotalBit;
                break;
            }
            if (word) {
                before += word - 1u;
                --t;
            } else if (++spins > kSpinLimit) {
                before += count_in_tile(a, t, kTileKeys, (uint32_t)d);
                --t;
            }
        }
        if (tile > 0) pub[d] = kTotalBit | (before + tot[q]);
        gbase[d] = a.start[d] + before - (q ? off + tot[0] : off);
    }
    __syncthreads();
    const int cnt = (int)min((int64_t)kTileKeys, a.n - tile0);
    for (int e = threadIdx.x; e < cnt; e += 256) {
        const uint64_t key = sk[e];
        const int32_t val = sv[e];
        const uint32_t p = gbase[(uint32_t)(key >> a.shift) & (kBins - 1)] + (uint32_t)e;
        a.kout[p] = key;
        a.vout[p] = val;
        if (a.kout2) a.kout2[p] = key;
        if (a.vout2) a.vout2[p] = val;
        if (a.rank_of) a.rank_of[val] = (int32_t)p;
    }
}

// Keys per tile: small sets need tiles enough for the chip, large ones long runs per digit.
static int sort_items(int64_t n) { return n >= (1 << 20) ? 16 : n >= (1 << 17) ? 8 : 4; }

static int64_t sort_scratch_words(int64_t n) {
    const int64_t tiles = (n + 256 * sort_items(n) - 1) / (256 * sort_items(n));
    return kSortHeadWords + 2 * tiles * kBins;
}

// scratch words for every n up to n_max (the tiles per key drop where the tile grows)
int64_t sort_scratch_cap(int64_t n_max) {
    int64_t words = sort_scratch_words(n_max);
    for (int64_t step : {(int64_t)1 << 17, (int64_t)1 << 20})
        if (n_max >= step) words = std::max(words, sort_scratch_words(step - 1));
    return words;
}

static int launch_pass(const SweepArgs& a, cudaStream_t s) {
    const int items = sort_items(a.n);
    const unsigned tiles = (unsigned)((a.n + 256 * items - 1) / (256 * items));
    if (items == 16) {
        k_radix_pass<16><<<tiles, 256, sweep_smem<16>(), s>>>(a);
    } else if (items == 8) {
        k_radix_pass<8><<<tiles, 256, sweep_smem<8>(), s>>>(a);
    } else {
        k_radix_pass<4><<<tiles, 256, sweep_smem<4>(), s>>>(a);
    }
    note_launch();
    return check_cuda(cudaGetLastError(), "radix pass");
}

// Scratch words: digit counts and tickets (zeroed), then two sets of published words used
// by the passes in turn (the first zeroed here, each pass zeroes the other).
static void zero_scratch(uint32_t* scratch, int64_t n, cudaStream_t s) {
    const int64_t set = (sort_scratch_words(n) - kSortHeadWords) / 2;
    cudaMemsetAsync(scratch, 0, (size_t)(kSortHeadWords + set) * sizeof(uint32_t), s);
}

// Passes over the digits of `bits` bits: (kbuf[0], vbuf[0] or the positions) -> ... ; the
// result ends in kbuf[passes & 1], vbuf[passes & 1].
static int radix_passes(uint64_t* const (&kbuf)[2], int32_t* const (&vbuf)[2], int64_t n, int passes, uint32_t* scratch,
                        uint64_t* keys_copy, int32_t* vals_copy, int32_t* rank_of, cudaStream_t s) {
    const int64_t set = (sort_scratch_words(n) - kSortHeadWords) / 2;
    uint32_t* sets[2] = {scratch + kSortHeadWords, scratch + kSortHeadWords + set};
    // With its static tables the largest tile is above the 48 KB that need no permission,
    // which belongs to the current device: given on every call, whichever device that is.
    if (sort_items(n) == 16) {
        int rc = check_cuda(cudaFuncSetAttribute(k_radix_pass<16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)sweep_smem<16>()), "radix pass shared memory");
        if (rc) return rc;
    }
    for (int p = 0; p < passes; ++p) {
        const bool last = p == passes - 1;
        SweepArgs a;
        a.kin = kbuf[p & 1];
        a.vin = p == 0 ? nullptr : vbuf[p & 1];
        a.kout = kbuf[(p + 1) & 1];
        a.vout = vbuf[(p + 1) & 1];
        a.kout2 = last ? keys_copy : nullptr;
        a.vout2 = last ? vals_copy : nullptr;
        a.rank_of = last ? rank_of : nullptr;
        a.n = n;
        a.shift = p * kDigitBits;
        a.start = scratch + p * kBins;
        a.counts = sets[p & 1];
        a.counts_next = sets[(p + 1) & 1];
        a.ticket = scratch + kKeyPasses * kBins + p;
        int rc = launch_pass(a, s);
        if (rc) return rc;
    }
    return SPHGRP_OK;
}

// Blocks of the kernels that count digits: at least 4 keys a thread and four blocks for each
// of the chip's 152 SMs, so that few of them add their counts to memory.
constexpr int64_t kCountBlocks = 152 * 4;

static void launch_keys(int64_t n, const double* pos, uint64_t* keys, uint32_t* hist, unsigned* err, cudaStream_t s) {
    const int64_t blocks = std::min<int64_t>((n + 1023) / 1024, kCountBlocks);
    k_keys<<<(unsigned)blocks, 256, 0, s>>>(n, pos, keys, hist, err);
    note_launch();
}

// Keys and stable order of the context's particles: c->keys, c->perm, c->rank_of, and copies
// for the caller (or null).
int sort_keys(Ctx* c, int64_t n, const double* pos, cudaStream_t s, uint64_t* keys_copy, int32_t* perm_copy) {
    if (sort_scratch_words(n) > c->hist_cap) return set_error(SPHGRP_EOVERFLOW, "radix scratch too small");
    zero_scratch(c->hist, n, s);
    launch_keys(n, pos, c->keys_alt, c->hist, c->err, s);
    uint64_t* const kbuf[2] = {c->keys_alt, c->keys};
    int32_t* const vbuf[2] = {c->perm_alt, c->perm};
    static_assert(kKeyPasses % 2 == 1, "the result ends in the second buffers");
    int rc = radix_passes(kbuf, vbuf, n, kKeyPasses, c->hist, keys_copy, perm_copy, c->rank_of, s);
    if (rc) return rc;
    return check_cuda(cudaGetLastError(), "sort");
}

// ---------------------------------------------------------------------------------
// Sort of several boxes at once: keys as above, then one stable pass per 9 bits of the box
// index, so that the order is (box, key); the context's keys and perm end in that order
// and box_of_rank holds every rank's box.
// ---------------------------------------------------------------------------------

// box of every rank (key order) and the digit counts of its passes
__global__ void __launch_bounds__(256) k_box_digit(int64_t n, const int32_t* __restrict__ perm,
                                                   const int64_t* __restrict__ box_off, int nbox,
                                                   uint64_t* __restrict__ dkey, int passes, uint32_t* hist) {
    __shared__ uint32_t h[kKeyPasses * kBins];
    for (int k = threadIdx.x; k < passes * kBins; k += 256) h[k] = 0u;
    __syncthreads();
    for (int64_t r = blockIdx.x * 256ll + threadIdx.x; r < n; r += gridDim.x * 256ll) {
        const int64_t i = perm[r];
        int lo = 0, hi = nbox;   // box_off[lo] <= i < box_off[hi]
        while (hi - lo > 1) {
            int mid = (lo + hi) >> 1;
            if (box_off[mid] <= i) lo = mid; else hi = mid;
        }
        dkey[r] = (uint64_t)lo;
        for (int p = 0; p < passes; ++p) atomicAdd(&h[p * kBins + ((lo >> (p * kDigitBits)) & (kBins - 1))], 1u);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < passes * kBins; k += 256)
        if (h[k]) atomicAdd(&hist[k], h[k]);
    scan_digit_counts(hist, passes, hist + kKeyPasses * kBins + kSortTickets - 1);
}

__global__ void k_box_gather(int64_t n, const int32_t* __restrict__ src, const uint64_t* __restrict__ keys,
                             const int32_t* __restrict__ perm, const uint64_t* __restrict__ dkey,
                             uint64_t* __restrict__ keys_out, int32_t* __restrict__ perm_out,
                             int32_t* __restrict__ rank_of, int32_t* __restrict__ box_of_rank) {
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int32_t r = src[p];
    const int32_t i = perm[r];
    keys_out[p] = keys[r];
    perm_out[p] = i;
    rank_of[i] = (int32_t)p;
    box_of_rank[p] = (int32_t)dkey[p];
}

int sort_keys_boxed(Ctx* c, int64_t n, const double* pos, const int64_t* box_off_dev, int nbox, uint64_t* tmp64a,
                    uint64_t* tmp64b, int32_t* tmp32a, int32_t* tmp32b, int32_t* box_of_rank, cudaStream_t s) {
    int rc = sort_keys(c, n, pos, s, nullptr, nullptr);
    if (rc) return rc;
    if (nbox <= 1) {
        cudaMemsetAsync(box_of_rank, 0, n * sizeof(int32_t), s);
        return check_cuda(cudaGetLastError(), "box sort");
    }
    int passes = 1;
    while ((int64_t)nbox > (int64_t)1 << (passes * kDigitBits)) ++passes;
    zero_scratch(c->hist, n, s);
    k_box_digit<<<(unsigned)std::min<int64_t>((n + 1023) / 1024, kCountBlocks), 256, 0, s>>>(
        n, c->perm, box_off_dev, nbox, tmp64a, passes, c->hist);
    note_launch();
    uint64_t* const kbuf[2] = {tmp64a, tmp64b};
    int32_t* const vbuf[2] = {tmp32b, tmp32a};
    if ((rc = radix_passes(kbuf, vbuf, n, passes, c->hist, nullptr, nullptr, nullptr, s))) return rc;
    // box digits in (box, key) order, and the rank in key order of every position
    k_box_gather<<<blocks_for(n, 256), 256, 0, s>>>(n, vbuf[passes & 1], c->keys, c->perm, kbuf[passes & 1], c->keys_alt,
                                                     c->perm_alt, c->rank_of, box_of_rank);
    note_launch();
    std::swap(c->keys, c->keys_alt);
    std::swap(c->perm, c->perm_alt);
    return check_cuda(cudaGetLastError(), "box sort");
}

// The same keys + stable radix sort on caller-provided buffers: the sorted keys and the
// permutation end in keys_out / perm_out, keys_alt / perm_alt are the other pair, scratch
// holds at least sort_scratch_words(n) words.  err receives the range-check flag.  No
// allocation.
int sort_keys_scratch(int64_t n, const double* pos, uint64_t* keys_out, int32_t* perm_out,
                      uint64_t* keys_alt, int32_t* perm_alt, uint32_t* scratch, int64_t scratch_words, unsigned* err,
                      cudaStream_t s) {
    if (sort_scratch_words(n) > scratch_words) return set_error(SPHGRP_EOVERFLOW, "radix scratch too small");
    zero_scratch(scratch, n, s);
    launch_keys(n, pos, keys_alt, scratch, err, s);
    uint64_t* const kbuf[2] = {keys_alt, keys_out};
    int32_t* const vbuf[2] = {perm_alt, perm_out};
    int rc = radix_passes(kbuf, vbuf, n, kKeyPasses, scratch, nullptr, nullptr, nullptr, s);
    if (rc) return rc;
    return check_cuda(cudaGetLastError(), "sort (caller buffers)");
}

}  // namespace sphgrp
