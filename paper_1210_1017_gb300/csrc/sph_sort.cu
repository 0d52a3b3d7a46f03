// Radix sort of (key, value) pairs, the scan that turns per-cell counts into
// first-index-per-cell offsets, and the cell sort (Sec. 3.1 of the paper:
// label, radix sort, reorder, first index of each cell).
//
// The sort is a stable least-significant-digit radix sort with 8-bit digits.
// Per digit place: the digit counts of each 4096-key tile, their scans per
// digit, and a scatter in which each tile ranks its keys in shared memory and
// moves them to their digit's run.  Up to kFewTiles tiles the scatter adds up
// the counts itself (no scan launch), and an input of one tile is sorted by one
// block in one launch, all places in shared memory.  The tiles are independent:
// a one-pass organisation, whose tiles wait for the offsets of the tiles before
// them, spent most of its time and half of its instructions in those waits and
// in __match_any_sync (one GB300: 4.0M pairs with 24-bit keys 197 us, 30M with
// 32-bit keys 1,223 us, 1,000 pairs 51 us; these kernels 115, 761 and 10.4).
// (__match_any_sync steps through the distinct digits of a warp, so that one was
// at its best on keys with hardly any: 300k equal 32-bit keys 42.9 us on the
// device, 38.0 here.)
#include "sph_internal.cuh"

namespace sph {

namespace {

constexpr uint32_t kFull = 0xffffffffu;
// Where the scan's launch costs more than every block adding up all counts: us
// per sort of random 24-bit keys without / with it, calls one after another (bound
// by the launches) and on the device alone (a graph):
//   tiles           49           96           128          160
//   calls           43.2 / 51.8  47.3 / 53.4  51.4 / 57.5  62.6 / 66.5
//   device          31.6 / 33.6  33.8 / 33.3  38.8 / 35.6  49.4 / 44.5
constexpr uint32_t kFewTiles = 128;

__device__ __forceinline__ uint32_t lanemask_lt() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Exclusive scan of one value per thread over a 256-thread block.
__device__ __forceinline__ uint32_t block_excl_scan_256(uint32_t v, uint32_t* s_w) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_w[w] = x;
    __syncthreads();
    if (w == 0) {
        uint32_t t = lane < 8 ? s_w[lane] : 0u;
        uint32_t inc = t;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
            uint32_t y = __shfl_up_sync(kFull, inc, o);
            if (lane >= o) inc += y;
        }
        if (lane < 8) s_w[lane] = inc - t;
    }
    __syncthreads();
    uint32_t r = x - v + s_w[w];
    __syncthreads();
    return r;
}

// Lanes of `act` whose 8-bit digit equals this lane's: one ballot per bit.
// (__match_any_sync steps through the distinct values, about 30 for random
// digits.)
__device__ __forceinline__ uint32_t same_digit(uint32_t d, uint32_t act) {
    uint32_t peers = act;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const bool bit = (d >> b) & 1u;
        const uint32_t set = __ballot_sync(kFull, bit);
        peers &= bit ? set : ~set;
    }
    return peers;
}

// One round of a warp's stable ranking: the rank of this lane's digit among
// the warp's keys so far (cnt: the warp's digit counts, updated).
__device__ __forceinline__ uint32_t rank_round(uint32_t d, bool ok, uint32_t* cnt) {
    const uint32_t peers = same_digit(d, __ballot_sync(kFull, ok));
    uint32_t prev = 0;
    if (ok) prev = cnt[d];
    __syncwarp();
    if (ok && (peers & lanemask_lt()) == 0u) cnt[d] = prev + __popc(peers);
    __syncwarp();
    return prev + __popc(peers & lanemask_lt());
}

__host__ __device__ __forceinline__ uint32_t digit_mask(int pass, int bits_total) {
    int b = bits_total - 8 * pass;
    b = b > 8 ? 8 : (b < 0 ? 0 : b);
    return (1u << b) - 1u;
}

// Digit counts of each tile: cnt[tile * 256 + d] for few tiles, else in the
// scan's order, cnt[d * tiles + tile]; *clear (may be null) becomes 0.  Two copies in shared memory (even and
// odd warps), four keys per load where the input is 16-byte aligned.
__global__ void __launch_bounds__(kOsThreads) k_tile_counts(const uint32_t* __restrict__ keys,
                                                            uint32_t n, int shift, uint32_t dmask,
                                                            uint32_t tiles,
                                                            uint32_t* __restrict__ cnt,
                                                            uint32_t* clear) {
    __shared__ uint32_t sh[2][256];
    if (clear && blockIdx.x == 0 && threadIdx.x == 0) *clear = 0u;
    sh[0][threadIdx.x] = 0u;
    sh[1][threadIdx.x] = 0u;
    __syncthreads();
    uint32_t* my = sh[(threadIdx.x >> 5) & 1];
    const uint32_t t0 = blockIdx.x * kOsTile;
    if (((uintptr_t)keys % 16u) == 0u && n - t0 >= (uint32_t)kOsTile) {
        uint4 k[kOsItems / 4];
#pragma unroll
        for (int r = 0; r < kOsItems / 4; ++r)
            k[r] = __ldg(reinterpret_cast<const uint4*>(keys + t0) + r * kOsThreads + threadIdx.x);
#pragma unroll
        for (int r = 0; r < kOsItems / 4; ++r) {
            atomicAdd(&my[(k[r].x >> shift) & dmask], 1u);
            atomicAdd(&my[(k[r].y >> shift) & dmask], 1u);
            atomicAdd(&my[(k[r].z >> shift) & dmask], 1u);
            atomicAdd(&my[(k[r].w >> shift) & dmask], 1u);
        }
    } else {
        for (uint32_t i = t0 + threadIdx.x; i < n && i < t0 + kOsTile; i += kOsThreads)
            atomicAdd(&my[(keys[i] >> shift) & dmask], 1u);
    }
    __syncthreads();
    const uint32_t c = sh[0][threadIdx.x] + sh[1][threadIdx.x];
    cnt[tiles <= kFewTiles ? blockIdx.x * 256u + threadIdx.x
                           : (size_t)threadIdx.x * tiles + blockIdx.x] = c;
}

// Exclusive scan of each digit's counts over the tiles, in place, one block per
// digit; its total to tot[d].  (The scatter's blocks add up the digits before
// theirs.  One scan over all counts with a look-back between its tiles took
// twice as long, 9 us for 977 tiles.)
__global__ void __launch_bounds__(kOsThreads) k_digit_scan(uint32_t* __restrict__ cnt, uint32_t tiles,
                                                           uint32_t* __restrict__ tot) {
    __shared__ uint32_t s_w[8];
    __shared__ uint32_t s_carry;
    uint32_t* c = cnt + (size_t)blockIdx.x * tiles;
    if (threadIdx.x == 0) s_carry = 0u;
    __syncthreads();
    for (uint32_t t0 = 0; t0 < tiles; t0 += kOsThreads * 4) {
        const uint32_t i = t0 + threadIdx.x * 4;
        uint32_t v[4], sum = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[k] = i + k < tiles ? c[i + k] : 0u;
            sum += v[k];
        }
        const uint32_t carry = s_carry;
        uint32_t run = carry + block_excl_scan_256(sum, s_w);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (i + k < tiles) c[i + k] = run;
            run += v[k];
        }
        if (threadIdx.x == kOsThreads - 1) s_carry = run;
        __syncthreads();
    }
    if (threadIdx.x == 0) tot[blockIdx.x] = s_carry;
}

// The scatter of one digit place.  tab: the tiles' counts (FEW tiles) or
// their scans per digit, tot the digits' totals.  Keys of a tile are ranked per
// warp (rounds of 32 in input order), moved to the tile's sorted order in shared
// memory and written from there in runs.
// (FEW as a run-time branch cost the other form 4%: 20M pairs, 24-bit keys, 382 us on
// the device against 397.)
template <bool FEW>
__global__ void __launch_bounds__(kOsThreads, 4) k_radix_scatter(
    const uint32_t* __restrict__ kin, const uint32_t* __restrict__ vin,
    uint32_t* __restrict__ kout, uint32_t* __restrict__ vout, uint32_t n, int shift,
    uint32_t dmask, uint32_t tiles, const uint32_t* __restrict__ tab,
    const uint32_t* __restrict__ tot) {
    constexpr int W = kOsThreads / 32;
    __shared__ uint32_t s_wh[W][256];       // per-warp digit counts, then offsets
    __shared__ uint32_t s_run[256];         // global first slot of the digit's run, less its
                                            // first slot in the tile
    __shared__ uint32_t s_w[8];
    __shared__ uint32_t s_keys[kOsTile];
    __shared__ uint32_t s_vals[kOsTile];

    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const uint32_t tile = blockIdx.x;
    const uint32_t base = tile * kOsTile + w * (kOsItems * 32);
    uint32_t k[kOsItems];
#pragma unroll
    for (int r = 0; r < kOsItems; ++r) {
        const uint32_t idx = base + r * 32 + lane;
        k[r] = idx < n ? kin[idx] : 0u;
    }
    // the global first slot of digit tid in this tile
    uint32_t before = 0, total = 0;
    if (FEW) {
        for (uint32_t t0 = 0; t0 < tiles; t0 += 16) {   // 16 loads in flight
            uint32_t c[16];
#pragma unroll
            for (uint32_t j = 0; j < 16; ++j) c[j] = t0 + j < tiles ? __ldg(tab + (t0 + j) * 256u + tid) : 0u;
#pragma unroll
            for (uint32_t j = 0; j < 16; ++j) {
                before += t0 + j < tile ? c[j] : 0u;
                total += c[j];
            }
        }
    } else {
        before = __ldg(tab + (size_t)tid * tiles + tile);
        total = __ldg(tot + tid);
    }
    const uint32_t first = block_excl_scan_256(total, s_w) + before;
    for (int i = tid; i < W * 256; i += kOsThreads) (&s_wh[0][0])[i] = 0;
    __syncthreads();
    uint32_t rk[kOsItems];
#pragma unroll
    for (int r = 0; r < kOsItems; ++r)
        rk[r] = rank_round((k[r] >> shift) & dmask, base + r * 32 + lane < n, s_wh[w]);
    __syncthreads();
    // Thread tid owns digit tid: the digit's first slot in the tile, and each
    // warp's first slot
    uint32_t run = 0;
#pragma unroll
    for (int ww = 0; ww < W; ++ww) run += s_wh[ww][tid];
    uint32_t slot = block_excl_scan_256(run, s_w);
    s_run[tid] = first - slot;
#pragma unroll
    for (int ww = 0; ww < W; ++ww) {
        const uint32_t c = s_wh[ww][tid];
        s_wh[ww][tid] = slot;
        slot += c;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kOsItems; ++r) {
        const uint32_t idx = base + r * 32 + lane;
        if (idx < n) {
            const uint32_t pos = s_wh[w][(k[r] >> shift) & dmask] + rk[r];
            s_keys[pos] = k[r];
            s_vals[pos] = vin ? vin[idx] : idx;
        }
    }
    __syncthreads();
    const uint32_t t0 = tile * kOsTile;
    const uint32_t nv = (n - t0) < (uint32_t)kOsTile ? (n - t0) : (uint32_t)kOsTile;
#pragma unroll 4
    for (uint32_t i = tid; i < nv; i += kOsThreads) {
        const uint32_t key = s_keys[i];
        const uint32_t g = s_run[(key >> shift) & dmask] + i;
        kout[g] = key;
        vout[g] = s_vals[i];
    }
}

// All digit places of an input of at most one tile, by one block.  The outputs
// may be the inputs (the selection sorts in place): no __restrict__.
__global__ void __launch_bounds__(kOsThreads) k_sort_tile(const uint32_t* kin, const uint32_t* vin,
                                                          uint32_t* kout, uint32_t* vout, uint32_t n,
                                                          int bits_total, uint32_t* clear) {
    if (clear && threadIdx.x == 0) *clear = 0u;
    constexpr int W = kOsThreads / 32;
    __shared__ uint32_t s_wh[W][256];
    __shared__ uint32_t s_w[8];
    __shared__ uint32_t s_keys[kOsTile];
    __shared__ uint32_t s_vals[kOsTile];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    // rounds of 32 keys per warp, the warps' shares consecutive
    const uint32_t rounds = (n + kOsThreads - 1) / kOsThreads;
    const uint32_t base = w * rounds * 32;
    uint32_t k[kOsItems], v[kOsItems], rk[kOsItems];
#pragma unroll
    for (int r = 0; r < kOsItems; ++r) {
        const uint32_t idx = base + r * 32 + lane;
        const bool ok = (uint32_t)r < rounds && idx < n;
        k[r] = ok ? kin[idx] : 0u;
        v[r] = ok ? (vin ? vin[idx] : idx) : 0u;
    }
    for (int shift = 0; shift < bits_total; shift += 8) {
        const uint32_t dmask = digit_mask(shift / 8, bits_total);
        for (int i = tid; i < W * 256; i += kOsThreads) (&s_wh[0][0])[i] = 0;
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kOsItems; ++r)
            if ((uint32_t)r < rounds)
                rk[r] = rank_round((k[r] >> shift) & dmask, base + r * 32 + lane < n, s_wh[w]);
        __syncthreads();
        uint32_t run = 0;
#pragma unroll
        for (int ww = 0; ww < W; ++ww) run += s_wh[ww][tid];
        uint32_t slot = block_excl_scan_256(run, s_w);
#pragma unroll
        for (int ww = 0; ww < W; ++ww) {
            const uint32_t c = s_wh[ww][tid];
            s_wh[ww][tid] = slot;
            slot += c;
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kOsItems; ++r) {
            const uint32_t idx = base + r * 32 + lane;
            if ((uint32_t)r < rounds && idx < n) {
                const uint32_t pos = s_wh[w][(k[r] >> shift) & dmask] + rk[r];
                s_keys[pos] = k[r];
                s_vals[pos] = v[r];
            }
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kOsItems; ++r) {
            const uint32_t idx = base + r * 32 + lane;
            if ((uint32_t)r < rounds && idx < n) {
                k[r] = s_keys[idx];
                v[r] = s_vals[idx];
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int r = 0; r < kOsItems; ++r) {
        const uint32_t idx = base + r * 32 + lane;
        if ((uint32_t)r < rounds && idx < n) {
            kout[idx] = k[r];
            vout[idx] = v[r];
        }
    }
}

// Self-test of the failure path: one warp runs the scan's look-back of tile 1
// against a tile 0 whose word stays zero (nothing publishes it), so the wait
// gives up after `limit` polls.
__global__ void k_lookback_selftest(const unsigned long long* words, uint32_t limit,
                                    uint32_t* err) {
    tile_lookback(words, 1u, 1u, limit, err);
}

// --- exclusive scan of the per-cell counts into cell offsets --------------

constexpr int kScanThreads = 256;
constexpr int kScanItems = 16;
constexpr int kScanChunk = kScanThreads * kScanItems;

__global__ void __launch_bounds__(kScanThreads) k_scan_reduce(const uint32_t* __restrict__ in,
                                                              uint64_t m,
                                                              uint32_t* __restrict__ bsum) {
    pdl_wait();
    __shared__ uint32_t s_w[8];
    const uint64_t b0 = (uint64_t)blockIdx.x * kScanChunk;
    uint32_t s = 0;
    for (int r = 0; r < kScanItems; ++r) {
        const uint64_t i = b0 + (uint64_t)r * kScanThreads + threadIdx.x;
        if (i < m) s += in[i];
    }
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t t = 0;
        for (int i = 0; i < 8; ++i) t += s_w[i];
        bsum[blockIdx.x] = t;
    }
}

// Exclusive scan of the block sums in place (one block).
__global__ void __launch_bounds__(256) k_scan_top(uint32_t* bsum, uint32_t nb) {
    pdl_wait();
    __shared__ uint32_t s_w[8];
    __shared__ uint32_t s_carry;
    if (threadIdx.x == 0) s_carry = 0;
    __syncthreads();
    for (uint32_t c0 = 0; c0 < nb; c0 += 256) {
        const uint32_t i = c0 + threadIdx.x;
        const uint32_t v = i < nb ? bsum[i] : 0u;
        const uint32_t ex = block_excl_scan_256(v, s_w);
        const uint32_t carry = s_carry;
        if (i < nb) bsum[i] = carry + ex;
        __syncthreads();
        if (threadIdx.x == 255) s_carry = carry + ex + v;
        __syncthreads();
    }
}

// out[i] = sum of in[0..i), i = 0..m (m + 1 outputs); clears in[] for the
// next use.
__global__ void __launch_bounds__(kScanThreads) k_scan_down(uint32_t* __restrict__ in, uint64_t m,
                                                            const uint32_t* __restrict__ bsum,
                                                            uint32_t* __restrict__ out,
                                                            int zero_in) {
    pdl_wait();
    __shared__ uint32_t s_w[8];
    const uint64_t b0 = (uint64_t)blockIdx.x * kScanChunk;
    const uint64_t t0 = b0 + (uint64_t)threadIdx.x * kScanItems;
    uint32_t v[kScanItems];
    uint32_t tot = 0;
#pragma unroll
    for (int r = 0; r < kScanItems; ++r) {
        const uint64_t i = t0 + r;
        v[r] = i < m ? in[i] : 0u;
        tot += v[r];
    }
    const uint32_t ex = block_excl_scan_256(tot, s_w) + (bsum ? bsum[blockIdx.x] : 0u);
    uint32_t run = ex;
#pragma unroll
    for (int r = 0; r < kScanItems; ++r) {
        const uint64_t i = t0 + r;
        if (i < m) {
            out[i] = run;
            if (zero_in) in[i] = 0u;
        }
        if (i == m) out[m] = run;
        run += v[r];
    }
}

// The same scan in one launch: tiles of kScanChunk entries taken in launch
// order from a ticket (ctl[0]), each publishing its total, finding the sum
// of the tiles before it by a decoupled look-back (tile_lookback, epoch in
// ctl[1]) and publishing its inclusive prefix.  The block of the last tile
// rearms the ticket and the epoch: its look-back ended on a prefix, so every
// tile has taken its ticket and read the epoch by then.
constexpr uint32_t kScanSpinLimit = 1u << 20;   // polls of a tile's look-back

__global__ void __launch_bounds__(kScanThreads) k_scan_onepass(uint32_t* __restrict__ in,
                                                               uint64_t m,
                                                               uint32_t* __restrict__ out,
                                                               int zero_in,
                                                               unsigned long long* words,
                                                               uint32_t* ctl, uint32_t* err) {
    pdl_wait();
    __shared__ uint32_t s_w[8];
    __shared__ uint32_t s_tile, s_ep, s_tot, s_excl;
    if (threadIdx.x == 0) {
        s_tile = atomicAdd(ctl, 1u);
        s_ep = *reinterpret_cast<volatile uint32_t*>(ctl + 1) & 0x3fffffffu;
    }
    __syncthreads();
    const uint32_t tile = s_tile, ep = s_ep;
    const uint64_t t0 = (uint64_t)tile * kScanChunk + (uint64_t)threadIdx.x * kScanItems;
    uint32_t v[kScanItems];
    uint32_t tot = 0;
#pragma unroll
    for (int r = 0; r < kScanItems; ++r) {
        const uint64_t i = t0 + r;
        v[r] = i < m ? in[i] : 0u;
        tot += v[r];
    }
    const uint32_t ex = block_excl_scan_256(tot, s_w);
    if (threadIdx.x == kScanThreads - 1) s_tot = ex + tot;
    __syncthreads();
    if (threadIdx.x < 32) {
        const uint32_t btot = s_tot;
        const unsigned long long tag = (unsigned long long)ep << 34;
        uint32_t excl = 0;
        if (tile > 0) {
            if (threadIdx.x == 0) st_relaxed64(words + tile, tag | (1ull << 32) | btot);
            excl = tile_lookback(words, tile, ep, kScanSpinLimit, err);
        }
        if (threadIdx.x == 0) {
            st_relaxed64(words + tile, tag | (2ull << 32) | (excl + btot));
            s_excl = excl;
            if ((uint64_t)tile == m / kScanChunk) {   // the tile that holds index m
                ctl[0] = 0u;
                ctl[1] = ep + 1u;
            }
        }
    }
    __syncthreads();
    uint32_t run = s_excl + ex;
#pragma unroll
    for (int r = 0; r < kScanItems; ++r) {
        const uint64_t i = t0 + r;
        if (i < m) {
            out[i] = run;
            if (zero_in) in[i] = 0u;
        }
        if (i == m) out[m] = run;
        run += v[r];
    }
}

}  // namespace

void launch_scan_onepass(uint32_t* in, uint64_t m, uint32_t* out, bool zero_in,
                         unsigned long long* words, uint32_t* ctl, uint32_t* err,
                         cudaStream_t st) {
    launch_pdl(k_scan_onepass, scan_bsum_count(m), kScanThreads, 0, st, in, m, out,
               zero_in ? 1 : 0, words, ctl, err);
}

uint32_t scan_bsum_count(uint64_t m) {
    // m + 1 outputs: the block that holds index m writes the total
    return (uint32_t)((m + 1 + kScanChunk - 1) / kScanChunk);
}

void launch_scan(uint32_t* in, uint64_t m, uint32_t* bsum, uint32_t* out, cudaStream_t st,
                 bool zero_in) {
    const uint32_t nb = scan_bsum_count(m);
    if (nb == 1) {
        // one block holds the whole array: no block sums needed
        launch_pdl(k_scan_down, 1, kScanThreads, 0, st, in, m, nullptr, out, zero_in ? 1 : 0);
        return;
    }
    launch_pdl(k_scan_reduce, nb, kScanThreads, 0, st, in, m, bsum);
    launch_pdl(k_scan_top, 1, 256, 0, st, bsum, nb);
    launch_pdl(k_scan_down, nb, kScanThreads, 0, st, in, m, bsum, out, zero_in ? 1 : 0);
}

// The per-cell counts (incl. the excluded bin) stay in cnt: the scatter of
// the cell sort counts them back down to zero.
void launch_scan_cells(const Dev& d, uint32_t* cnt, uint32_t* off, unsigned long long* words,
                       uint32_t* ctl, uint32_t* err, cudaStream_t st) {
    launch_scan_onepass(cnt, (uint64_t)d.ncells + 1, off, false, words, ctl, err, st);
}

// Sec. 3.1 cell sort as one counting-sort pass (a radix sort whose single
// digit is the whole cell label): the label kernel's per-cell counts are the
// histogram, the cell offsets its exclusive scan, and each particle takes a
// slot of its cell's range by a warp-aggregated atomic decrement of its
// cell's count (which leaves the counts at zero for the next rebuild).  The
// order inside a cell is left arbitrary: the reorder ranks every particle by
// id within its cell, which makes the result the (label, id) order.
__global__ void __launch_bounds__(256) k_cell_scatter(const uint32_t* __restrict__ key, uint32_t n,
                                                      const uint32_t* __restrict__ off,
                                                      uint32_t* cnt, uint32_t* __restrict__ kout,
                                                      uint32_t* __restrict__ vout,
                                                      uint32_t* status) {
    pdl_wait();
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = i < n;
    const uint32_t act = __ballot_sync(kFull, valid);
    if (!valid) return;
    const uint32_t k = key[i];
    const uint32_t peers = __match_any_sync(act, k);
    const int leader = __ffs(peers) - 1;
    const uint32_t np = __popc(peers);
    uint32_t old = 0;
    if ((int)(threadIdx.x & 31) == leader) old = atomicSub(cnt + k, np);
    old = __shfl_sync(peers, old, leader);
    const uint32_t slot = off[k] + old - np + __popc(peers & lanemask_lt());
    if (!in_bounds(slot < n, status)) return;
    kout[slot] = k;
    vout[slot] = i;
}

void launch_cell_scatter(const uint32_t* key, uint32_t n, const uint32_t* off, uint32_t* cnt,
                         uint32_t* kout, uint32_t* vout, uint32_t* status, cudaStream_t st) {
    if (n == 0) return;
    launch_pdl(k_cell_scatter, (n + 255) / 256, 256, 0, st, key, n, off, cnt, kout, vout, status);
}

void launch_lookback_selftest(uint32_t* zeroed, uint32_t limit, uint32_t* err, cudaStream_t st) {
    cudaMemsetAsync(zeroed, 0, 4 * sizeof(uint32_t), st);
    k_lookback_selftest<<<1, 32, 0, st>>>(reinterpret_cast<const unsigned long long*>(zeroed), limit,
                                          err);
}

size_t radix_sort_words(uint32_t n) {
    return (size_t)os_tiles(n) * 256 + 256;   // counts, then the digits' totals
}

void launch_radix_sort(const uint32_t* kin, const uint32_t* vin, uint32_t* kout, uint32_t* vout,
                       uint32_t* tk, uint32_t* tv, uint32_t n, int key_bits, uint32_t* words,
                       uint32_t* clear, cudaStream_t st) {
    const uint32_t tiles = os_tiles(n);
    if (tiles == 0) return;
    if (tiles == 1) {
        k_sort_tile<<<1, kOsThreads, 0, st>>>(kin, vin, kout, vout, n, key_bits, clear);
        return;
    }
    uint32_t* cnt = words;
    uint32_t* tot = cnt + (size_t)tiles * 256;
    const int passes = (key_bits + 7) / 8;
    const uint32_t* ck = kin;
    const uint32_t* cv = vin;
    for (int p = 0; p < passes; ++p) {
        // ping-pong so that the last place lands in the outputs
        const bool to_out = ((passes - 1 - p) % 2) == 0;
        uint32_t* ok = to_out ? kout : tk;
        uint32_t* ov = to_out ? vout : tv;
        const uint32_t dm = digit_mask(p, key_bits);
        k_tile_counts<<<tiles, kOsThreads, 0, st>>>(ck, n, 8 * p, dm, tiles, cnt,
                                                      p == 0 ? clear : nullptr);
        if (tiles <= kFewTiles) {
            k_radix_scatter<true><<<tiles, kOsThreads, 0, st>>>(ck, cv, ok, ov, n, 8 * p, dm, tiles,
                                                                cnt, tot);
        } else {
            k_digit_scan<<<256, kOsThreads, 0, st>>>(cnt, tiles, tot);
            k_radix_scatter<false><<<tiles, kOsThreads, 0, st>>>(ck, cv, ok, ov, n, 8 * p, dm, tiles,
                                                                 cnt, tot);
        }
        ck = ok;
        cv = ov;
    }
}

}  // namespace sph
