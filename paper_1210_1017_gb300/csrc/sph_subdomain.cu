// Sub-domain selection of Sec. 4.2-4.3 on one GPU: the data a sub-domain of
// a one-dimensional decomposition along x sends to its neighbours (the edge
// particles that build their halos, or the particles that migrated), found
// the way the paper does it: a labelling kernel, a radix sort of the
// particles by (label, id), and a copy of the labelled ones.
//
// Only the labelled particles are ordered.  While every id is below n (and
// no two of a label are equal), their order is that of two bit maps over the ids,
// one per label: the labelling kernel sets a particle's bit and notes its state
// index under its label and id, one pass sums the maps' bits per block and one
// lists the state indexes in (label, id) order and clears the maps.  Other ids are sorted: the labelling kernel
// compacts the labelled particles (their slots come from a warp-aggregated
// counter, so their order is arbitrary), a sort by id and a stable one by
// label then give the (label, id) order of the paper's worked example for any
// 32-bit ids.  (The maps cost a pass over n / 4 bytes whatever the number
// selected; 2.1M particles, device destinations: 67 us a call, 141 with sorts.)  The state itself keeps its cell order.
#include <string.h>

#include "sph_ctx.cuh"

namespace sph {

namespace {

constexpr uint32_t kFull = 0xffffffffu;
constexpr uint32_t kIdxBits = 26;                     // state index < 2^26
constexpr uint32_t kIdxMask = (1u << kIdxBits) - 1u;

// Order-preserving integer image of a finite double: a < b exactly when
// ordered(a) < ordered(b), with -0 and +0 both 0.  The labels compare these
// on the integer pipe (GB300 issues FP64 instructions at 1/64 of the FP32
// rate, which would bound this pass instead of HBM).
__host__ __device__ __forceinline__ long long ordered(long long bits) {
    const long long mag = bits & 0x7fffffffffffffffLL;
    return bits < 0 ? -mag : mag;
}

struct SubLabelArgs {
    const double* x;
    const uint32_t* id;
    const uint32_t* off;      // cell offsets: off[ncells] = in-domain count
    uint32_t ncells, n;
    int mode;
    long long xlo, xhi, lo_edge, hi_edge;   // ordered images of the bounds
    uint32_t* key;            // id of each selected particle
    uint32_t* val;            // (label << 26) | state index
                              // (maps: state index by id, val label 1, key label 2)
    uint32_t* cnt;            // [0] in-domain count, [1..2] per label, [3] selected,
                              // [4] not 0: a bit was set twice
    uint32_t* bits;           // bit maps of the ids, label 1 then label 2; null: compact
    uint32_t words;           // words per map
};

constexpr int kLabelItems = 4;   // state entries per thread, their loads in flight together

// Labels of the state entries (in-domain entries k < off[ncells] only).  Only
// warps holding labelled particles touch the counters (label 0 is the rest
// of the in-domain count), so the pass stays a read of x.
__global__ void __launch_bounds__(256) k_sub_label(const SubLabelArgs a) {
    const uint32_t k0 = blockIdx.x * (256 * kLabelItems) + threadIdx.x;
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t n_in = a.off[a.ncells];
    if (k0 == 0) a.cnt[0] = n_in;
    long long x[kLabelItems];
#pragma unroll
    for (int j = 0; j < kLabelItems; ++j) {
        const uint32_t k = k0 + j * 256;
        x[j] = k < n_in ? ordered(__double_as_longlong(a.x[k])) : 0;
    }
#pragma unroll
    for (int j = 0; j < kLabelItems; ++j) {
        const uint32_t k = k0 + j * 256;
        uint32_t l = 0;
        if (k < n_in) {
            if (a.mode == SPH_SUBDOMAIN_EDGE) {
                if (x[j] >= a.xlo && x[j] < a.lo_edge) l = 1;
                else if (x[j] >= a.hi_edge && x[j] < a.xhi) l = 2;
            } else {
                if (x[j] < a.xlo) l = 1;
                else if (x[j] >= a.xhi) l = 2;
            }
        }
        const uint32_t m1 = __ballot_sync(kFull, l == 1u);
        const uint32_t m2 = __ballot_sync(kFull, l == 2u);
        const uint32_t sel = m1 | m2;
        if (sel == 0u) continue;                     // warp-uniform
        uint32_t base = 0;
        if (lane == 0) {
            if (m1) atomicAdd(a.cnt + 1, __popc(m1));
            if (m2) atomicAdd(a.cnt + 2, __popc(m2));
            base = atomicAdd(a.cnt + 3, __popc(sel));
        }
        if (a.bits) {
            if (l != 0u) {
                const uint32_t id = a.id[k];
                const uint32_t bit = 1u << (id & 31u);
                if (atomicOr(a.bits + (size_t)(l - 1u) * a.words + (id >> 5), bit) & bit)
                    atomicOr(a.cnt + 4, 1u);
                (l == 1u ? a.val : a.key)[id] = k;
            }
        } else {
            base = __shfl_sync(kFull, base, 0);
            if (l != 0u) {
                const uint32_t slot = base + __popc(sel & ((1u << lane) - 1u));
                a.key[slot] = a.id[k];
                a.val[slot] = (l << kIdxBits) | k;
            }
        }
    }
}

// Bits of one thread's eight words of the maps (m words in all).
struct BitWords {
    uint32_t w[8];
    uint32_t pop;
};
__device__ __forceinline__ BitWords load_bits(const uint32_t* bits, uint32_t m) {
    BitWords b;
    b.pop = 0;
    const uint32_t i0 = blockIdx.x * kBitWords + threadIdx.x * 8;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        b.w[j] = i0 + j < m ? bits[i0 + j] : 0u;
        b.pop += __popc(b.w[j]);
    }
    return b;
}

// Set bits per block of the maps.
__global__ void __launch_bounds__(256) k_sub_sums(const uint32_t* __restrict__ bits, uint32_t m,
                                                  uint32_t* __restrict__ bsum) {
    __shared__ uint32_t s_w[8];
    const uint32_t t = __reduce_add_sync(kFull, load_bits(bits, m).pop);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t s = 0;
        for (int k = 0; k < 8; ++k) s += s_w[k];
        bsum[blockIdx.x] = s;
    }
}

// State indexes of the set bits in map order: sidx[rank of the bit] = by_id1[id]
// in the map of label 1, by_id2[id] in that of label 2.  Leaves the maps clear.
__global__ void __launch_bounds__(256) k_sub_list(uint32_t* bits, uint32_t m, uint32_t words,
                                                  const uint32_t* __restrict__ bsum,
                                                  const uint32_t* __restrict__ by_id1,
                                                  const uint32_t* __restrict__ by_id2,
                                                  uint32_t* __restrict__ sidx) {
    __shared__ uint32_t s_b[8], s_w[8];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (bsum[blockIdx.x] == 0u) return;              // block-uniform
    uint32_t before = 0;
    for (uint32_t b = threadIdx.x; b < blockIdx.x; b += 256) before += __ldg(bsum + b);
    before = __reduce_add_sync(kFull, before);
    const BitWords b = load_bits(bits, m);
    uint32_t incl = b.pop;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) s_w[w] = incl;
    if (lane == 0) s_b[w] = before;
    __syncthreads();
    uint32_t slot = incl - b.pop;
#pragma unroll
    for (int k = 0; k < 8; ++k) slot += s_b[k] + (k < w ? s_w[k] : 0u);
    const uint32_t i0 = blockIdx.x * kBitWords + threadIdx.x * 8;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const uint32_t i = i0 + j, id0 = 32u * (i < words ? i : i - words);
        const uint32_t* by_id = i < words ? by_id1 : by_id2;
        for (uint32_t q = b.w[j]; q; q &= q - 1u) sidx[slot++] = by_id[id0 + __ffs(q) - 1];
        if (b.w[j]) bits[i] = 0u;
    }
}

// Keys and values of the second (label) sort from the id-sorted pairs.
__global__ void __launch_bounds__(256) k_sub_relabel(const uint32_t* __restrict__ val_in,
                                                     uint32_t m, uint32_t* __restrict__ key_out,
                                                     uint32_t* __restrict__ val_out) {
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < m) {
        const uint32_t v = val_in[t];
        key_out[t] = v >> kIdxBits;
        val_out[t] = v & kIdxMask;
    }
}

// Copy of the selected particles' state in the sorted order.
__global__ void __launch_bounds__(256) k_sub_gather(const uint32_t* __restrict__ sidx, uint32_t m,
                                                    const double* __restrict__ x,
                                                    const double* __restrict__ y,
                                                    const double* __restrict__ z,
                                                    const float4* __restrict__ vr,
                                                    const uint32_t* __restrict__ id,
                                                    double* __restrict__ pos3,
                                                    float* __restrict__ vel3,
                                                    float* __restrict__ rho,
                                                    uint32_t* __restrict__ ids) {
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < m) {
        const uint32_t k = sidx[t];
        pos3[3 * (size_t)t + 0] = x[k];
        pos3[3 * (size_t)t + 1] = y[k];
        pos3[3 * (size_t)t + 2] = z[k];
        const float4 v = vr[k];
        vel3[3 * (size_t)t + 0] = v.x;
        vel3[3 * (size_t)t + 1] = v.y;
        vel3[3 * (size_t)t + 2] = v.z;
        rho[t] = v.w;
        ids[t] = id[k];
    }
}

inline uint32_t blocks256(uint32_t n) { return n ? (n + 255u) / 256u : 1u; }

}  // namespace

}  // namespace sph

using namespace sph;

extern "C" int sph_subdomain_select(sph_ctx* c, int mode, double xlo, double xhi,
                                    uint32_t* counts, uint32_t capacity, double* pos, float* vel,
                                    float* rho, uint32_t* ids) {
    const TraceRange trace("sph_subdomain_select");
    if (!c) return SPH_ERR_INVALID_ARG;
    if (!counts) return fail(c, SPH_ERR_INVALID_ARG, "NULL counts");
    if (mode != SPH_SUBDOMAIN_EDGE && mode != SPH_SUBDOMAIN_MIGRATE)
        return fail(c, SPH_ERR_INVALID_ARG, "unknown sub-domain mode");
    if (!(xhi > xlo)) return fail(c, SPH_ERR_INVALID_ARG, "empty sub-domain");
    const double cs = 2.0 * c->p.h;
    if (mode == SPH_SUBDOMAIN_EDGE && !(xhi - xlo >= 2.0 * cs))
        return fail(c, SPH_ERR_INVALID_ARG, "sub-domain narrower than its two edges (4h)");
    if (c->n_inst != 1) return fail(c, SPH_ERR_STATE, "sub-domains of a single simulation only");
    if (!c->have_state || !c->cells_valid) return fail(c, SPH_ERR_STATE, "cells not built");
    cudaStream_t st = c->st;
    const uint32_t n = c->n;

    SubLabelArgs la;
    la.x = c->x[c->cur];
    la.id = c->id[c->cur];
    la.off = c->off;
    la.ncells = (uint32_t)c->ncells;
    la.n = n;
    la.mode = mode;
    // xlo + 2h and xhi - 2h rounded once in FP64, then mapped
    const double bounds[4] = {xlo, xhi, xlo + cs, xhi - cs};
    long long ob[4];
    for (int i = 0; i < 4; ++i) {
        long long b;
        memcpy(&b, &bounds[i], sizeof(b));
        ob[i] = ordered(b);
    }
    la.xlo = ob[0];
    la.xhi = ob[1];
    la.lo_edge = ob[2];
    la.hi_edge = ob[3];
    la.key = c->sub_key[0];
    la.val = c->sub_val[0];
    la.cnt = c->sub_cnt;
    la.words = (n + 31u) / 32u;
    const uint32_t map_words = 2u * la.words, map_blocks = sub_bit_blocks(n);
    // ids all below n: bit maps; two equal ids of one label: sort.  (Nothing but
    // the labels before the counts are here: a selection that is empty ends then.)
    bool maps = c->ids_dense && !c->ids_pending;
    uint32_t cnt[5];
    for (;;) {
        la.bits = maps ? c->sub_bits : nullptr;
        // the counters, and with them the maps behind, unless the last call left
        // them clear (20 us instead of 26 for an empty selection of 92k particles)
        const size_t clear = maps && !c->sub_clear ? (size_t)(c->sub_bits - c->sub_cnt) + map_words : 5u;
        cudaMemsetAsync(c->sub_cnt, 0, clear * sizeof(uint32_t), st);
        if (maps) c->sub_clear = false;
        k_sub_label<<<(n + 256 * kLabelItems - 1) / (256 * kLabelItems), 256, 0, st>>>(la);
        int rc = cuda_check(c, cudaGetLastError(), "sub-domain labels");
        if (rc) return rc;
        memset(cnt, 0, sizeof(cnt));
        cudaMemcpyAsync(cnt, c->sub_cnt, sizeof(cnt), cudaMemcpyDeviceToHost, st);
        rc = cuda_check(c, cudaStreamSynchronize(st), "sub-domain counts");
        if (rc) return rc;
        if (!maps || cnt[4] == 0u) break;
        maps = false;
    }
    counts[0] = cnt[0] - cnt[1] - cnt[2];
    counts[1] = cnt[1];
    counts[2] = cnt[2];
    const uint32_t m = cnt[3];
    if (maps && m == 0) c->sub_clear = true;   // no bit was set
    if (m > capacity) return fail(c, SPH_ERR_CAPACITY, "output capacity below the selected count");
    if (m == 0) return SPH_OK;

    uint32_t* sidx = c->sub_val[1];            // state indexes in (label, id) order
    if (maps) {
        k_sub_sums<<<map_blocks, 256, 0, st>>>(c->sub_bits, map_words, c->sub_bsum);
        k_sub_list<<<map_blocks, 256, 0, st>>>(c->sub_bits, map_words, la.words, c->sub_bsum,
                                               c->sub_val[0], c->sub_key[0], sidx);
        c->sub_clear = cudaPeekAtLastError() == cudaSuccess;
    } else {
        // sort A: by id (four places, in place); sort B: stable by label
        launch_radix_sort(c->sub_key[0], c->sub_val[0], c->sub_key[0], c->sub_val[0], c->sub_key[1],
                          c->sub_val[1], m, 32, c->sub_os, nullptr, st);
        k_sub_relabel<<<blocks256(m), 256, 0, st>>>(c->sub_val[0], m, c->sub_key[1], c->sub_val[1]);
        launch_radix_sort(c->sub_key[1], c->sub_val[1], c->sub_key[0], c->sub_val[0], nullptr,
                          nullptr, m, 2, c->sub_os, nullptr, st);
        sidx = c->sub_val[0];
    }
    // gather straight into destinations on this device, else into the
    // transfer staging (ids into the free key buffer)
    const size_t m3 = 3 * (size_t)m;
    const bool dp = on_this_device(pos, m3), dv = on_this_device(vel, m3),
               dr = on_this_device(rho, m), di = on_this_device(ids, m);
    double* spos = dp ? pos : c->stage_pos;
    float* svel = dv ? vel : c->stage_vr;
    float* srho = dr ? rho : c->stage_vr + 3 * (size_t)n;
    uint32_t* sids = di ? ids : c->sub_key[1];
    k_sub_gather<<<blocks256(m), 256, 0, st>>>(sidx, m, c->x[c->cur], c->y[c->cur], c->z[c->cur],
                                               c->vr[c->cur], c->id[c->cur], spos, svel, srho, sids);
    const int rc = cuda_check(c, cudaGetLastError(), "sub-domain order and gather");
    if (rc) return rc;
    // cudaMemcpyDefault: host or device destinations (unified addressing)
    if (pos && !dp) cudaMemcpyAsync(pos, spos, 3 * (size_t)m * sizeof(double), cudaMemcpyDefault, st);
    if (vel && !dv) cudaMemcpyAsync(vel, svel, 3 * (size_t)m * sizeof(float), cudaMemcpyDefault, st);
    if (rho && !dr) cudaMemcpyAsync(rho, srho, (size_t)m * sizeof(float), cudaMemcpyDefault, st);
    if (ids && !di) cudaMemcpyAsync(ids, sids, (size_t)m * sizeof(uint32_t), cudaMemcpyDefault, st);
    return cuda_check(c, cudaStreamSynchronize(st), "sub-domain copy");
}
