// Linear layers of the surrogate network on the tcgen05 tensor cores:
//   out[m, :] = epilogue( A[m, :] * B^T + bias )     (A: M x K bf16, B: N x K bf16)
// with the epilogues the message-passing network needs (bias, ReLU,
// residual add, the factorised edge-MLP input with gathered node terms, the
// ReLU mask of the backward pass) fused after the tcgen05.ld of the fp32
// accumulator.  Also the weight gradient dW = X^T dY, reduced over rows in
// TMEM per block and then across blocks in a fixed order.
#include <cuda.h>
#include <cuda_bf16.h>

#include <mutex>

#include "sur_gemm.cuh"
#include "sur_internal.cuh"

namespace sur {

namespace {

template <int N>
__device__ __forceinline__ constexpr uint32_t tmem_cols() {
    return N <= 32 ? 32u : (N <= 64 ? 64u : (N <= 128 ? 128u : 256u));
}

// Issue the asynchronous copies of a (128 x K) bf16 tile (rows past nrows
// zero-filled) into the canonical K-major layout; two lanes take the 32 bytes
// of a memory sector, consecutive pairs consecutive rows.
template <int K, int THR = 128>
__device__ __forceinline__ void issue_rows(unsigned char* dst, const __nv_bfloat16* src,
                                           uint32_t row0, uint32_t nrows, uint32_t ld) {
#pragma unroll
    for (int c = threadIdx.x; c < 128 * (K / 8); c += THR) {
        const int r = (c >> 1) & 127, gk = 2 * (c >> 8) + (c & 1);
        const bool ok = row0 + r < nrows;
        const __nv_bfloat16* p = ok ? src + (size_t)(row0 + r) * ld + gk * 8 : src;
        cp_async16(dst + kmajor_offset(r, gk * 8, K), p, ok);
    }
}

__device__ __forceinline__ void unpack8(const uint4& u, float* f) {
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float2 t = __bfloat1622float2(h[q]);
        f[2 * q] = t.x;
        f[2 * q + 1] = t.y;
    }
}

// Epilogue operands of one row and NP columns, in registers: bf16 rows in
// a (residual, ReLU mask, P[src]) and b (Q[dst]); an fp32 row (gradient
// accumulation) spans a then b.
template <int NP>
struct EpiOps {
    uint4 a[NP / 8];
    uint4 b[NP / 8];
};

// NV 16-byte pieces of a row, 32 bytes per load when `wide` (the L1 takes one
// 128-byte line per clock and a thread's row is a line of its own, so halving
// the loads halves that cost).
template <int NV>
__device__ __forceinline__ void load_pieces(uint4* v, const void* row, bool wide) {
    const uint4* p = reinterpret_cast<const uint4*>(row);
    if (wide) {
#pragma unroll
        for (int i = 0; i < NV; i += 2) ld32(p + i, v[i], v[i + 1]);
    } else {
#pragma unroll
        for (int i = 0; i < NV; ++i) v[i] = p[i];
    }
}

template <int N, int NP>
__device__ __forceinline__ void epi_load(EpiOps<NP>& o, const LinearArgs& g, uint32_t m,
                                         uint32_t gi, uint32_t gj, uint32_t ldr, int col0) {
    switch (g.epi) {
        case kEpiEdge1:
            load_pieces<NP / 8>(o.a, g.gp + (size_t)gi * N + col0, g.wide);
            load_pieces<NP / 8>(o.b, g.gq + (size_t)gj * N + col0, g.wide);
            break;
        case kEpiResidual:
        case kEpiReluMask:
            load_pieces<NP / 8>(o.a, g.res + (size_t)m * ldr + col0, g.wide);
            break;
        case kEpiAccum: {
            const float* p = g.out_f32 + (size_t)m * g.ldo + col0;
            load_pieces<NP / 8>(o.a, p, g.wide);
            load_pieces<NP / 8>(o.b, p + NP / 2, g.wide);
            break;
        }
        default: break;
    }
}

// Forward-type GEMM with fused epilogue; persistent over 128-row tiles.  The
// A tile is double-buffered: the copies of the next tile are in flight while
// the tensor cores multiply the current one and the epilogue drains it.
// Block size of k_linear: 256 threads (the two warps sharing a TMEM lane
// quarter split the output columns) when N >= 32, else 128.
template <int N>
__host__ __device__ constexpr int linear_threads() { return N >= 32 ? 256 : 128; }

template <int K, int N>
__global__ void __launch_bounds__(linear_threads<N>(), 1) k_linear(const LinearArgs g) {
    constexpr int THR = linear_threads<N>();
    constexpr int NCOL = N / (THR / 128);             // output columns per thread
    extern __shared__ __align__(128) unsigned char s_raw[];
    __shared__ __align__(16) float s_bias[N];          // read by every row: staged once
    unsigned char* sb = s_raw;                        // N x K (weights)
    unsigned char* sa0 = s_raw + N * K * 2;           // 2 x (128 x K)
    __shared__ __align__(8) uint64_t s_bar;
    __shared__ uint32_t s_tmem;
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    if (w == 0) tmem_alloc(&s_tmem, tmem_cols<N>());
    if (tid == 0) mbar_init1(&s_bar);
    const uint32_t lda = g.lda ? g.lda : (uint32_t)K;
    const uint32_t ldr = g.ldr ? g.ldr : (uint32_t)N;
    const uint32_t ntiles = (g.M + 127) / 128;
    // weights and the first tile
    for (int c = tid; c < N * (K / 8); c += THR) {
        const int r = c % N, gk = c / N;
        cp_async16(sb + kmajor_offset(r, gk * 8, K), g.Bt + (size_t)r * K + gk * 8, true);
    }
    for (int c = tid; c < N; c += THR) s_bias[c] = g.bias ? g.bias[c] : 0.f;
    if (blockIdx.x < ntiles) issue_rows<K, THR>(sa0, g.A, blockIdx.x * 128, g.M, lda);
    cp_async_commit();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    uint32_t phase = 0, buf = 0;
    bool ok = true;
    for (uint32_t tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x, buf ^= 1u) {
        unsigned char* sa = sa0 + buf * (128 * K * 2);
        cp_async_wait_all();
        fence_async_shared();
        __syncthreads();
        if (tid == 0) {
            tc_fence_after();
#pragma unroll
            for (int s = 0; s < K / 16; ++s) {
                const uint64_t ad = smem_desc(sm_addr(sa) + s * 256, kLBO, (K / 8) * 128);
                const uint64_t bd = smem_desc(sm_addr(sb) + s * 256, kLBO, (K / 8) * 128);
                tc_mma(tmem, ad, bd, idesc_bf16(N), s > 0 ? 1u : 0u);
            }
            tc_commit(&s_bar);
        }
        // next tile into the other buffer (its last reader, the previous
        // tile's MMA, has completed)
        const uint32_t next = tile + gridDim.x;
        if (next < ntiles) issue_rows<K, THR>(sa0 + (buf ^ 1u) * (128 * K * 2), g.A, next * 128, g.M, lda);
        cp_async_commit();
        // this thread's row and columns: its epilogue operands load while the MMA runs
        const int wq = w & 3, col0 = (w >> 2) * NCOL;
        const uint32_t m = tile * 128 + wq * 32 + lane;
        const bool valid = m < g.M;
        uint32_t gi = 0, gj = 0;
        if (g.epi == kEpiEdge1 && valid) {
            gi = g.src[m];
            gj = g.dst[m];
        }
        constexpr int NP = NCOL < 128 ? NCOL : 128;   // columns per epilogue pass
        EpiOps<NP> op;
        if (valid) epi_load<N, NP>(op, g, m, gi, gj, ldr, col0);
        const bool got = mbar_wait(&s_bar, phase);
        ok = __syncthreads_and(got) != 0;
        if (!ok) {
            if (tid == 0 && g.status) atomicOr(g.status, 1u);
            break;
        }
        phase ^= 1u;
        tc_fence_after();
#pragma unroll
        for (int h = 0; h < NCOL / NP; ++h) {
            if (h > 0 && valid) epi_load<N, NP>(op, g, m, gi, gj, ldr, col0 + h * NP);
#pragma unroll
            for (int cl = 0; cl < NP; cl += 16) {
                const int c0 = col0 + h * NP + cl;
                alignas(16) float v[16];
                tmem_ld16(tmem + ((uint32_t)(wq * 32) << 16) + c0, v);
                if (!valid) continue;
                if (g.bias) {
                    const float4* b4 = reinterpret_cast<const float4*>(s_bias + c0);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float4 b = b4[q];
                        v[4 * q] += b.x;
                        v[4 * q + 1] += b.y;
                        v[4 * q + 2] += b.z;
                        v[4 * q + 3] += b.w;
                    }
                }
                float t[16], u[16];
                switch (g.epi) {
                    case kEpiEdge1:   // relu(acc + P[src] + Q[dst] + b)
                        unpack8(op.a[cl / 8], t);
                        unpack8(op.a[cl / 8 + 1], t + 8);
                        unpack8(op.b[cl / 8], u);
                        unpack8(op.b[cl / 8 + 1], u + 8);
#pragma unroll
                        for (int i = 0; i < 16; ++i) v[i] = fmaxf(v[i] + t[i] + u[i], 0.f);
                        break;
                    case kEpiRelu:
#pragma unroll
                        for (int i = 0; i < 16; ++i) v[i] = fmaxf(v[i], 0.f);
                        break;
                    case kEpiResidual:
                        unpack8(op.a[cl / 8], t);
                        unpack8(op.a[cl / 8 + 1], t + 8);
#pragma unroll
                        for (int i = 0; i < 16; ++i) v[i] += t[i];
                        break;
                    case kEpiReluMask:   // backward through a ReLU: keep where act > 0
                        unpack8(op.a[cl / 8], t);
                        unpack8(op.a[cl / 8 + 1], t + 8);
#pragma unroll
                        for (int i = 0; i < 16; ++i) v[i] = t[i] > 0.f ? v[i] : 0.f;
                        break;
                    case kEpiAccum:
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const int k = cl / 4 + q;
                            const uint4 x = k < NP / 8 ? op.a[k % (NP / 8)] : op.b[k % (NP / 8)];
                            v[4 * q] += __uint_as_float(x.x);
                            v[4 * q + 1] += __uint_as_float(x.y);
                            v[4 * q + 2] += __uint_as_float(x.z);
                            v[4 * q + 3] += __uint_as_float(x.w);
                        }
                        break;
                    default: break;
                }
                if (g.out_f32) {
                    const uint4* vv = reinterpret_cast<const uint4*>(v);
                    uint4* o = reinterpret_cast<uint4*>(g.out_f32 + (size_t)m * g.ldo + c0);
                    if (g.wide) {
                        stg32(o, vv[0], vv[1]);
                        stg32(o + 2, vv[2], vv[3]);
                    } else {
#pragma unroll
                        for (int q = 0; q < 4; ++q) o[q] = vv[q];
                    }
                }
                if (g.out_bf16) {
                    __nv_bfloat162 hh[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) hh[q] = __floats2bfloat162_rn(v[2 * q], v[2 * q + 1]);
                    const uint4 h0 = *reinterpret_cast<uint4*>(&hh[0]);
                    const uint4 h1 = *reinterpret_cast<uint4*>(&hh[4]);
                    uint4* o = reinterpret_cast<uint4*>(g.out_bf16 + (size_t)m * g.ldo + c0);
                    if (g.wide) {
                        stg32(o, h0, h1);
                    } else {
                        o[0] = h0;
                        o[1] = h1;
                    }
                }
            }
        }
        tc_fence_before();
        __syncthreads();
    }
    cp_async_wait_all();
    __syncthreads();
    if (w == 0) tmem_dealloc(tmem, tmem_cols<N>());
}

// Transposed staging in two halves: the global loads of a (128-row x C)
// tile into registers (each job: 8 rows of one 8-column block), then the
// register transpose into the (C x 128) K-major tile in shared memory.
template <int C>
struct TRegs {
    static constexpr int kJobs = (C / 8) * 16;
    static constexpr int kPer = (kJobs + 127) / 128;
    uint4 v[kPer][8];
};

template <int C>
__device__ __forceinline__ void load_t(TRegs<C>& r, const __nv_bfloat16* src, uint32_t row0,
                                       uint32_t nrows, uint32_t ld) {
#pragma unroll
    for (int jj = 0; jj < TRegs<C>::kPer; ++jj) {
        const int j = threadIdx.x + jj * 128;
        const int cb = j % (C / 8), rg = j / (C / 8);
#pragma unroll
        for (int rr = 0; rr < 8; ++rr) {
            const uint32_t m = row0 + rg * 8 + rr;
            r.v[jj][rr] = make_uint4(0u, 0u, 0u, 0u);
            if (j < TRegs<C>::kJobs && m < nrows)
                r.v[jj][rr] = *reinterpret_cast<const uint4*>(src + (size_t)m * ld + cb * 8);
        }
    }
}

template <int C>
__device__ __forceinline__ void store_t(unsigned char* dst, const TRegs<C>& r) {
#pragma unroll
    for (int jj = 0; jj < TRegs<C>::kPer; ++jj) {
        const int j = threadIdx.x + jj * 128;
        if (j >= TRegs<C>::kJobs) continue;
        const int cb = j % (C / 8), rg = j / (C / 8);
        __nv_bfloat16 t[8][8];
#pragma unroll
        for (int rr = 0; rr < 8; ++rr) {
            const __nv_bfloat16* e = reinterpret_cast<const __nv_bfloat16*>(&r.v[jj][rr]);
#pragma unroll
            for (int cc = 0; cc < 8; ++cc) t[cc][rr] = e[cc];
        }
#pragma unroll
        for (int cc = 0; cc < 8; ++cc)
            *reinterpret_cast<uint4*>(dst + kmajor_offset(cb * 8 + cc, rg * 8, 128)) =
                *reinterpret_cast<const uint4*>(t[cc]);
    }
}

// Weight gradient dW[C x N] = X^T dY over rows [0, M) for N = 16: X is M x C, dY is
// M x N (bf16, row-major).  Block b accumulates the row tiles b, b + grid,
// ... in TMEM (C = 128 rows of the MMA, one MMA chain per tile), then writes
// its partial; k_wgrad_reduce adds the partials in block order.  The loads
// of the next tile are in flight while the tensor cores work on this one.
template <int N>
__global__ void __launch_bounds__(128) k_wgrad(const WgradArgs g) {
    extern __shared__ __align__(128) unsigned char s_raw[];
    unsigned char* sa = s_raw;                  // X^T tile: 128 x 128 (features x rows)
    unsigned char* sb = s_raw + 128 * 128 * 2;  // dY^T tile: N x 128
    __shared__ __align__(8) uint64_t s_bar;
    __shared__ uint32_t s_tmem;
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    if (w == 0) tmem_alloc(&s_tmem, tmem_cols<N>());
    if (tid == 0) mbar_init1(&s_bar);
    const uint32_t ldp = g.ldp ? g.ldp : 128u, ldq = g.ldq ? g.ldq : (uint32_t)N;
    const uint32_t ntiles = (g.M + 127) / 128;
    TRegs<128> rx;
    TRegs<N> ry;
    if (blockIdx.x < ntiles) {
        load_t<128>(rx, g.X, blockIdx.x * 128, g.M, ldp);
        load_t<N>(ry, g.dY, blockIdx.x * 128, g.M, ldq);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    uint32_t phase = 0, first = 1;
    bool ok = true;
    for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        store_t<128>(sa, rx);
        store_t<N>(sb, ry);
        fence_async_shared();
        __syncthreads();
        if (tid == 0) {
            tc_fence_after();
#pragma unroll
            for (int s = 0; s < 128 / 16; ++s) {
                const uint64_t ad = smem_desc(sm_addr(sa) + s * 256, kLBO, 16 * 128);
                const uint64_t bd = smem_desc(sm_addr(sb) + s * 256, kLBO, 16 * 128);
                tc_mma(tmem, ad, bd, idesc_bf16(N), (first && s == 0) ? 0u : 1u);
            }
            tc_commit(&s_bar);
        }
        first = 0;
        const uint32_t next = tile + gridDim.x;
        if (next < ntiles) {
            load_t<128>(rx, g.X, next * 128, g.M, ldp);
            load_t<N>(ry, g.dY, next * 128, g.M, ldq);
        }
        const bool got = mbar_wait(&s_bar, phase);
        ok = __syncthreads_and(got) != 0;
        if (!ok) {
            if (tid == 0 && g.status) atomicOr(g.status, 1u);
            break;
        }
        phase ^= 1u;
        tc_fence_before();
        __syncthreads();
    }
    tc_fence_after();
    float* part = g.partial + (size_t)blockIdx.x * 128 * N;
    const uint32_t r = w * 32 + lane;   // feature row of dW
#pragma unroll 1
    for (int c0 = 0; c0 < N; c0 += 16) {
        float v[16];
        tmem_ld16(tmem + ((uint32_t)(w * 32) << 16) + c0, v);
        float4* o = reinterpret_cast<float4*>(part + (size_t)r * N + c0);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const bool z = first || !ok;
            o[q] = z ? make_float4(0.f, 0.f, 0.f, 0.f)
                     : make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (w == 0) tmem_dealloc(tmem, tmem_cols<N>());
}

// The same for N = 128, the rows by TMA: a tile of 128 rows of X and of dY lands
// in shared memory as it lies in memory (feature-contiguous, 128-byte swizzle)
// and is the MMA's operand in that form (both "MN-major": the transposes are the
// descriptors'), so no register ever holds a row.  Three stages of 64 KB keep
// 192 KB in flight per SM: one thread loads, one issues the MMAs.  The tiles of
// a block take turns with four accumulators (the 512 TMEM columns), added in
// FP32 at the end, so no accumulation chain is longer than with the three
// blocks per SM of the register version, and the partials are a third as many.
// Bound by HBM (512 B per row).  On one GB300 with the sum of the partials, us at
// 976k / 250k / 17k rows: 192 / 76 / 22.5 with rows transposed in registers, 98 /
// 39 / 16.4 now (5.1 TB/s, 75% of the copy bandwidth); errors against 64 bits
// 1.5e-8 / 1.4e-8 / 2.1e-8 of the sum of absolute terms before, 1.1e-8 / 5.6e-9 /
// 9.4e-9 now.
constexpr int kWgStages = 3, kWgAcc = 4;
constexpr uint32_t kWgMinTiles = 2;   // tiles per block where there are enough (fewer partials)
constexpr size_t kWgSmem = (size_t)kWgStages * 2 * 32768 + 1024;

// Up to kWgradBatch gradients over the same rows, one per blockIdx.y, and their
// outputs: a small system's rows fill the chip once for all of them, with one
// reduction (a training step of 17k particles and 10 layers: 11.92 -> 11.54 ms
// with the five node gradients of a layer in two launches and its four column
// sums finished in one).
struct WgradMaps {
    CUtensorMap x[kWgradBatch], y[kWgradBatch];
};
struct WgradOuts {
    float* dW[kWgradBatch];
};

__global__ void __launch_bounds__(128, 1)
    k_wgrad_tma(const WgradArgs g, const __grid_constant__ WgradMaps maps) {
    constexpr int N = 128;
    constexpr uint32_t T = 128 * 128 * 2, BOX = T / 2;
    extern __shared__ unsigned char s_dyn[];
    __shared__ __align__(8) uint64_t s_full[kWgStages], s_empty[kWgStages], s_done;
    __shared__ uint32_t s_tmem;
    unsigned char* s_raw = s_dyn + ((1024u - (sm_addr(s_dyn) & 1023u)) & 1023u);
    const int tid = threadIdx.x, w = tid >> 5;
    if (w == 0) tmem_alloc(&s_tmem, 512);
    if (tid == 0) {
        for (int s = 0; s < kWgStages; ++s) {
            mbar_init1(&s_full[s]);
            mbar_init1(&s_empty[s]);
        }
        mbar_init1(&s_done);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    const CUtensorMap *map_x = &maps.x[blockIdx.y], *map_y = &maps.y[blockIdx.y];
    const uint32_t ntiles = (g.M + 127) / 128;
    const uint32_t mine = blockIdx.x < ntiles ? (ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
    bool ok = true;
    if (tid == 0) {                                      // loads
        for (uint32_t i = 0; i < mine && ok; ++i) {
            const uint32_t s = i % kWgStages, use = i / kWgStages;
            if (use > 0) ok = mbar_wait(&s_empty[s], (use - 1) & 1u);
            if (!ok) break;
            unsigned char* x = s_raw + s * 2 * T;
            const int row = (int)((blockIdx.x + i * gridDim.x) * 128);
            mbar_expect(&s_full[s], 2 * T);
            tma_load(x, map_x, 0, row, &s_full[s]);
            tma_load(x + BOX, map_x, 64, row, &s_full[s]);
            tma_load(x + T, map_y, 0, row, &s_full[s]);
            tma_load(x + T + BOX, map_y, 64, row, &s_full[s]);
        }
    } else if (tid == 32) {                              // MMAs
        for (uint32_t i = 0; i < mine && ok; ++i) {
            const uint32_t s = i % kWgStages, use = i / kWgStages;
            ok = mbar_wait(&s_full[s], use & 1u);
            if (!ok) break;
            tc_fence_after();
            const uint32_t x = sm_addr(s_raw + s * 2 * T);
#pragma unroll
            for (int k = 0; k < 8; ++k)                  // 16 rows of the tile each
                tc_mma(tmem + (i % kWgAcc) * N, smem_desc_mn128(x + k * 2048, BOX),
                       smem_desc_mn128(x + T + k * 2048, BOX), idesc_bf16(N) | kIdescMN,
                       (i >= (uint32_t)kWgAcc || k > 0) ? 1u : 0u);
            tc_commit(&s_empty[s]);
        }
        tc_commit(&s_done);
    }
    __syncwarp();
    const bool all = __syncthreads_and(ok) != 0;
    const bool got = mbar_wait(&s_done, 0);              // every MMA issued has completed
    if (!(all && got)) {
        if (tid == 0) {
            if (g.status) atomicOr(g.status, 1u);
            for (int s = 0; s < kWgStages; ++s) {        // let copies in flight land first
                const uint32_t uses = (mine + kWgStages - 1 - s) / kWgStages;
                if (uses) mbar_wait(&s_full[s], (uses - 1) & 1u);
            }
        }
    }
    tc_fence_after();
    const uint32_t used = all && got ? (mine < (uint32_t)kWgAcc ? mine : (uint32_t)kWgAcc) : 0u;
    uint4* o = reinterpret_cast<uint4*>(g.partial + ((size_t)(blockIdx.y * gridDim.x + blockIdx.x) * 128 + tid) * N);
    const uint32_t quarter = (uint32_t)(w * 32) << 16;   // feature row tid of dW
#pragma unroll 1
    for (int c0 = 0; c0 < N; c0 += 16) {
        float v[16] = {};
        for (uint32_t a = 0; a < used; ++a) {
            float t[16];
            tmem_ld16(tmem + quarter + a * N + c0, t);
#pragma unroll
            for (int q = 0; q < 16; ++q) v[q] += t[q];
        }
        const uint4* vv = reinterpret_cast<const uint4*>(v);
#pragma unroll
        for (int q = 0; q < 4; ++q) o[c0 / 4 + q] = vv[q];
    }
    tc_fence_before();
    __syncthreads();
    if (w == 0) tmem_dealloc(tmem, 512);
}

// Adds the partials: 32 outputs per block (128 bytes of each partial), its
// eight warps taking every eighth partial, their sums added in warp order.
__global__ void __launch_bounds__(256) k_wgrad_reduce(const float* __restrict__ partials, int nparts,
                                                      int count, const WgradOuts outs, float scale) {
    __shared__ float s_sum[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int i = blockIdx.x * 32 + lane;
    const float* __restrict__ partial = partials + (size_t)blockIdx.y * nparts * count;
    float s = 0.f;
    if (i < count) {
#pragma unroll 8
        for (int b = w; b < nparts; b += 8) s += partial[(size_t)b * count + i];
    }
    s_sum[w][lane] = s;
    __syncthreads();
    if (w != 0 || i >= count) return;
    s = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) s += s_sum[k][lane];
    outs.dW[blockIdx.y][i] = s * scale;
}

// The network's edge encoder (its two edge layers) in one kernel, per
// 128-edge tile: tcgen05 MMA 1 (x W1, K = 16: the edge features) into X; the
// first epilogue writes z = relu(acc + b1) to TMEM as MMA 2's A operand (and to
// global memory for the backward pass); MMA 2 (z W2) back into X; the second
// epilogue writes e0 = acc + b2 to shared memory in the 128-byte swizzle, from
// where it is stored by TMA.  z never reaches HBM in inference.  X and Y are the
// halves of 256 TMEM columns and change roles from tile to tile, so MMA 1 of
// the next tile runs under this tile's second epilogue.  Bound by HBM: 32 B of
// features in, 256 B out (512 with Z); row stores by thread held the L1 at one
// line per clock.  256 threads, two blocks per SM (77 KB of shared memory): the
// two warps that share a TMEM lane quarter split the columns.
constexpr int kEncK = 16;
constexpr uint32_t kETile = 128 * 128 * 2;                  // bytes of a 128 x 128 bf16 tile
// e0 and W2, then W1 and two x tiles; alignment
constexpr size_t kEncSmem = (size_t)2 * kETile + (size_t)128 * kEncK * 2 * 3 + 1024;

__global__ void __launch_bounds__(256, 2)
    k_edge_encoder(const EdgeArgs g, const __grid_constant__ CUtensorMap map_out, const bool wide) {
    constexpr int K1 = kEncK, N = 128, NT = 256;
    constexpr uint32_t T = kETile, BOX = T / 2;
    constexpr uint32_t T1 = 128 * K1 * 2;          // bytes of one 128 x K1 tile
    extern __shared__ unsigned char s_dyn[];
    unsigned char* so = s_dyn + ((1024u - (sm_addr(s_dyn) & 1023u)) & 1023u);   // e0 tile
    unsigned char* sw2 = so + T;                   // W2^T, N x N
    unsigned char* sw1 = sw2 + T;                  // W1^T, N x K1
    unsigned char* sx0 = sw1 + T1;                 // 2 x x tile
    __shared__ __align__(16) float s_b1[128], s_b2[128];
    __shared__ __align__(8) uint64_t s_bar[2];     // MMA 1, MMA 2
    __shared__ uint32_t s_tmem;
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    if (w == 0) tmem_alloc(&s_tmem, 256);
    if (tid == 0) {
        mbar_init1(&s_bar[0]);
        mbar_init1(&s_bar[1]);
    }
    const uint32_t ntiles = (g.M + 127) / 128;
    for (int c = tid; c < N * (K1 / 8); c += NT) {
        const int r = c % N, gk = c / N;
        cp_async16(sw1 + kmajor_offset(r, gk * 8, K1), g.W1t + (size_t)r * K1 + gk * 8, true);
    }
    for (int c = tid; c < N * (N / 8); c += NT) {
        const int r = c % N, gk = c / N;
        cp_async16(sw2 + kmajor_offset(r, gk * 8, N), g.W2t + (size_t)r * N + gk * 8, true);
    }
    if (tid < 128) {
        s_b1[tid] = g.b1[tid];
        s_b2[tid] = g.b2[tid];
    }
    uint32_t tile = blockIdx.x;
    if (tile < ntiles) issue_rows<K1, NT>(sx0, g.E, tile * 128, g.M, K1);
    cp_async_commit();
    cp_async_wait_all();
    fence_async_shared();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    const int wq = w & 3, part = w >> 2;                 // lane quarter, column half
    const uint32_t quarter = (uint32_t)(wq * 32) << 16;
    const int r = wq * 32 + lane;                        // this thread's row of a tile
    auto mma1 = [&](const unsigned char* sx, uint32_t d) {
        tc_fence_after();
        tc_mma(d, smem_desc(sm_addr(sx), kLBO, (K1 / 8) * 128),
               smem_desc(sm_addr(sw1), kLBO, (K1 / 8) * 128), idesc_bf16(N), 0u);
        tc_commit(&s_bar[0]);
    };
    uint32_t phase = 0, x = 0, buf = 0;                  // x: column offset of X (0 or 128)
    bool ok = true;
    if (tile < ntiles && tid == 0) mma1(sx0, tmem);
    for (; tile < ntiles; tile += gridDim.x) {
        const uint32_t m = tile * 128 + (uint32_t)r;
        const uint32_t next = tile + gridDim.x;
        // the next tile's x into the other buffer (its last reader, MMA 1 of
        // the tile before, has completed)
        if (next < ntiles) issue_rows<K1, NT>(sx0 + (buf ^ 1u) * T1, g.E, next * 128, g.M, K1);
        cp_async_commit();
        bool got = mbar_wait(&s_bar[0], phase);          // MMA 1
        tc_fence_after();
        // epilogue 1: z = relu(acc + b1) into Y, and to Z
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int c0 = part * 64 + 16 * k;
            float v[16];
            tmem_ld16(tmem + x + quarter + c0, v);
            const float4* b4 = reinterpret_cast<const float4*>(s_b1 + c0);
            uint32_t z[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const float4 bb = b4[q >> 1];
                const float2 a = __fadd2_rn(make_float2(v[2 * q], v[2 * q + 1]),
                                            q & 1 ? make_float2(bb.z, bb.w) : make_float2(bb.x, bb.y));
                // rounding and the maximum with 0 commute
                const __nv_bfloat162 zz =
                    __hmax2(__floats2bfloat162_rn(a.x, a.y), __floats2bfloat162_rn(0.f, 0.f));
                z[q] = *reinterpret_cast<const uint32_t*>(&zz);
            }
            tmem_st8(tmem + (x ^ 128u) + quarter + (uint32_t)(c0 / 2), z);
            if (g.Z && m < g.M) {
                uint4* o = reinterpret_cast<uint4*>(g.Z + (size_t)m * N + c0);
                const uint4 z0 = make_uint4(z[0], z[1], z[2], z[3]);
                const uint4 z1 = make_uint4(z[4], z[5], z[6], z[7]);
                if (wide) {
                    stg32(o, z0, z1);
                } else {
                    o[0] = z0;
                    o[1] = z1;
                }
            }
        }
        tmem_st_wait();
        cp_async_wait_all();                             // the next tile's x
        if (tid == 32) bulk_wait_read();                 // the e0 tile has been read
        fence_async_shared();
        tc_fence_before();
        ok = __syncthreads_and(got) != 0;                // z and the next x complete
        if (!ok) break;
        if (tid == 0) {
            tc_fence_after();
#pragma unroll
            for (int s = 0; s < N / 16; ++s) {
                const uint64_t bd = smem_desc(sm_addr(sw2) + s * 256, kLBO, (N / 8) * 128);
                tc_mma_ta(tmem + x, tmem + (x ^ 128u) + s * 8, bd, idesc_bf16(N), s > 0 ? 1u : 0u);
            }
            tc_commit(&s_bar[1]);
        }
        got = mbar_wait(&s_bar[1], phase);               // MMA 2
        tc_fence_after();
        // z has been read: MMA 1 of the next tile over it
        if (got && tid == 0 && next < ntiles) mma1(sx0 + (buf ^ 1u) * T1, tmem + (x ^ 128u));
        // epilogue 2: e0 = acc + b2
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int c0 = part * 64 + 16 * k;
            float v[16];
            tmem_ld16(tmem + x + quarter + c0, v);
            const float4* b4 = reinterpret_cast<const float4*>(s_b2 + c0);
            __nv_bfloat162 hh[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const float4 bb = b4[q >> 1];
                const float2 a = __fadd2_rn(make_float2(v[2 * q], v[2 * q + 1]),
                                            q & 1 ? make_float2(bb.z, bb.w) : make_float2(bb.x, bb.y));
                hh[q] = __floats2bfloat162_rn(a.x, a.y);
            }
            *reinterpret_cast<uint4*>(so + part * BOX + sw128_offset(r, 2 * k)) =
                *reinterpret_cast<uint4*>(&hh[0]);
            *reinterpret_cast<uint4*>(so + part * BOX + sw128_offset(r, 2 * k + 1)) =
                *reinterpret_cast<uint4*>(&hh[4]);
        }
        fence_async_shared();
        tc_fence_before();
        ok = __syncthreads_and(got) != 0;                // X free, e0 complete
        if (!ok) break;
        if (tid == 32) {
            tma_store(&map_out, so, 0, (int)(tile * 128));
            tma_store(&map_out, so + BOX, 64, (int)(tile * 128));
            bulk_commit();
        }
        x ^= 128u;
        buf ^= 1u;
        phase ^= 1u;
    }
    if (!ok) {
        if (tid == 0 && g.status) atomicOr(g.status, 1u);
        mbar_wait(&s_bar[0], phase);                     // let an MMA in flight land first
        mbar_wait(&s_bar[1], phase);
    }
    if (tid == 32) bulk_wait();
    cp_async_wait_all();
    tc_fence_before();
    __syncthreads();
    if (w == 0) tmem_dealloc(tmem, 256);
}

// AND-reduction over the 256 threads of one half of a 512-thread block (named
// barriers 1 and 2).
__device__ __forceinline__ bool half_and(int h, bool v) {
    uint32_t r;
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.and.pred q, %2, 256, p;\n"
        " selp.u32 %0, 1, 0, q;\n}"
        : "=r"(r)
        : "r"((uint32_t)v), "r"(h + 1)
        : "memory");
    return r != 0;
}

// The fused edge update of a message-passing layer, per 128-edge tile:
//   z = relu(e W1c + b1 + P[src] + Q[dst]),  e' = e + z W2 + b2
// as two independent halves of 256 threads that share the weights: half h
// takes the tiles 2 b + h, 2 b + h + 2 grid, ... of block b with its own
// mbarriers, 256 TMEM columns and named barrier, so one half's MMAs, copies
// and barriers overlap the other half's epilogues.
//
// HBM is the floor (e in, e' out: 512 B per edge, 768 with Z), so the loads
// of a tile are in flight before its turn and nothing goes through L1 row by
// row that can go as a tile: with per-thread copies of the e, e' and z rows
// the kernel ran at the L1's rate of one 128-byte line per clock (69% of it,
// 0.68 instructions per clock).  The e tile comes by TMA in the 128-byte
// swizzle, is read by MMA 1 and by the second epilogue (a thread per row: no
// bank conflicts), overwritten in place by e' and stored by TMA.  z is MMA
// 2's A operand in TMEM (tcgen05.st), which leaves shared memory for two e
// tiles per half; the gathered rows go to registers a tile ahead, 32 bytes
// per load.  Accumulators and z alternate between the halves X and Y of the
// 256 columns: MMA 1 of tile t in X, z in Y, MMA 2 back into X, and MMA 1 of
// tile t + 1 into Y as soon as MMA 2 has read z, under tile t's second
// epilogue.  On one GB300, with Z, 1.5M edges: 572 us with the loads issued at
// the end of a tile, 466 with z in TMEM and the loads ahead, 300 with the
// tiles by TMA (3.9 TB/s of e, e' and z, 57% of the copy bandwidth).
constexpr size_t kEdgePPSmem = (size_t)6 * kETile + 1024;   // W1c, W2, 2 x 2 e tiles; alignment

__global__ void __launch_bounds__(512, 1)
    k_edge_pp(const EdgeArgs g, const __grid_constant__ CUtensorMap map_e,
              const __grid_constant__ CUtensorMap map_out, const bool wide) {
    constexpr int N = 128;
    constexpr uint32_t T = kETile, BOX = T / 2;          // a box: 64 columns of 128 rows
    extern __shared__ unsigned char s_dyn[];
    __shared__ __align__(16) float s_b1[128], s_b2[128];
    // completions of MMA 1 and of MMA 2, per half (a barrier each: MMA 1 of the
    // next tile may complete before every thread has seen MMA 2); e tile loaded,
    // per half and buffer
    __shared__ __align__(8) uint64_t s_bar[2][2], s_full[2][2];
    __shared__ uint32_t s_tmem;
    unsigned char* s_raw = s_dyn + ((1024u - (sm_addr(s_dyn) & 1023u)) & 1023u);
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const int h = tid >> 8, lt = tid & 255;              // half, thread within the half
    unsigned char* sw1 = s_raw;                          // W1c^T
    unsigned char* sw2 = s_raw + T;                      // W2^T
    if (w == 0) tmem_alloc(&s_tmem, 512);
    if (tid == 0)
        for (int k = 0; k < 2; ++k) {
            mbar_init1(&s_bar[k][0]);
            mbar_init1(&s_bar[k][1]);
            mbar_init1(&s_full[k][0]);
            mbar_init1(&s_full[k][1]);
        }
    for (int c = tid; c < N * (N / 8); c += 512) {
        const int r = c % N, gk = c / N;
        cp_async16(sw1 + kmajor_offset(r, gk * 8, N), g.W1t + (size_t)r * N + gk * 8, true);
        cp_async16(sw2 + kmajor_offset(r, gk * 8, N), g.W2t + (size_t)r * N + gk * 8, true);
    }
    if (tid < 128) {
        s_b1[tid] = g.b1[tid];
        s_b2[tid] = g.b2[tid];
    }
    cp_async_wait_all();
    fence_async_shared();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t ntiles = (g.M + 127) / 128;
    const uint32_t stride = 2 * gridDim.x;
    unsigned char* se0 = s_raw + (2 + 2 * h) * T;        // this half's two e tiles
    const int wq = w & 3, part = (w >> 2) & 1;           // lane quarter, column half
    const int r = wq * 32 + lane;                        // this thread's row of a tile
    const bool mover = lt == 32;                         // moves the half's tiles
    auto load_e = [&](uint32_t t, uint32_t b) {
        mbar_expect(&s_full[h][b], T);
        tma_load(se0 + b * T, &map_e, 0, (int)(t * 128), &s_full[h][b]);
        tma_load(se0 + b * T + BOX, &map_e, 64, (int)(t * 128), &s_full[h][b]);
    };
    // this thread's 64 columns of a node row (wide: 32-byte aligned rows)
    auto load_row = [&](uint4 (&v)[8], const __nv_bfloat16* rows, uint32_t row, bool ok) {
        const uint4* q = reinterpret_cast<const uint4*>(rows + (size_t)(ok ? row : 0u) * N + part * 64);
        if (wide) {
#pragma unroll
            for (int k = 0; k < 8; k += 2) ldg32(q + k, v[k], v[k + 1]);
        } else {
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = __ldg(q + k);
        }
    };
    uint4 pv[8], qv[8];                                  // P[src], Q[dst] of the tile in hand
    uint32_t tile = 2 * blockIdx.x + (uint32_t)h;
    uint32_t nsrc = 0, ndst = 0;                         // node rows of the half's next tile
    if (tile < ntiles) {
        if (mover) {
            load_e(tile, 0);
            if (tile + stride < ntiles) load_e(tile + stride, 1);
        }
        const uint32_t m0 = tile * 128 + (uint32_t)r, m1 = m0 + stride * 128;
        load_row(pv, g.P, m0 < g.M ? g.src[m0] : 0u, m0 < g.M);
        load_row(qv, g.Q, m0 < g.M ? g.dst[m0] : 0u, m0 < g.M);
        if (tile + stride < ntiles && m1 < g.M) {
            nsrc = g.src[m1];
            ndst = g.dst[m1];
        }
    }
    const uint32_t tmem = s_tmem + (uint32_t)(h * 256);
    const uint32_t quarter = (uint32_t)(wq * 32) << 16;
    // MMA 1 of the e tile in buffer se into accumulator columns d (one thread)
    auto mma1 = [&](const unsigned char* se, uint32_t d) {
        tc_fence_after();
#pragma unroll
        for (int s = 0; s < N / 16; ++s) {
            const uint64_t ad = smem_desc_sw128(sm_addr(se) + (s >> 2) * BOX + (s & 3) * 32);
            const uint64_t bd = smem_desc(sm_addr(sw1) + s * 256, kLBO, (N / 8) * 128);
            tc_mma(d, ad, bd, idesc_bf16(N), s > 0 ? 1u : 0u);
        }
        tc_commit(&s_bar[h][0]);
    };
    uint32_t phase = 0, x = 0, buf = 0, epar = 0;        // x: column offset of X (0 or 128);
                                                         // bit b of epar: phase of s_full[h][b]
    bool ok = true, first = true;
    if (tile < ntiles && lt == 0 && mbar_wait(&s_full[h][0], 0)) mma1(se0, tmem);
    for (; tile < ntiles; tile += stride) {
        unsigned char* se = se0 + buf * T + part * BOX;  // this thread's box of the tile
        const uint32_t m = tile * 128 + (uint32_t)r;
        const uint32_t next = tile + stride;
        bool got = mbar_wait(&s_bar[h][0], phase);       // MMA 1
        tc_fence_after();
        // epilogue 1: z = relu(((acc + b1) + P[src]) + Q[dst]) into Y, and to Z
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            // the next tile's e, once the store of the tile before this one has
            // read that buffer (it has by the middle of this epilogue)
            if (k == 2 && mover && !first && next < ntiles) {
                bulk_wait_read();
                load_e(next, buf ^ 1u);
            }
            if (k == 2) __syncwarp();
            const int c0 = part * 64 + 16 * k;
            float v[16];
            tmem_ld16(tmem + x + quarter + c0, v);
            float t[16], u[16];
            unpack8(pv[2 * k], t);
            unpack8(pv[2 * k + 1], t + 8);
            unpack8(qv[2 * k], u);
            unpack8(qv[2 * k + 1], u + 8);
            const float4* b4 = reinterpret_cast<const float4*>(s_b1 + c0);
            uint32_t z[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const float4 bb = b4[q >> 1];
                float2 s = __fadd2_rn(make_float2(v[2 * q], v[2 * q + 1]),
                                      q & 1 ? make_float2(bb.z, bb.w) : make_float2(bb.x, bb.y));
                s = __fadd2_rn(s, make_float2(t[2 * q], t[2 * q + 1]));
                s = __fadd2_rn(s, make_float2(u[2 * q], u[2 * q + 1]));
                // rounding and the maximum with 0 commute
                const __nv_bfloat162 zz =
                    __hmax2(__floats2bfloat162_rn(s.x, s.y), __floats2bfloat162_rn(0.f, 0.f));
                z[q] = *reinterpret_cast<const uint32_t*>(&zz);
            }
            tmem_st8(tmem + (x ^ 128u) + quarter + (uint32_t)(c0 / 2), z);
            if (g.Z && m < g.M) {
                uint4* o = reinterpret_cast<uint4*>(g.Z + (size_t)m * N + c0);
                const uint4 z0 = make_uint4(z[0], z[1], z[2], z[3]);
                const uint4 z1 = make_uint4(z[4], z[5], z[6], z[7]);
                if (wide) {
                    stg32(o, z0, z1);
                } else {
                    o[0] = z0;
                    o[1] = z1;
                }
            }
        }
        tmem_st_wait();
        tc_fence_before();
        ok = half_and(h, got);                           // z complete
        if (!ok) break;
        if (lt == 0) {
            tc_fence_after();
#pragma unroll
            for (int s = 0; s < N / 16; ++s) {
                const uint64_t bd = smem_desc(sm_addr(sw2) + s * 256, kLBO, (N / 8) * 128);
                tc_mma_ta(tmem + x, tmem + (x ^ 128u) + s * 8, bd, idesc_bf16(N), s > 0 ? 1u : 0u);
            }
            tc_commit(&s_bar[h][1]);
        }
        // the next tile's node rows into registers, the row numbers of the
        // one after
        if (next < ntiles) {
            const bool nok = next * 128 + (uint32_t)r < g.M;
            load_row(pv, g.P, nsrc, nok);
            load_row(qv, g.Q, ndst, nok);
            const uint32_t m2 = (next + stride) * 128 + (uint32_t)r;
            if (next + stride < ntiles && m2 < g.M) {
                nsrc = __ldg(g.src + m2);
                ndst = __ldg(g.dst + m2);
            }
        }
        got = mbar_wait(&s_bar[h][1], phase);            // MMA 2
        tc_fence_after();
        // z has been read: MMA 1 of the next tile over it
        if (got && lt == 0 && next < ntiles) {
            got = mbar_wait(&s_full[h][buf ^ 1u], (epar >> (buf ^ 1u)) & 1u);
            if (got) mma1(se0 + (buf ^ 1u) * T, tmem + (x ^ 128u));
        }
        // this tile's e has long landed (MMA 1 read it): the wait makes it
        // visible to this thread
        got = mbar_wait(&s_full[h][buf], (epar >> buf) & 1u) && got;
        epar ^= 1u << buf;
        // epilogue 2: e' = (acc + b2) + e, over e
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int c0 = part * 64 + 16 * k;
            float v[16];
            tmem_ld16(tmem + x + quarter + c0, v);
            uint4* e0 = reinterpret_cast<uint4*>(se + sw128_offset(r, 2 * k));
            uint4* e1 = reinterpret_cast<uint4*>(se + sw128_offset(r, 2 * k + 1));
            float t[16];
            unpack8(*e0, t);
            unpack8(*e1, t + 8);
            const float4* b4 = reinterpret_cast<const float4*>(s_b2 + c0);
            __nv_bfloat162 hh[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const float4 bb = b4[q >> 1];
                float2 s = __fadd2_rn(make_float2(v[2 * q], v[2 * q + 1]),
                                      q & 1 ? make_float2(bb.z, bb.w) : make_float2(bb.x, bb.y));
                s = __fadd2_rn(s, make_float2(t[2 * q], t[2 * q + 1]));
                hh[q] = __floats2bfloat162_rn(s.x, s.y);
            }
            *e0 = *reinterpret_cast<uint4*>(&hh[0]);
            *e1 = *reinterpret_cast<uint4*>(&hh[4]);
        }
        fence_async_shared();
        tc_fence_before();
        ok = half_and(h, got);                           // X free, e' complete
        if (!ok) break;
        if (mover) {
            tma_store(&map_out, se0 + buf * T, 0, (int)(tile * 128));
            tma_store(&map_out, se0 + buf * T + BOX, 64, (int)(tile * 128));
            bulk_commit();
        }
        first = false;
        x ^= 128u;
        buf ^= 1u;
        phase ^= 1u;
    }
    if (!ok) {
        if (lt == 0 && g.status) atomicOr(g.status, 1u);
        mbar_wait(&s_bar[h][0], phase);                  // let MMAs and copies in flight
        mbar_wait(&s_bar[h][1], phase);                  // land first
        mbar_wait(&s_full[h][0], epar & 1u);
        mbar_wait(&s_full[h][1], (epar >> 1) & 1u);
    }
    if (mover) bulk_wait();
    tc_fence_before();
    __syncthreads();
    if (w == 0) tmem_dealloc(s_tmem, 512);
}

template <int K, int N>
size_t linear_smem() { return (size_t)2 * 128 * K * 2 + (size_t)N * K * 2; }

// Sums of 16 columns over the 32 rows (lanes) of a warp: lane l gets column
// l mod 16, added in a fixed tree (16 shuffles).
__device__ __forceinline__ float warp_colsum16(const float (&v)[16], int lane) {
    float a[8], b[4], c[2], d;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float keep = lane & 8 ? v[i + 8] : v[i], give = lane & 8 ? v[i] : v[i + 8];
        a[i] = keep + __shfl_xor_sync(0xffffffffu, give, 8);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float keep = lane & 4 ? a[i + 4] : a[i], give = lane & 4 ? a[i] : a[i + 4];
        b[i] = keep + __shfl_xor_sync(0xffffffffu, give, 4);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const float keep = lane & 2 ? b[i + 2] : b[i], give = lane & 2 ? b[i] : b[i + 2];
        c[i] = keep + __shfl_xor_sync(0xffffffffu, give, 2);
    }
    d = (lane & 1 ? c[1] : c[0]) + __shfl_xor_sync(0xffffffffu, lane & 1 ? c[0] : c[1], 1);
    return d + __shfl_xor_sync(0xffffffffu, d, 16);
}

// The backward pass of the fused edge update, per 128-edge tile:
//   v = dE + node[src],  dpre = v W2^T where z > 0 and 0 elsewhere,
//   dE = v + dpre W1c^T
// with bf16 copies of v and dpre for the weight gradients and the column sums
// of v (FP32) and dpre for the bias gradients.  Two independent halves of 256
// threads per block, as in k_edge_pp, a thread per row and 64 columns.
//
// Bound by HBM: dE in and out, z in, both copies out, 1,792 B per edge; as five
// kernels (gather, two layers, column sums) the same work moved 3,600 B.  The
// bf16 tiles go by TMA in the 128-byte swizzle (dpre over z in place), the dE
// rows by 32-byte accesses a tile ahead, through registers; v waits in TMEM
// for the second product and is added to it in FP32.  Edges are sorted by src,
// so the lanes of a gathering warp share one or two node rows.  The column
// sums of v come from the rows in registers by shuffles, those of dpre from
// the tile in shared memory, each tile summed for itself first.
// On one GB300, 976k edges: 770 us as five kernels, 401 as one (4.4 TB/s of
// those bytes, 64% of the copy bandwidth).
constexpr size_t kEdgeBwdSmem = (size_t)6 * kETile + 1024;   // W2, W1c, 2 x (v, z) tiles; alignment

__global__ void __launch_bounds__(512, 1)
    k_edge_bwd(const EdgeBwdArgs g, const __grid_constant__ CUtensorMap map_z,
               const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_p,
               const bool wide) {
    constexpr int N = 128;
    constexpr uint32_t T = kETile, BOX = T / 2;          // a box: 64 columns of 128 rows
    extern __shared__ unsigned char s_dyn[];
    // completions of MMA 1 and MMA 2, z tile loaded, per half
    __shared__ __align__(8) uint64_t s_bar[2][2], s_full[2];
    __shared__ uint32_t s_tmem;
    __shared__ float s_ce[2][4][N], s_cp[2][4][N];       // column sums of the half's row groups
    unsigned char* s_raw = s_dyn + ((1024u - (sm_addr(s_dyn) & 1023u)) & 1023u);
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const int h = tid >> 8, lt = tid & 255;              // half, thread within the half
    unsigned char* sw2 = s_raw;                          // W2
    unsigned char* sw1 = s_raw + T;                      // W1c
    unsigned char* sv = s_raw + (2 + 2 * h) * T;         // v as bf16
    unsigned char* sz = sv + T;                          // z, then dpre
    if (w == 0) tmem_alloc(&s_tmem, 512);
    if (tid == 0)
        for (int k = 0; k < 2; ++k) {
            mbar_init1(&s_bar[k][0]);
            mbar_init1(&s_bar[k][1]);
            mbar_init1(&s_full[k]);
        }
    for (int c = tid; c < N * (N / 8); c += 512) {
        const int r = c % N, gk = c / N;
        cp_async16(sw2 + kmajor_offset(r, gk * 8, N), g.W2 + (size_t)r * N + gk * 8, true);
        cp_async16(sw1 + kmajor_offset(r, gk * 8, N), g.W1 + (size_t)r * N + gk * 8, true);
    }
    cp_async_wait_all();
    fence_async_shared();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t ntiles = (g.M + 127) / 128;
    const uint32_t stride = 2 * gridDim.x;
    const int wq = w & 3, part = (w >> 2) & 1;           // lane quarter, column half
    const int r = wq * 32 + lane;                        // this thread's row of a tile
    const bool mover = lt == 32;                         // moves the half's tiles
    const uint32_t quarter = (uint32_t)(wq * 32) << 16;
    const uint32_t tv = s_tmem + (uint32_t)(h * 256) + quarter;       // v
    const uint32_t tx = s_tmem + (uint32_t)(h * 256) + 128u;          // the products
    auto load_z = [&](uint32_t t) {
        mbar_expect(&s_full[h], T);
        tma_load(sz, &map_z, 0, (int)(t * 128), &s_full[h]);
        tma_load(sz + BOX, &map_z, 64, (int)(t * 128), &s_full[h]);
    };
    uint4 dv[16];                                        // dE of the tile in hand: 64 columns
    auto load_de = [&](uint32_t m) {
        const uint4* p = reinterpret_cast<const uint4*>(g.dE + (size_t)(m < g.M ? m : 0u) * N + part * 64);
        if (m >= g.M) {
#pragma unroll
            for (int k = 0; k < 16; ++k) dv[k] = make_uint4(0u, 0u, 0u, 0u);
        } else if (wide) {
#pragma unroll
            for (int k = 0; k < 16; k += 2) ld32(p + k, dv[k], dv[k + 1]);
        } else {
#pragma unroll
            for (int k = 0; k < 16; ++k) dv[k] = p[k];
        }
    };
    // D = A B^T of the tile `a` (128-byte swizzle) and weights `b` (one thread)
    auto mma = [&](const unsigned char* a, const unsigned char* b, uint64_t* bar) {
        tc_fence_after();
#pragma unroll
        for (int s = 0; s < N / 16; ++s) {
            const uint64_t ad = smem_desc_sw128(sm_addr(a) + (s >> 2) * BOX + (s & 3) * 32);
            const uint64_t bd = smem_desc(sm_addr(b) + s * 256, kLBO, (N / 8) * 128);
            tc_mma(tx, ad, bd, idesc_bf16(N), s > 0 ? 1u : 0u);
        }
        tc_commit(bar);
    };
    float ce[4] = {0.f, 0.f, 0.f, 0.f};                  // columns part 64 + 16 k + lane mod 16 of v
    float cp[2] = {0.f, 0.f};                            // columns 2 (lt mod 64) and + 1 of dpre
    uint32_t tile = 2 * blockIdx.x + (uint32_t)h;
    uint32_t row = 0;                                    // node row of this thread's edge
    if (tile < ntiles) {
        if (mover) load_z(tile);
        const uint32_t m = tile * 128 + (uint32_t)r;
        load_de(m);
        if (m < g.M) row = __ldg(g.src + m);
    }
    uint32_t phase = 0;
    bool ok = true;
    for (; tile < ntiles; tile += stride) {
        const uint32_t m = tile * 128 + (uint32_t)r;
        const uint32_t next = tile + stride;
        // v = dE + node[src]: to TMEM, as bf16 to the tile, into the column sums
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            uint4 q[4] = {};
            if (m < g.M) {
                const uint4* p = reinterpret_cast<const uint4*>(g.node + (size_t)row * g.ldn + part * 64 + 16 * k);
                if (wide) {
                    ldg32(p, q[0], q[1]);
                    ldg32(p + 2, q[2], q[3]);
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i) q[i] = __ldg(p + i);
                }
            }
            float v[16];
            uint32_t u[16];
            __nv_bfloat162 hh[8];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint4 e = dv[4 * k + i];
                v[4 * i] = __uint_as_float(e.x) + __uint_as_float(q[i].x);
                v[4 * i + 1] = __uint_as_float(e.y) + __uint_as_float(q[i].y);
                v[4 * i + 2] = __uint_as_float(e.z) + __uint_as_float(q[i].z);
                v[4 * i + 3] = __uint_as_float(e.w) + __uint_as_float(q[i].w);
            }
#pragma unroll
            for (int i = 0; i < 16; ++i) u[i] = __float_as_uint(v[i]);
            tmem_st8(tv + (uint32_t)(part * 64 + 16 * k), u);
            tmem_st8(tv + (uint32_t)(part * 64 + 16 * k + 8), u + 8);
#pragma unroll
            for (int i = 0; i < 8; ++i) hh[i] = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
            *reinterpret_cast<uint4*>(sv + part * BOX + sw128_offset(r, 2 * k)) =
                *reinterpret_cast<uint4*>(&hh[0]);
            *reinterpret_cast<uint4*>(sv + part * BOX + sw128_offset(r, 2 * k + 1)) =
                *reinterpret_cast<uint4*>(&hh[4]);
            ce[k] += warp_colsum16(v, lane);
        }
        tmem_st_wait();
        fence_async_shared();
        tc_fence_before();
        ok = half_and(h, ok);                            // v complete, the products' columns free
        if (!ok) break;
        if (lt == 0) mma(sv, sw2, &s_bar[h][0]);
        if (mover) {
            tma_store(&map_v, sv, 0, (int)(tile * 128));
            tma_store(&map_v, sv + BOX, 64, (int)(tile * 128));
            bulk_commit();
        }
        // the next tile's rows
        if (next < ntiles) {
            const uint32_t m1 = next * 128 + (uint32_t)r;
            load_de(m1);
            row = m1 < g.M ? __ldg(g.src + m1) : 0u;
        }
        bool got = mbar_wait(&s_bar[h][0], phase);
        got = mbar_wait(&s_full[h], phase) && got;
        tc_fence_after();
        // dpre over z
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int c0 = part * 64 + 16 * k;
            float v[16], t[16];
            tmem_ld16(tx + quarter + c0, v);
            uint4* z0 = reinterpret_cast<uint4*>(sz + part * BOX + sw128_offset(r, 2 * k));
            uint4* z1 = reinterpret_cast<uint4*>(sz + part * BOX + sw128_offset(r, 2 * k + 1));
            unpack8(*z0, t);
            unpack8(*z1, t + 8);
            __nv_bfloat162 hh[8];
#pragma unroll
            for (int i = 0; i < 8; ++i)
                hh[i] = __floats2bfloat162_rn(t[2 * i] > 0.f ? v[2 * i] : 0.f,
                                              t[2 * i + 1] > 0.f ? v[2 * i + 1] : 0.f);
            *z0 = *reinterpret_cast<uint4*>(&hh[0]);
            *z1 = *reinterpret_cast<uint4*>(&hh[4]);
        }
        fence_async_shared();
        tc_fence_before();
        ok = half_and(h, got);                           // dpre complete
        if (!ok) break;
        if (lt == 0) mma(sz, sw1, &s_bar[h][1]);
        if (mover) {
            tma_store(&map_p, sz, 0, (int)(tile * 128));
            tma_store(&map_p, sz + BOX, 64, (int)(tile * 128));
            bulk_commit();
        }
        {   // column sums of dpre: two columns and 32 rows per thread
            const uint32_t pr = (uint32_t)lt & 63u, r0 = (uint32_t)(lt >> 6) * 32u;
            const unsigned char* col = sz + (pr >> 5) * BOX + (pr & 3u) * 4u;
            float s0 = 0.f, s1 = 0.f;
#pragma unroll 8
            for (uint32_t i = 0; i < 32; ++i) {
                const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(
                    col + sw128_offset(r0 + i, (pr & 31u) >> 2)));
                s0 += f.x;
                s1 += f.y;
            }
            cp[0] += s0;
            cp[1] += s1;
        }
        got = mbar_wait(&s_bar[h][1], phase);
        tc_fence_after();
        if (mover) bulk_wait_read();                     // both copies have been read
        ok = half_and(h, got);                           // the tiles are free
        if (!ok) break;
        if (mover && next < ntiles) load_z(next);
        // dE = v + dpre W1c^T
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int c0 = part * 64 + 16 * k;
            float v[16], x[16];
            tmem_ld16(tv + c0, v);
            tmem_ld16(tx + quarter + c0, x);
            if (m < g.M) {
                uint4 o[4];
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    o[i] = make_uint4(__float_as_uint(x[4 * i] + v[4 * i]),
                                      __float_as_uint(x[4 * i + 1] + v[4 * i + 1]),
                                      __float_as_uint(x[4 * i + 2] + v[4 * i + 2]),
                                      __float_as_uint(x[4 * i + 3] + v[4 * i + 3]));
                uint4* p = reinterpret_cast<uint4*>(g.dE + (size_t)m * N + c0);
                if (wide) {
                    stg32(p, o[0], o[1]);
                    stg32(p + 2, o[2], o[3]);
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i) p[i] = o[i];
                }
            }
        }
        phase ^= 1u;
    }
    if (!ok) {
        if (lt == 0 && g.status) atomicOr(g.status, 1u);
        mbar_wait(&s_bar[h][0], phase);                  // let MMAs and copies in flight
        mbar_wait(&s_bar[h][1], phase);                  // land first
        mbar_wait(&s_full[h], phase);
    }
    if (mover) bulk_wait();
    if (lane < 16) {
#pragma unroll
        for (int k = 0; k < 4; ++k) s_ce[h][wq][part * 64 + 16 * k + lane] = ce[k];
    }
    s_cp[h][lt >> 6][2 * (lt & 63)] = cp[0];
    s_cp[h][lt >> 6][2 * (lt & 63) + 1] = cp[1];
    tc_fence_before();
    __syncthreads();
    if (w == 0) tmem_dealloc(s_tmem, 512);
    {
        const int c = lt & 127;
        const float(*s)[N] = lt < 128 ? s_ce[h] : s_cp[h];
        float* out = lt < 128 ? g.part_v : g.part_p;
        out[(size_t)(2 * blockIdx.x + h) * N + c] = ((s[0][c] + s[1][c]) + s[2][c]) + s[3][c];
    }
}

// The node update of a message-passing layer and the node terms of the next
// layer's edge update in one kernel, per 128-node tile (x = [h, agg], 256 columns):
//   y = relu(x W3 + b3),  h' = h + y W4 + b4,  P = h' W1a,  Q = h' W1b
// x comes by TMA (128-byte swizzle) and serves MMA 1 and the residual; y and h'
// go to TMEM as the A operands of the next products, so nothing returns from HBM
// between the layers.  The weights (160 KB) and one x tile (64 KB) fill the
// shared memory; the next tile's x loads under MMA 3.  512 threads: the four
// warps of a TMEM lane quarter split the columns.  A small system has one tile
// per SM and is bound by the chain of three products, a large one by HBM (512 B
// in, 768 out per node; 1,792 and four launches as separate layers).
// On one GB300, us per layer, four launches / one: 17k nodes 36 / 18, 1.39M
// nodes 860 / 361 (4.9 TB/s).
// TMEM columns: accumulators of MMA 1 at 0, y at 128, accumulators of MMA 2 at
// 256, h' at 384; those of MMA 3 at 0 .. 255, over what MMA 2 has read.
constexpr size_t kNodeSmem = (size_t)7 * kETile + 1024;   // W3 (2), W4, W1a and W1b, x (2); alignment

__global__ void __launch_bounds__(512, 1)
    k_node_update(const NodeArgs g, const __grid_constant__ CUtensorMap map_x, const bool wide) {
    constexpr int N = 128;
    constexpr uint32_t T = kETile, BOX = T / 2;          // a box: 64 columns of 128 rows
    extern __shared__ unsigned char s_dyn[];
    __shared__ __align__(16) float s_b3[128], s_b4[128];
    __shared__ __align__(8) uint64_t s_full, s_bar[3];   // x loaded; MMAs 1 to 3
    __shared__ uint32_t s_tmem;
    unsigned char* s_raw = s_dyn + ((1024u - (sm_addr(s_dyn) & 1023u)) & 1023u);
    unsigned char* sx = s_raw;                           // four boxes
    unsigned char* sw3 = sx + 2 * T;                     // N x 256
    unsigned char* sw4 = sw3 + 2 * T;                    // N x N
    unsigned char* swp = sw4 + T;                        // 2 N x N: W1a, then W1b
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const bool mover = tid == 32;
    if (w == 0) tmem_alloc(&s_tmem, 512);
    if (tid == 0) {
        mbar_init1(&s_full);
        for (int k = 0; k < 3; ++k) mbar_init1(&s_bar[k]);
    }
    for (int c = tid; c < N * (2 * N / 8); c += 512) {
        const int r = c % N, gk = c / N;
        cp_async16(sw3 + kmajor_offset(r, gk * 8, 2 * N), g.W3t + (size_t)r * 2 * N + gk * 8, true);
    }
    cp_async_commit();
    for (int c = tid; c < N * (N / 8); c += 512) {
        const int r = c % N, gk = c / N;
        cp_async16(sw4 + kmajor_offset(r, gk * 8, N), g.W4t + (size_t)r * N + gk * 8, true);
        if (g.P) {
            cp_async16(swp + kmajor_offset(r, gk * 8, N), g.Wpt + (size_t)r * N + gk * 8, true);
            cp_async16(swp + kmajor_offset(N + r, gk * 8, N), g.Wqt + (size_t)r * N + gk * 8, true);
        }
    }
    cp_async_commit();
    if (tid < 128) {
        s_b3[tid] = g.b3[tid];
        s_b4[tid] = g.b4[tid];
    }
    asm volatile("cp.async.wait_group 1;" ::: "memory"); // W3
    fence_async_shared();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    const uint32_t ntiles = (g.n + 127) / 128;
    const int wq = w & 3, part = w >> 2;                 // lane quarter, column part
    const int r = wq * 32 + lane;                        // this thread's row of a tile
    const uint32_t quarter = (uint32_t)(wq * 32) << 16;
    auto load_x = [&](uint32_t t) {
        mbar_expect(&s_full, 2 * T);
#pragma unroll
        for (int b = 0; b < 4; ++b) tma_load(sx + b * BOX, &map_x, 64 * b, (int)(t * 128), &s_full);
    };
    auto put = [&](__nv_bfloat16* row, const uint32_t (&v)[8]) {   // 16 columns of a row
        uint4* o = reinterpret_cast<uint4*>(row);
        const uint4 a = make_uint4(v[0], v[1], v[2], v[3]), b = make_uint4(v[4], v[5], v[6], v[7]);
        if (wide) {
            stg32(o, a, b);
        } else {
            o[0] = a;
            o[1] = b;
        }
    };
    uint32_t tile = blockIdx.x, phase = 0;
    bool ok = true, weights = false;
    if (mover && tile < ntiles) load_x(tile);
    for (; tile < ntiles; tile += gridDim.x) {
        const uint32_t m = tile * 128 + (uint32_t)r, next = tile + gridDim.x;
        bool got = mbar_wait(&s_full, phase);            // x, for MMA 1 and the residual
        if (got && tid == 0) {
            tc_fence_after();
#pragma unroll
            for (int s = 0; s < 2 * N / 16; ++s)
                tc_mma(tmem, smem_desc_sw128(sm_addr(sx) + (s >> 2) * BOX + (s & 3) * 32),
                       smem_desc(sm_addr(sw3) + s * 256, kLBO, (2 * N / 8) * 128), idesc_bf16(N),
                       s > 0 ? 1u : 0u);
            tc_commit(&s_bar[0]);
        }
        if (!weights) {                                  // the other weights, under MMA 1
            cp_async_wait_all();
            fence_async_shared();
            weights = true;
        }
        got = got && mbar_wait(&s_bar[0], phase);
        tc_fence_after();
        // y = relu(acc + b3)
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int c0 = part * 32 + 16 * k;
            float v[16];
            tmem_ld16(tmem + quarter + c0, v);
            uint32_t z[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const __nv_bfloat162 t = __floats2bfloat162_rn(fmaxf(v[2 * q] + s_b3[c0 + 2 * q], 0.f),
                                                               fmaxf(v[2 * q + 1] + s_b3[c0 + 2 * q + 1], 0.f));
                z[q] = *reinterpret_cast<const uint32_t*>(&t);
            }
            tmem_st8(tmem + quarter + 128u + (uint32_t)(c0 / 2), z);
            if (g.Y && m < g.n) put(g.Y + (size_t)m * N + c0, z);
        }
        tmem_st_wait();
        tc_fence_before();
        ok = __syncthreads_and(got) != 0;                // y complete
        if (!ok) break;
        if (tid == 0) {
            tc_fence_after();
#pragma unroll
            for (int s = 0; s < N / 16; ++s)
                tc_mma_ta(tmem + 256u, tmem + 128u + s * 8,
                          smem_desc(sm_addr(sw4) + s * 256, kLBO, (N / 8) * 128), idesc_bf16(N),
                          s > 0 ? 1u : 0u);
            tc_commit(&s_bar[1]);
        }
        got = mbar_wait(&s_bar[1], phase);
        tc_fence_after();
        // h' = (acc + b4) + h
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int c0 = part * 32 + 16 * k;
            float v[16], t[16];
            tmem_ld16(tmem + quarter + 256u + c0, v);
            const unsigned char* box = sx + (c0 >> 6) * BOX;
            unpack8(*reinterpret_cast<const uint4*>(box + sw128_offset(r, (c0 & 63) / 8)), t);
            unpack8(*reinterpret_cast<const uint4*>(box + sw128_offset(r, (c0 & 63) / 8 + 1)), t + 8);
            uint32_t z[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const __nv_bfloat162 u =
                    __floats2bfloat162_rn(v[2 * q] + s_b4[c0 + 2 * q] + t[2 * q],
                                          v[2 * q + 1] + s_b4[c0 + 2 * q + 1] + t[2 * q + 1]);
                z[q] = *reinterpret_cast<const uint32_t*>(&u);
            }
            if (g.P) tmem_st8(tmem + quarter + 384u + (uint32_t)(c0 / 2), z);
            if (m < g.n) put(g.H + (size_t)m * (2 * N) + c0, z);
        }
        tmem_st_wait();
        tc_fence_before();
        ok = __syncthreads_and(got) != 0;                // h' complete, x free
        if (!ok) break;
        if (mover && next < ntiles) load_x(next);
        if (g.P) {
            if (tid == 0) {
                tc_fence_after();
#pragma unroll
                for (int s = 0; s < N / 16; ++s)
                    tc_mma_ta(tmem, tmem + 384u + s * 8,
                              smem_desc(sm_addr(swp) + s * 256, kLBO, (N / 8) * 128), idesc_bf16(2 * N),
                              s > 0 ? 1u : 0u);
                tc_commit(&s_bar[2]);
            }
            got = mbar_wait(&s_bar[2], phase);
            tc_fence_after();
            __nv_bfloat16* out = (part < 2 ? g.P : g.Q) + (size_t)m * N + (part & 1) * 64;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                float v[16];
                tmem_ld16(tmem + quarter + (uint32_t)(part * 64 + 16 * k), v);
                uint32_t z[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const __nv_bfloat162 u = __floats2bfloat162_rn(v[2 * q], v[2 * q + 1]);
                    z[q] = *reinterpret_cast<const uint32_t*>(&u);
                }
                if (m < g.n) put(out + 16 * k, z);
            }
            tc_fence_before();
            ok = __syncthreads_and(got) != 0;            // MMA 3's columns free
            if (!ok) break;
        }
        phase ^= 1u;
    }
    if (!ok) {
        if (tid == 0 && g.status) atomicOr(g.status, 1u);
        mbar_wait(&s_full, phase);                       // let MMAs and copies in flight
        mbar_wait(&s_full, phase ^ 1u);
        for (int k = 0; k < 3; ++k) mbar_wait(&s_bar[k], phase);   // land first
    }
    cp_async_wait_all();
    tc_fence_before();
    __syncthreads();
    if (w == 0) tmem_dealloc(tmem, 512);
}

template <int K, int N>
void launch_linear_t(const LinearArgs& g, int sms, cudaStream_t st) {
    static bool init = false;
    const size_t smem = linear_smem<K, N>();
    if (!init) {
        cudaFuncSetAttribute(k_linear<K, N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        init = true;
    }
    // resident blocks per SM: shared memory, registers and the SM's 512
    // TMEM columns
    static int per_sm = 0;
    if (!per_sm) {
        cudaFuncAttributes fa{};
        cudaFuncGetAttributes(&fa, k_linear<K, N>);
        const int cols = N <= 32 ? 32 : (N <= 64 ? 64 : (N <= 128 ? 128 : 256));
        const int by_smem = (int)((228u * 1024u) / (smem + fa.sharedSizeBytes + 1024u));
        const int by_regs = fa.numRegs > 0 ? 65536 / (linear_threads<N>() * fa.numRegs) : 1;
        per_sm = by_smem < by_regs ? by_smem : by_regs;
        if (per_sm > 512 / cols) per_sm = 512 / cols;
        if (per_sm < 1) per_sm = 1;
    }
    const uint32_t tiles = (g.M + 127) / 128;
    uint32_t grid = (uint32_t)(sms * per_sm);
    if (grid > tiles) grid = tiles ? tiles : 1;
    k_linear<K, N><<<grid, linear_threads<N>(), smem, st>>>(g);
}

// Tensor map of an M x cols bf16 matrix (row stride ld) in boxes of 128 rows x 64 columns with
// the 128-byte swizzle.  Rows past M load as zeros and are not stored.
bool tile_map(CUtensorMap* map, const void* base, uint32_t M, uint32_t ld = 128,
              uint32_t cols = 128) {
    using Encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static const Encode encode = [] {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault,
                                             &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            fn = nullptr;
        }
        return reinterpret_cast<Encode>(fn);
    }();
    if (!encode) return false;
    const cuuint64_t dims[2] = {cols, M}, strides[1] = {(cuuint64_t)ld * 2};
    const cuuint32_t box[2] = {64, 128}, step[2] = {1, 1};
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides,
                  box, step, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
           CUDA_SUCCESS;
}

template <int N>
void launch_wgrad_t(const WgradArgs& g, int sms, cudaStream_t st) {
    static bool init = false;
    const size_t smem = (size_t)128 * 128 * 2 + (size_t)N * 128 * 2;
    if (!init) {
        cudaFuncSetAttribute(k_wgrad<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        init = true;
    }
    const uint32_t tiles = (g.M + 127) / 128;
    uint32_t grid = (uint32_t)g.nparts;
    if (grid > tiles) grid = tiles ? tiles : 1;
    k_wgrad<N><<<grid, 128, smem, st>>>(g);
    const int count = 128 * N;
    WgradOuts outs = {};
    outs.dW[0] = g.dW;
    k_wgrad_reduce<<<(count + 31) / 32, 256, 0, st>>>(g.partial, (int)grid, count, outs, g.scale);
}

bool launch_wgrad_tma(const WgradArgs* gs, int batch, int sms, cudaStream_t st) {
    static std::once_flag once;
    std::call_once(once, [] {
        cudaFuncSetAttribute(k_wgrad_tma, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWgSmem);
    });
    constexpr int count = 128 * 128;
    const WgradArgs& g = gs[0];
    WgradMaps maps;
    WgradOuts outs = {};
    for (int k = 0; k < batch; ++k) {
        outs.dW[k] = gs[k].dW;
        if (g.M == 0) {
            if (cudaMemsetAsync(gs[k].dW, 0, count * sizeof(float), st) != cudaSuccess) return false;
        } else if (!tile_map(&maps.x[k], gs[k].X, g.M, gs[k].ldp ? gs[k].ldp : 128u) ||
                   !tile_map(&maps.y[k], gs[k].dY, g.M, gs[k].ldq ? gs[k].ldq : 128u)) {
            return false;
        }
    }
    if (g.M == 0) return true;
    const uint32_t tiles = (g.M + 127) / 128;
    uint32_t grid = (tiles + kWgMinTiles - 1) / kWgMinTiles;
    const uint32_t most = (uint32_t)sms / (uint32_t)batch, parts = g.nparts / (uint32_t)batch;
    if (grid > most) grid = most ? most : 1;
    if (grid > parts) grid = parts;
    k_wgrad_tma<<<dim3(grid, batch), 128, kWgSmem, st>>>(g, maps);
    k_wgrad_reduce<<<dim3((count + 31) / 32, batch), 256, 0, st>>>(g.partial, (int)grid, count, outs,
                                                                   g.scale);
    return true;
}

int g_sms = 0;

}  // namespace

int num_sms() {
    if (!g_sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev);
        if (g_sms <= 0) g_sms = 1;
    }
    return g_sms;
}

bool launch_linear(int K, int N, const LinearArgs& args, cudaStream_t st) {
    const int sms = num_sms();
    if (args.M == 0) return true;
    LinearArgs g = args;
    // every row and 16-column group that the epilogue touches 32-byte aligned
    const uintptr_t all = reinterpret_cast<uintptr_t>(g.res) | reinterpret_cast<uintptr_t>(g.gp) |
                          reinterpret_cast<uintptr_t>(g.gq) | reinterpret_cast<uintptr_t>(g.out_bf16) |
                          reinterpret_cast<uintptr_t>(g.out_f32);
    g.wide = all % 32u == 0u && (g.ldr | g.ldo) % 16u == 0u;
    if (K == 16 && N == 128) launch_linear_t<16, 128>(g, sms, st);
    else if (K == 128 && N == 128) launch_linear_t<128, 128>(g, sms, st);
    else if (K == 256 && N == 128) launch_linear_t<256, 128>(g, sms, st);
    else if (K == 128 && N == 16) launch_linear_t<128, 16>(g, sms, st);
    else if (K == 16 && N == 16) launch_linear_t<16, 16>(g, sms, st);
    else if (K == 128 && N == 256) launch_linear_t<128, 256>(g, sms, st);
    else return false;
    return true;
}

// The layer: two halves per block, one block per SM (193 KB of shared memory,
// the SM's 512 TMEM columns).
bool launch_edge_layer(const EdgeArgs& g, cudaStream_t st) {
    static std::once_flag once;
    std::call_once(once, [] {
        cudaFuncSetAttribute(k_edge_pp, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kEdgePPSmem);
    });
    if (g.M == 0) return true;
    CUtensorMap map_e, map_out;
    if (!tile_map(&map_e, g.E, g.M) || !tile_map(&map_out, g.Eout, g.M)) return false;
    const uintptr_t all = reinterpret_cast<uintptr_t>(g.P) | reinterpret_cast<uintptr_t>(g.Q) |
                          reinterpret_cast<uintptr_t>(g.Z);
    const uint32_t tiles = (g.M + 127) / 128;
    uint32_t grid = (uint32_t)num_sms();
    if (grid > (tiles + 1) / 2) grid = (tiles + 1) / 2;
    k_edge_pp<<<grid, 512, kEdgePPSmem, st>>>(g, map_e, map_out, all % 32u == 0u);
    return true;
}

bool launch_edge_backward(const EdgeBwdArgs& g, uint32_t* nparts, cudaStream_t st) {
    static std::once_flag once;
    std::call_once(once, [] {
        cudaFuncSetAttribute(k_edge_bwd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kEdgeBwdSmem);
    });
    *nparts = 0;
    if (g.M == 0) return true;
    CUtensorMap map_z, map_v, map_p;
    if (!tile_map(&map_z, g.Z, g.M) || !tile_map(&map_v, g.dEb, g.M) || !tile_map(&map_p, g.dpre, g.M))
        return false;
    const uintptr_t all = reinterpret_cast<uintptr_t>(g.dE) | reinterpret_cast<uintptr_t>(g.node);
    const uint32_t tiles = (g.M + 127) / 128;
    uint32_t grid = (uint32_t)num_sms();
    if (grid > (tiles + 1) / 2) grid = (tiles + 1) / 2;
    *nparts = 2 * grid;
    k_edge_bwd<<<grid, 512, kEdgeBwdSmem, st>>>(g, map_z, map_v, map_p, all % 32u == 0u && g.ldn % 8u == 0u);
    return true;
}

bool launch_node_update(const NodeArgs& g, cudaStream_t st) {
    static std::once_flag once;
    std::call_once(once, [] {
        cudaFuncSetAttribute(k_node_update, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kNodeSmem);
    });
    if (g.n == 0) return true;
    CUtensorMap map_x;
    if (!tile_map(&map_x, g.X, g.n, 256, 256)) return false;
    const uintptr_t all = reinterpret_cast<uintptr_t>(g.Y) | reinterpret_cast<uintptr_t>(g.H) |
                          reinterpret_cast<uintptr_t>(g.P) | reinterpret_cast<uintptr_t>(g.Q);
    const uint32_t tiles = (g.n + 127) / 128;
    const uint32_t sms = (uint32_t)num_sms();
    k_node_update<<<tiles < sms ? tiles : sms, 512, kNodeSmem, st>>>(g, map_x, all % 32u == 0u);
    return true;
}

// The encoder: two 256-thread blocks per SM.
bool launch_edge_encoder(const EdgeArgs& g, cudaStream_t st) {
    static std::once_flag once;
    std::call_once(once, [] {
        cudaFuncSetAttribute(k_edge_encoder, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kEncSmem);
    });
    if (g.M == 0) return true;
    CUtensorMap map_out;
    if (!tile_map(&map_out, g.Eout, g.M)) return false;
    const uint32_t tiles = (g.M + 127) / 128;
    uint32_t grid = (uint32_t)(num_sms() * 2);
    if (grid > tiles) grid = tiles;
    k_edge_encoder<<<grid, 256, kEncSmem, st>>>(g, map_out, reinterpret_cast<uintptr_t>(g.Z) % 32u == 0u);
    return true;
}

bool launch_wgrads(const WgradArgs* g, int batch, cudaStream_t st) {
    return launch_wgrad_tma(g, batch, num_sms(), st);
}

bool launch_wgrad(int N, const WgradArgs& g, cudaStream_t st) {
    if (N == 128) return launch_wgrad_tma(&g, 1, num_sms(), st);
    if (N == 16) launch_wgrad_t<16>(g, num_sms(), st);
    else return false;
    return true;
}

}  // namespace sur
