// The 27-cell pair interaction (Eqs. 7 and 9) with its candidate test on the
// tcgen05 tensor cores of sm_103a.  The earlier shapes (test in half precision
// on the CUDA cores) are in sph_kernels.cu, with the description of units and
// staging that both share.
//
// What bounds the interaction is the number of instructions a warp issues per
// candidate and per hit (2.0 warp instructions per clock with 16 warps per SM;
// DRAM and the FP32 pipes are far from their limits).  So the distances of a
// unit's 128 particles to its staged candidates are one tcgen05.mma per 256
// candidates (a product of K = 16, exact to about 2e-3 of (2h)^2), whose
// accumulator rows a warp reads back with lane = particle: one funnel shift
// per candidate makes a hit mask, against about three instructions on the
// CUDA cores, and the masks span cells, so there are about half as many words
// as with one word per cell.  The non-empty words go to per-lane lists in
// shared memory and the pair phase pops them with the next word always
// loaded (ten instructions per hit).  Blocks have no barrier inside the
// candidate loop: the last warp done with a piece issues the next one's MMA.
// (Two accumulators of 128 candidates, the MMA two pieces ahead, hid the MMA's
// latency but cost a hundred instructions per warp and piece: 20.4 against
// 18.8 ms at 35.4M particles.)  Both sides on one GB300, ms per launch (the
// counter-scheduled 4 x 2 shape of sph_kernels.cu / this kernel): 35.4M
// particles 24.0 / 18.4, 1.39M with obstacles 0.956 / 0.701, 256 dam breaks
// (5.5M) 3.85 / 3.15, 64k with the cubic spline 0.094 / 0.072, 17k 0.0229 /
// 0.0196.  Next to the pair phase (0.23 ms of it at 1.39M) the largest share is
// the units' set-up, 0.20: the latency of the staging copies.
#include <cuda_fp16.h>
#include <math.h>

#include "sph_internal.cuh"
#include "sph_pair.cuh"
#include "sur_gemm.cuh"

namespace sph {

namespace {

// Fixed-point x of posu: cells of 2^26 units, modulo 2^32 (64 cells).
constexpr int kXBits = 26;

// Rows of the two MMA operands (K = 16 halves, 32 bytes), in cells about the
// unit's centre, x split into two halves each, x = xh + xl, y and z rounded to
// one: the product of particle q's row and candidate p's row is
// (|q|^2 - thr) + |p|^2 - 2 q.p
//   q:  -2xh -2xh -2xl -2y -2z  1  1 nh | nl 0 ..
//   p:    xh   xl   xh   y   z mh ml  1 |  1 0 ..
// n = |q|^2 - thr and m = |p|^2 of the rounded coordinates, in two halves
// each.  Candidate rows differ in their first 16 bytes only.
__device__ __forceinline__ uint32_t bits2(__half2 v) { return *reinterpret_cast<uint32_t*>(&v); }

// v as two halves (the high one in the low 16 bits).
__device__ __forceinline__ __half2 split_half(float v) {
    const float h = __half2float(__float2half_rn(v));
    return __floats2half2_rn(h, v - h);
}

constexpr uint32_t kFarHalf = 0x7b00u;   // 57344: a row that never tests as a hit

__device__ __forceinline__ uint4 candidate_row(float X, float Y, float Z) {
    const __half2 x = split_half(X), yz = __floats2half2_rn(Y, Z);
    const float2 fx = __half22float2(x), f = __half22float2(yz);
    const float x1 = fx.x + fx.y;
    const __half2 m = split_half(fmaf(x1, x1, fmaf(f.x, f.x, f.y * f.y)));
    // xh xl | xh y | z mh | ml 1
    return make_uint4(bits2(x), __byte_perm(bits2(x), bits2(yz), 0x5410),
                      __byte_perm(bits2(yz), bits2(m), 0x5432),
                      __byte_perm(bits2(m), 0x3c00u, 0x5432));
}

__device__ __forceinline__ void particle_row(unsigned char* row, bool valid, float X, float Y,
                                             float Z, float thr) {
    const __half2 x = split_half(X), yz = __floats2half2_rn(Y, Z);
    const float2 fx = __half22float2(x), f = __half22float2(yz);
    const float x1 = fx.x + fx.y;
    const __half2 n = split_half(fmaf(x1, x1, fmaf(f.x, f.x, f.y * f.y)) - thr);
    const __half2 m2 = __float2half2_rn(-2.f);
    const uint32_t x2 = bits2(__hmul2(x, m2)), yz2 = bits2(__hmul2(yz, m2)), nn = bits2(n);
    uint4 a = make_uint4(__byte_perm(x2, x2, 0x1010), __byte_perm(x2, yz2, 0x5432),
                         __byte_perm(yz2, 0x3c00u, 0x5432), __byte_perm(0x3c00u, nn, 0x5410));
    uint4 b = make_uint4(nn >> 16, 0u, 0u, 0u);
    if (!valid) {   // no particle: no candidate tests as a hit
        a = make_uint4(0u, 0u, 0u, kFarHalf << 16);
        b = make_uint4(0u, 0u, 0u, 0u);
    }
    *reinterpret_cast<uint4*>(row) = a;
    *reinterpret_cast<uint4*>(row + sur::kLBO) = b;
}

// tcgen05 instruction descriptor: FP32 accumulator, A and B half precision,
// both K-major, M = 128, N.
__device__ __forceinline__ uint32_t idesc_half(uint32_t N) {
    return (1u << 4) | ((N >> 3) << 17) | ((128u >> 4) << 24);
}

// Sign bits of 32 (16, 8) consecutive FP32 accumulator columns of this
// thread's TMEM lane, column k at bit k.
__device__ __forceinline__ uint32_t signs32(uint32_t taddr) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,"
        "%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
        "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
        "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
    uint32_t c[4] = {0u, 0u, 0u, 0u};   // four independent chains of eight columns
#pragma unroll
    for (int k = 7; k >= 0; --k)
#pragma unroll
        for (int q = 0; q < 4; ++q) c[q] = __funnelshift_l(r[8 * q + k], c[q], 1);
    return __byte_perm(__byte_perm(c[0], c[1], 0x0040), __byte_perm(c[2], c[3], 0x0040), 0x5410);
}

__device__ __forceinline__ uint32_t signs16(uint32_t taddr) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,"
        "%9,%10,%11,%12,%13,%14,%15}, [%16];\n tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
    uint32_t c[2] = {0u, 0u};
#pragma unroll
    for (int k = 7; k >= 0; --k)
#pragma unroll
        for (int q = 0; q < 2; ++q) c[q] = __funnelshift_l(r[8 * q + k], c[q], 1);
    return c[0] | (c[1] << 8);
}

__device__ __forceinline__ uint32_t signs8(uint32_t taddr) {
    uint32_t r[8];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7"
        "}, [%8];\n tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7])
        : "r"(taddr)
        : "memory");
    uint32_t c = 0u;
#pragma unroll
    for (int k = 7; k >= 0; --k) c = __funnelshift_l(r[k], c, 1);
    return c;
}

// A lane's list of hit words: (hit mask, entry base) pairs 256 bytes apart,
// empty words left out, ended by a word without hits.  push_word appends one
// at lp.
__device__ __forceinline__ void push_word(uint32_t& lp, uint32_t mask, uint32_t base) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.u32 p, %1, 0;\n @p st.shared.v2.u32 [%0], {%1, %2};\n"
        " @p add.u32 %0, %0, 256;\n}"
        : "+r"(lp)
        : "r"(mask), "r"(base)
        : "memory");
}

// Cursor over such a list: the word in hand and the next one, already loaded.
struct HitCursor {
    uint32_t m, base, next_m, next_base, rp;
};

// Which candidate a column is: the SPLIT parts of a group take alternate
// candidates, column c of part p being candidate SPLIT c + p.  With TURN, in
// turns that change from eight to eight: SPLIT c + (p ^ (c / M mod SPLIT)), M = 8 /
// SPLIT, because with the same turn throughout a warp's 16-byte loads of its hits
// meet half of the banks only.  Two more instructions per hit for fewer bank
// conflicts: ms per launch without / with, 35.4M particles 18.8 / 18.3, 1.39M
// 0.713 / 0.697; in units of 64 particles (256 dam breaks 3.12 / 3.14) it does not pay.
template <uint32_t SPLIT, bool TURN>
struct Turns {
    static constexpr uint32_t M = 8 / SPLIT, S1 = SPLIT - 1;
    // the candidate that part p takes of SPLIT consecutive ones, at candidate t
    static __device__ __forceinline__ uint32_t turn(uint32_t t, uint32_t p) {
        return TURN ? p ^ ((t >> 3) & S1) : p;
    }
    // part and column of candidate t
    static __device__ __forceinline__ uint32_t part(uint32_t t) { return turn(t, t & S1); }
    static __device__ __forceinline__ uint32_t column(uint32_t t) { return t / SPLIT; }
    // columns of part p before candidate t
    static __device__ __forceinline__ uint32_t before(uint32_t t, uint32_t p) {
        return (t + S1 - turn(t, p)) / SPLIT;
    }
};

// The next hit's entry: base + 16 (SPLIT bit + its turn); mp = M part (TURN).
// The ending word has no bit (bfind gives all ones): its base makes the entry
// the pad's from then on.
template <uint32_t SPLIT, bool TURN>
__device__ __forceinline__ uint32_t pop_hit(HitCursor& h, uint32_t end, uint32_t mp) {
    using T = Turns<SPLIT, TURN>;
    uint32_t e, b;
    asm volatile(
        "{\n .reg .pred p;\n .reg .u32 t;\n setp.eq.u32 p, %1, 0;\n @p mov.u32 %1, %3;\n"
        " @p mov.u32 %2, %4;\n @p ld.shared.v2.u32 {%3, %4}, [%5];\n @p add.u32 %5, %5, 256;\n"
        " @p min.u32 %5, %5, %6;\n bfind.u32 %0, %1;\n mov.u32 t, 1;\n shl.b32 t, t, %0;\n"
        " xor.b32 %1, %1, t;\n}"
        : "=&r"(b), "+r"(h.m), "+r"(h.base), "+r"(h.next_m), "+r"(h.next_base), "+r"(h.rp)
        : "r"(end)
        : "memory");
    e = h.base + b * (16u * SPLIT);
    if (TURN) e += ((b & (T::M * T::S1)) ^ mp) * (16u / T::M);
    return e;
}

// Shape of a variant: W warps of particles (units of 32 W), SPLIT warps per
// group of 32 particles, STAGE staged candidates, WCAP hit words per lane,
// PIECE candidates per MMA (an accumulator of PIECE TMEM columns).
template <int W, int SPLIT, int STAGE, int WCAP, int PIECE>
struct TcShape {
    // staged posu and velrhop (one slot more: the pad), A, B, lists, the
    // sums of the parts 1 ..
    static constexpr size_t stage_bytes = (size_t)(STAGE + 1) * sizeof(float4);
    static constexpr size_t a_off = (2 * stage_bytes + 127) / 128 * 128;
    static constexpr size_t b_off = a_off + 128 * 32;
    static constexpr size_t l_off = b_off + (size_t)PIECE * 32;
    static constexpr size_t c_off = l_off + (size_t)W * SPLIT * (WCAP + 1) * 256;
    static constexpr size_t smem = c_off + (size_t)(SPLIT - 1) * W * 7 * 32 * 4;
    static constexpr int fb_cap = 2 * stage_bytes / ((size_t)W * SPLIT * 32 * 4) < 64
                                      ? (int)(2 * stage_bytes / ((size_t)W * SPLIT * 32 * 4))
                                      : 64;
    static_assert(fb_cap >= 16, "fallback lists must fit in the staging area");
    static_assert(PIECE % (8 * SPLIT) == 0 && PIECE % 32 == 0, "a piece's columns and rows");
};

// Largest of a warp's values; a NaN counts only if all of them are NaN.  (Five
// shuffles and maxima before, three times per warp and unit: 17k particles
// 0.0200 -> 0.0196 ms, 1.39M 0.717 -> 0.713.)
__device__ __forceinline__ float warp_max(float v) {
    float m;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(m) : "f"(v));
    return m;
}

// mbar_wait_bounded with the thread suspended for up to 1 us per try (fewer
// polls: they take issue slots from the warps that compute).
__device__ __forceinline__ bool mbar_sleep_bounded(uint64_t* bar, uint32_t parity) {
    for (uint32_t k = 0; k < (1u << 20); ++k) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
            " selp.u32 %0, 1, 0, p;\n}"
            : "=r"(ok)
            : "r"(smem_u32(bar)), "r"(parity), "r"(1000u)
            : "memory");
        if (ok) return true;
    }
    return false;
}

// What a block needs to know of a unit (one copy in shared memory, written by
// the first warp during the unit before).
struct UnitPlan {
    uint32_t i0, i1;        // particles; i0 = kNoUnit: no unit left
    uint32_t q;             // instance
    uint32_t done;          // the instance has reached its end time
    uint32_t rowbase;       // label of cell 0 of the unit's row
    int ncx, ncxy;          // cells per row, per layer
    int ulo, nce;           // first neighbour cell, cell offsets per neighbour row
    uint32_t okrows;        // bit r: neighbour row r is inside the grid
    uint32_t xc;            // centre in fixed-point x
    float half_span;        // largest |x| of a candidate from it, in cells
    uint32_t id_fluid;
    float c0;
};
constexpr uint32_t kNoUnit = 0xffffffffu;

__device__ __forceinline__ UnitPlan plan_unit(const Dev& d, uint2 unit, uint32_t key0,
                                              uint32_t keyl) {
    UnitPlan p;
    p.i0 = unit.x;
    p.i1 = unit.y;
    p.q = find_instance(d.cell_base, d.n_inst, key0);
    p.done = __ldg(d.is.done + p.q);
    const Inst& I = d.inst[p.q];
    const uint32_t lrow = (key0 - I.cell_base) / (uint32_t)I.ncx;
    p.rowbase = I.cell_base + lrow * (uint32_t)I.ncx;
    p.ncx = I.ncx;
    p.ncxy = I.ncx * I.ncy;
    const int cz = (int)(lrow / (uint32_t)I.ncy), cy = (int)lrow - cz * I.ncy;
    const int xb = (int)(key0 - p.rowbase), xe = (int)(keyl - p.rowbase);
    p.ulo = xb > 0 ? xb - 1 : 0;
    const int uhi = xe + 1 < I.ncx ? xe + 1 : I.ncx - 1;
    p.nce = uhi - p.ulo + 2;
    const uint32_t yok = (cy > 0 ? 0x49u : 0u) | 0x92u | (cy + 1 < I.ncy ? 0x124u : 0u);
    const uint32_t zok = (cz > 0 ? 0x7u : 0u) | 0x38u | (cz + 1 < I.ncz ? 0x1c0u : 0u);
    p.okrows = yok & zok;
    p.xc = (uint32_t)(xb + xe + 1) << (kXBits - 1);
    p.half_span = 0.5f * (float)(xe - xb + 3);
    p.id_fluid = I.id_fluid;
    p.c0 = I.c0;
    return p;
}

template <int W, int SPLIT, int STAGE, int WCAP, int PIECE, int MINB, bool COUNTS, int KERN>
__global__ void __launch_bounds__(W * SPLIT * 32, MINB) k_interact_tc(const Dev d,
                                                                      const InteractArgs a) {
    using SH = TcShape<W, SPLIT, STAGE, WCAP, PIECE>;
    constexpr bool TURN = W == 4;
    using TN = Turns<SPLIT, TURN>;
    constexpr int NW = W * SPLIT, NT = NW * 32;
    constexpr int FBCAP = SH::fb_cap;
    constexpr uint32_t kPad = (uint32_t)STAGE * 16u;       // list entry of the pad slot
    constexpr uint32_t kPartCols = PIECE / SPLIT;          // of one part of a piece
    constexpr int kBuilders = PIECE / 32;                  // groups of 32 rows of a piece
    static_assert(NW >= 4 && (PIECE == 128 || PIECE == 256), "TMEM lane quarters and columns");
    extern __shared__ __align__(128) unsigned char s_raw[];
    float4* s_p = reinterpret_cast<float4*>(s_raw);
    float4* s_v = s_p + STAGE + 1;
    unsigned char* s_a = s_raw + SH::a_off;
    unsigned char* s_b = s_raw + SH::b_off;
    __shared__ __align__(8) uint64_t s_bar, s_mbar;   // staging copies, MMA
    __shared__ uint32_t s_arr;                   // warps done with a piece
    __shared__ uint32_t s_tmem;
    __shared__ uint32_t s_rs[9], s_base[10];
    __shared__ uint32_t s_offb[2][9][kSpan + 3];
    __shared__ UnitPlan s_plan[2];
    __shared__ uint32_t s_sum[kSpan + 3];        // cell offsets summed over the 9 rows
    __shared__ float2 s_shift[9];                // (y, z) of a run's row in the unit's frame
    __shared__ uint32_t s_nui;
    __shared__ __align__(8) uint32_t s_nx[4];    // the next unit: particles, first and last label
    __shared__ int s_mode;
    __shared__ uint32_t s_ru[NW][4];             // per warp: counters over this block's units
    __shared__ uint32_t s_stop[NW][8];           // where a warp with a full list stopped

    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int part = w / W;
    if (w == 0) sur::tmem_alloc(&s_tmem, PIECE);
    if (tid == 0) {
        mbar_init(&s_bar, 1);
        mbar_init(&s_mbar, 1);
        s_arr = 0u;
    }
    pdl_wait();
    sur::tc_fence_before();
    __syncthreads();
    sur::tc_fence_after();
    const uint32_t tmem = s_tmem;
    const uint32_t lane_base = tmem + ((uint32_t)((w & 3) * 32) << 16);
    unsigned char* wlist = s_raw + SH::l_off + (size_t)w * (WCAP + 1) * 256;   // this warp's lists
    const uint32_t list0 = smem_u32(wlist) + 8u * (uint32_t)lane;
    const float inv_cs = 1.0f / d.csf;
    const float fx_cell = 1.0f / (float)(1 << kXBits);
    const float fx_len = d.csf * fx_cell;                  // fixed-point x to length
    const uint32_t nunits = *a.n_units;
    // the constant second halves of operand B's rows
    for (int t = tid; t < PIECE; t += NT)
        *reinterpret_cast<uint4*>(s_b + sur::kmajor_offset((uint32_t)t, 8, 16)) =
            make_uint4(0x3c00u, 0u, 0u, 0u);
    sur::fence_async_shared();
    uint32_t phase = 0, mphase = 0;
    if (lane < 4) s_ru[w][lane] = 0u;
    if (tid < 9)
        s_shift[tid] = make_float2((float)(tid % 3 - 1) * d.csf, (float)(tid / 3 - 1) * d.csf);
    // asynchronous 4-byte copies of a planned unit's cell offsets (9 rows)
    auto fetch_offsets = [&](const UnitPlan& p, uint32_t (*o)[kSpan + 3]) {
        for (int r = w; r < 9; r += NW) {
            const bool okr = (p.okrows >> r) & 1u;
            const uint32_t* src = a.off + (int64_t)p.rowbase + (r % 3 - 1) * p.ncx +
                                  (int64_t)(r / 3 - 1) * p.ncxy + p.ulo;
            for (int c = lane; c < p.nce; c += 32) {
                if (okr)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                                     smem_u32(&o[r][c])),
                                 "l"(src + c)
                                 : "memory");
                else
                    o[r][c] = 0u;
            }
        }
    };
    // the plan of unit `u` (first warp)
    auto make_plan = [&](UnitPlan* out, uint32_t u) {
        UnitPlan p;
        p.i0 = kNoUnit;
        if (u < nunits) {
            const uint2 unit = a.units[u];
            p = plan_unit(d, unit, __ldg(a.key + unit.x), __ldg(a.key + unit.y - 1));
        }
        if (lane == 0) *out = p;
    };
    int sb = 0;
    // units are taken from a counter (the first one is blockIdx.x); the next
    // unit's plan and cell offsets are fetched during this one
    if (w == 0) make_plan(&s_plan[0], blockIdx.x);
    __syncthreads();
    if (s_plan[0].i0 != kNoUnit) fetch_offsets(s_plan[0], s_offb[0]);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    while (s_plan[sb].i0 != kNoUnit) {
    uint32_t (*s_off)[kSpan + 3] = s_offb[sb];
    if (tid == 0) s_nui = gridDim.x + atomicAdd(a.sched, 1u);
    const uint32_t i0 = s_plan[sb].i0, i1 = s_plan[sb].i1, q = s_plan[sb].q;
    if (!in_bounds(i0 < i1 && i1 <= d.n && i1 - i0 <= (uint32_t)(W * 32), d.status)) break;
    if (s_plan[sb].done) {                           // block-uniform
        __syncthreads();                             // s_nui written
        if (w == 0) make_plan(&s_plan[sb ^ 1], s_nui);
        __syncthreads();
        sb ^= 1;
        if (s_plan[sb].i0 != kNoUnit) fetch_offsets(s_plan[sb], s_offb[sb]);
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        continue;
    }
    const float c0 = s_plan[sb].c0;
    const int ncx = s_plan[sb].ncx, ulo = s_plan[sb].ulo, nce = s_plan[sb].nce;
    const uint32_t rowbase = s_plan[sb].rowbase, xc = s_plan[sb].xc;
    // staging plan and copies by the first warp: lane r < 9 owns run r
    if (w == 0) {
        const uint32_t len = lane < 9 ? s_off[lane][nce - 1] - s_off[lane][0] : 0u;
        uint32_t incl = len;
#pragma unroll
        for (int o = 1; o < 16; o <<= 1) {
            const uint32_t t = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += t;
        }
        const uint32_t base = incl - len;
        const uint32_t total = __shfl_sync(kFull, incl, 8);
        if (lane < 9) {
            s_base[lane] = base;
            s_rs[lane] = s_off[lane][0];
        }
        if (lane == 0) {
            s_base[9] = total;
            s_mode = total <= (uint32_t)STAGE;
            if (total <= (uint32_t)STAGE)
                mbar_expect_tx(&s_bar, total * 2u * (uint32_t)sizeof(float4));
        }
        __syncwarp();
        // the expected byte count is registered before any copy is issued
        if (total <= (uint32_t)STAGE && lane < 18) {
            const int r = lane >> 1;
            const uint32_t rl = __shfl_sync(0x3ffffu, len, r);
            const uint32_t rbase = __shfl_sync(0x3ffffu, base, r);
            const uint32_t rs = s_off[r][0];
            if (rl) {
                if (lane & 1)
                    bulk_g2s(s_v + rbase, a.velrhop + rs, rl * (uint32_t)sizeof(float4), &s_bar);
                else
                    bulk_g2s(s_p + rbase, a.posu + rs, rl * (uint32_t)sizeof(float4), &s_bar);
            }
        }
    } else if (w == 1) {
        for (int c = lane; c < nce; c += 32) {
            uint32_t t = 0;
#pragma unroll
            for (int r = 0; r < 9; ++r) t += s_off[r][c];
            s_sum[c] = t;
        }
    }
    // own particle, while the copies are in flight
    const uint32_t i = i0 + (uint32_t)((w % W) * 32 + lane);
    const bool valid = i < i1;
    float4 pi = make_float4(0.f, 0.f, 0.f, 0.f), vi = make_float4(0.f, 0.f, 0.f, 1.f);
    int cx = 0;
    bool fluid = false;
    if (valid) {
        pi = a.posu[i];
        vi = a.velrhop[i];
        cx = (int)(__ldg(a.key + i) - rowbase);
        fluid = a.id[i] >= s_plan[sb].id_fluid;
    }
    const uint32_t xi = __float_as_uint(pi.x);
    const float rri = vi.w * d.inv_rho0;
    const float ci = c0 * rri * rri * rri;
    // MMA operand A: the warps of the first four TMEM lane quarters write
    // their particles' rows (a group shared by several quarters is repeated)
    if (w < 4) {
        const float hs = s_plan[sb].half_span;
        const float thr = fmaf(0x1p-16f * hs, hs, 1.0f + 0x1p-9f);
        particle_row(s_a + sur::kmajor_offset((uint32_t)(w * 32 + lane), 0, 16), valid,
                     (float)(int)(xi - xc) * fx_cell, fmaf(pi.y, inv_cs, -0.5f),
                     fmaf(pi.z, inv_cs, -0.5f), thr);
    }
    if (tid == 0) {
        // the pad: 32 cells away along x (modulo 64), out of reach of every i
        s_p[STAGE] = make_float4(__uint_as_float(xc ^ 0x80000000u), 0.f, 0.f, 0.f);
        s_v[STAGE] = make_float4(0.f, 0.f, 0.f, d.rho0);
    }
    PairAcc acc = {0.f, 0.f, 0.f, 0.f, 0.f, 0u};
    __syncthreads();
    const bool staged = s_mode != 0;
    // the next unit (taken by thread 0 at the top of this one): its record
    // now, its end labels once the record has landed, its plan after the
    // candidate test (first warp)
    const uint32_t nui = s_nui;
    if (tid == 0 && nui < nunits) {
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(s_nx)),
                     "l"(a.units + nui)
                     : "memory");
    }
    const uint32_t act = __ballot_sync(kFull, valid);
    const int wxmin = __reduce_min_sync(kFull, valid ? cx : 0x7fffffff);
    const int wxmax = __reduce_max_sync(kFull, valid ? cx : -1);
    // the warp's cells; a warp without particles reads no candidates
    const int xlo = act ? (wxmin > 0 ? wxmin - 1 : 0) : ulo;
    const int xhi = act ? (wxmax + 1 < ncx ? wxmax + 1 : ncx - 1) : ulo;
    // candidates of the 27 cells
    if (part == 0) {
        const uint32_t nc = valid ? s_sum[(cx + 1 < ncx ? cx + 2 : ncx) - ulo] -
                                        s_sum[(cx > 0 ? cx - 1 : 0) - ulo]
                                  : 0u;
        const uint32_t t = __reduce_add_sync(kFull, nc);
        if (lane == 0) s_ru[w][1] += t;
    }
    bool ok = true;
    if (staged) {
        ok = mbar_wait_bounded(&s_bar, phase);
        phase ^= 1u;
        // The staged candidates go through the tensor cores in pieces of
        // PIECE.  Operand B's rows are ordered so that a part's accumulator
        // columns are contiguous (Turns).
        const uint32_t nst = s_base[9];
        const uint32_t npc = (nst + PIECE - 1) / PIECE;
        // 32 rows of piece k: shift the candidates' y, z into the frame of
        // the unit's row (in place), then their operand rows; slots past the
        // last candidate get a row that never tests as a hit
        auto build = [&](uint32_t k, uint32_t g) {
            const uint32_t t = g * 32u + (uint32_t)lane;
            const uint32_t j = k * PIECE + t;
            unsigned char* row =
                s_b + sur::kmajor_offset(TN::part(t) * kPartCols + TN::column(t), 0, 16);
            if (j < nst) {
                int r = 0;
#pragma unroll
                for (int q2 = 1; q2 < 9; ++q2) r += s_base[q2] <= j ? 1 : 0;
                float4 v = s_p[j];
                const float2 sh = s_shift[r];
                v.y += sh.x;
                v.z += sh.y;
                s_p[j] = v;
                const float X = (float)(int)(__float_as_uint(v.x) - xc) * fx_cell;
                *reinterpret_cast<uint4*>(row) =
                    candidate_row(X, fmaf(v.y, inv_cs, -0.5f), fmaf(v.z, inv_cs, -0.5f));
            } else {
                *reinterpret_cast<uint4*>(row) = make_uint4(0u, 0u, kFarHalf << 16, 0x3c000000u);
            }
            sur::fence_async_shared();
        };
        auto issue = [&]() {                             // by one thread
            sur::tc_fence_after();
            sur::tc_mma(tmem, sur::smem_desc(smem_u32(s_a), sur::kLBO, 256),
                        sur::smem_desc(smem_u32(s_b), sur::kLBO, 256), idesc_half(PIECE), 0u);
            sur::tc_commit(&s_mbar);
        };
        PairAcc2 acc2 = {dup2(0.f), dup2(0.f), dup2(0.f), dup2(0.f), dup2(0.f), 0.f};
        const bool anyfluid = __any_sync(kFull, fluid);
        uint32_t lp = list0, hits = 0;                  // next word of this lane's list, its hits
        for (int g = w; g < kBuilders; g += NW) build(0, g);
        sur::fence_async_shared();
        if (__syncthreads_and(ok) == 0) {
            if (tid == 0) atomicOr(a.status, kStatusTimeout);
            mbar_wait_bounded(&s_bar, phase ^ 1u);   // let copies in flight land first
            break;
        }
        if (tid == 0) issue();
        if (tid == 0 && nui < nunits) {
            asm volatile("cp.async.wait_all;" ::: "memory");
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(s_nx + 2)),
                         "l"(a.key + s_nx[0])
                         : "memory");
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(s_nx + 3)),
                         "l"(a.key + s_nx[1] - 1)
                         : "memory");
        }
        // fill the lists piece by piece; a warp one of whose lists is nearly
        // full evaluates its pairs and goes on where it stopped
        bool full = false;
        do {
            // this warp's window of each run (lane r: run r), in staged indexes
            uint32_t win_a = 0, win_b = 0;
            if (lane < 9 && act) {
                const uint32_t s0 = s_base[lane] - s_rs[lane];
                win_a = s0 + s_off[lane][xlo - ulo];
                win_b = s0 + s_off[lane][xhi + 1 - ulo];
            }
            uint32_t runs = __ballot_sync(kFull, win_a < win_b);   // runs left to read
            uint32_t wa = 0xffffffffu, wb = 0;                     // the window in hand
            auto next_window = [&]() {
                const int r = __ffs(runs) - 1;
                wa = __shfl_sync(kFull, win_a, r & 31);
                wb = __shfl_sync(kFull, win_b, r & 31);
                if (!runs) wa = 0xffffffffu;
                runs &= runs - 1;
            };
            uint32_t k = 0, c = 0;                       // piece; its columns below c are done
            bool in_piece = full;
            if (full) {                                  // goes on where it stopped
                k = s_stop[w][0];
                c = s_stop[w][1];
                wa = s_stop[w][2];
                wb = s_stop[w][3];
                runs = s_stop[w][4];
                full = false;
            } else {
                next_window();
            }
            while (k < npc) {
                const bool more = k + 1 < npc;
                if (!in_piece) {
                    ok = __all_sync(kFull, mbar_sleep_bounded(&s_mbar, mphase));
                    if (!ok) break;
                    mphase ^= 1u;
                    sur::tc_fence_after();
                    // the next piece's rows, now that the MMA has read this one's
                    if (more) {
                        for (int g = w; g < kBuilders; g += NW) build(k + 1, g);
                        __syncwarp();
                    }
                    c = 0;
                    in_piece = true;
                }
                const uint32_t p0 = k * PIECE, p1 = p0 + PIECE;
                const uint32_t tcol = lane_base + part * kPartCols;
                const uint32_t e0 = (p0 + (TURN ? 0u : (uint32_t)part)) * 16u;
                while (wa < p1) {
                    // columns [ca, cb) of this part.
                    // The test rejects the neighbouring columns of a load (of
                    // candidates outside the window), so loads are cut at 8.
                    const uint32_t ja = wa > p0 ? wa - p0 : 0u, jb = (wb < p1 ? wb : p1) - p0;
                    const uint32_t ca = TN::before(ja, part) & ~7u, cb = TN::before(jb, part);
                    c = ca > c ? ca : c;
                    while (c < cb) {
                        full = __any_sync(kFull, lp >= list0 + WCAP * 256u);
                        if (full) break;
                        const uint32_t rem = cb - c, ec = e0 + c * (16u * SPLIT);
                        uint32_t m;
                        if (rem > 24u) {
                            m = signs32(tcol + c);
                            c += 32u;
                        } else if (rem > 8u) {
                            m = signs16(tcol + c);
                            c += 16u;
                        } else {
                            m = signs8(tcol + c);
                            c += 8u;
                        }
                        hits += __popc(m);
                        push_word(lp, m, ec);
                    }
                    if (full || wb > p1) break;          // goes on in the next piece
                    next_window();
                }
                if (full) {
                    if (lane == 0) {
                        s_stop[w][0] = k;
                        s_stop[w][1] = c;
                        s_stop[w][2] = wa;
                        s_stop[w][3] = wb;
                        s_stop[w][4] = runs;
                    }
                    break;
                }
                if (more) {
                    // the last warp done with the piece issues the next one's MMA
                    sur::tc_fence_before();
                    __syncwarp();
                    if (lane == 0) {
                        __threadfence_block();
                        if (atomicAdd(&s_arr, 1u) == (uint32_t)NW - 1u) {
                            __threadfence_block();
                            s_arr = 0u;
                            issue();
                        }
                    }
                    __syncwarp();
                }
                ++k;
                in_piece = false;
            }
            if (!full) {
                // every piece read (or a wait that gave up): the last one's
                // accumulators before the next unit's first MMA (the barrier
                // below), the next unit's plan, then its cell offsets
                sur::tc_fence_before();
                if (w == 0) {
                    asm volatile("cp.async.wait_all;" ::: "memory");
                    __syncwarp();
                    UnitPlan p;
                    p.i0 = kNoUnit;
                    if (s_nui < nunits)
                        p = plan_unit(d, make_uint2(s_nx[0], s_nx[1]), s_nx[2], s_nx[3]);
                    if (lane == 0) s_plan[sb ^ 1] = p;
                }
                ok = __syncthreads_and(ok) != 0;
                if (!ok) break;
                if (s_plan[sb ^ 1].i0 != kNoUnit) fetch_offsets(s_plan[sb ^ 1], s_offb[sb ^ 1]);
            }
            // pair phase: each lane pops its hits, two per iteration (the packed
            // halves); lanes that run out get the pad, which contributes
            // nothing and is not counted
            const uint32_t mx = __reduce_max_sync(kFull, hits);
            const uint32_t pad_base = kPad + 16u * (TURN ? 1u + (uint32_t)part : (uint32_t)SPLIT);
            const uint32_t mp = TN::M * (uint32_t)part;
            asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(lp), "r"(0u), "r"(pad_base)
                         : "memory");
            HitCursor hc = {0u, pad_base, 0u, pad_base, list0};
            asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];"
                         : "=r"(hc.next_m), "=r"(hc.next_base)
                         : "r"(list0)
                         : "memory");
            hc.rp = list0 + 256u < lp ? list0 + 256u : lp;
            for (uint32_t t = 0; t < mx; t += 2) {
                uint32_t e0 = pop_hit<SPLIT, TURN>(hc, lp, mp), e1 = pop_hit<SPLIT, TURN>(hc, lp, mp);
                if (!in_bounds(e0 < s_base[9] * 16u || e0 == kPad, d.status)) e0 = kPad;
                if (!in_bounds(e1 < s_base[9] * 16u || e1 == kPad, d.status)) e1 = kPad;
                const float4 pa = *reinterpret_cast<const float4*>(s_raw + e0);
                const float4 va = *reinterpret_cast<const float4*>(s_raw + SH::stage_bytes + e0);
                const float4 pb = *reinterpret_cast<const float4*>(s_raw + e1);
                const float4 vb = *reinterpret_cast<const float4*>(s_raw + SH::stage_bytes + e1);
                // exact difference in fixed point, rounded once
                const float2 dx = __fmul2_rn(ff2((float)(int)(xi - __float_as_uint(pa.x)),
                                                 (float)(int)(xi - __float_as_uint(pb.x))),
                                             dup2(fx_len));
                const float2 m1 = dup2(-1.0f);
                const float2 dy = __ffma2_rn(ff2(pa.y, pb.y), m1, dup2(pi.y));
                const float2 dz = __ffma2_rn(ff2(pa.z, pb.z), m1, dup2(pi.z));
                if (anyfluid)
                    pair_terms2<KERN, true>(d, c0, pi, vi, ci, dx, dy, dz, pa, va, pb, vb, acc2);
                else
                    pair_terms2<KERN, false>(d, c0, pi, vi, ci, dx, dy, dz, pa, va, pb, vb, acc2);
            }
            acc.np += (uint32_t)acc2.npf.x + (uint32_t)acc2.npf.y;
            acc2.npf = dup2(0.f);
            lp = list0;
            hits = 0;
        } while (full);
        if (!ok) {
            if (tid == 0) atomicOr(a.status, kStatusTimeout);
            // let an MMA in flight land first
            mbar_wait_bounded(&s_mbar, mphase);
            break;
        }
        add_pairs2(acc2, acc);
    } else {
        if (w == 0) make_plan(&s_plan[sb ^ 1], s_nui);
        __syncthreads();
        if (s_plan[sb ^ 1].i0 != kNoUnit) fetch_offsets(s_plan[sb ^ 1], s_offb[sb ^ 1]);
        // candidates straight from global memory (unit too large to stage):
        // FP32 test on the cell-relative positions, 32-bit lists in the
        // staging area
        uint32_t* lst = reinterpret_cast<uint32_t*>(s_raw) + w * (FBCAP * 32);
        const int ey = act ? xhi : xlo - 1;   // no cells for a warp without particles
        const float4 pc = valid ? a.posc[i] : make_float4(0.f, 0.f, 0.f, 0.f);
        uint32_t cnt = 0;
        auto flush = [&]() {
            const uint32_t mx = __reduce_max_sync(kFull, cnt);
            for (uint32_t t = 0; t < mx; ++t) {
                if (t < cnt) {
                    const uint32_t e = lst[t * 32 + lane];
                    uint32_t j = e & kIdxMask;
                    if (!in_bounds(j < d.n, d.status)) j = i;
                    const float ox = (float)((int)((e >> 26) & 3u) - 1);
                    const float oy = (float)((int)((e >> 28) & 3u) - 1);
                    const float oz = (float)((int)(e >> 30) - 1);
                    const float4 pj = __ldg(a.posc + j);
                    const float4 vj = __ldg(a.velrhop + j);
                    pair_terms<KERN>(d, c0, pc, vi, ci, fmaf(ox, d.csf, pc.x) - pj.x,
                                           fmaf(oy, d.csf, pc.y) - pj.y,
                                           fmaf(oz, d.csf, pc.z) - pj.z, pj, vj, acc);
                }
            }
            acc.np += cnt;
            cnt = 0;
        };
        for (int r = 0; r < 9; ++r) {
            const int dy = r % 3 - 1, dz = r / 3 - 1;
            const float qy = fmaf((float)(-dy), d.csf, pc.y);
            const float qz = fmaf((float)(-dz), d.csf, pc.z);
            const uint32_t code_yz = ((uint32_t)(1 - dy) << 28) | ((uint32_t)(1 - dz) << 30);
            for (int xx = xlo + (part + r) % SPLIT; xx <= ey; xx += SPLIT) {
                const uint32_t gs = s_off[r][xx - ulo], ge = s_off[r][xx - ulo + 1];
                const int ox = cx - xx;
                const bool adj = valid && ox >= -1 && ox <= 1;
                if (gs == ge) continue;
                const float qx = fmaf((float)ox, d.csf, pc.x);
                const uint32_t code = code_yz | ((uint32_t)(ox + 1) << 26);
                for (uint32_t c0i = gs; c0i < ge; c0i += FBCAP) {
                    const uint32_t c1 = (ge - c0i) > (uint32_t)FBCAP ? c0i + FBCAP : ge;
                    if (__reduce_max_sync(kFull, cnt) + (c1 - c0i) > (uint32_t)FBCAP) flush();
#pragma unroll 4
                    for (uint32_t j = c0i; j < c1; ++j) {
                        const float4 pj = __ldg(a.posc + j);
                        const float dx = qx - pj.x, dy2 = qy - pj.y, dz2 = qz - pj.z;
                        const float d2 = fmaf(dx, dx, fmaf(dy2, dy2, dz2 * dz2));
                        if (adj && d2 < d.r2max) {
                            lst[cnt * 32 + lane] = j | code;
                            ++cnt;
                        }
                    }
                }
            }
        }
        flush();
        fence_staging();   // the lists lie where the next unit's copies go
    }

    // parts 1 .. SPLIT-1 hand their sums to part 0, which adds them in part
    // order (a fixed order).  The barrier also ends the unit: staging, lists
    // and the next unit's offsets are free or complete behind it, and the
    // sums are not written again before the next unit's barriers.
    float* s_comb = reinterpret_cast<float*>(s_raw + SH::c_off);
    if (part > 0) {
        float* c = s_comb + (size_t)(w - W) * (7 * 32) + lane;
        c[0 * 32] = acc.ax;
        c[1 * 32] = acc.ay;
        c[2 * 32] = acc.az;
        c[3 * 32] = acc.dr;
        c[4 * 32] = acc.mu;
        c[5 * 32] = __uint_as_float(acc.np);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (part == 0) {
#pragma unroll
        for (int pp = 1; pp < SPLIT; ++pp) {
            const float* c = s_comb + (size_t)(w + (pp - 1) * W) * (7 * 32) + lane;
            acc.ax += c[0 * 32];
            acc.ay += c[1 * 32];
            acc.az += c[2 * 32];
            acc.dr += c[3 * 32];
            acc.mu = fmaxf(acc.mu, c[4 * 32]);
            acc.np += __float_as_uint(c[5 * 32]);
        }
    }
    if (part == 0) {                                // writes these particles' results
        const float m = d.mass;
        // boundary particles keep gravity only (their momentum sums are dropped)
        const float4 out = make_float4(fmaf(m, fluid ? acc.ax : 0.f, d.gx),
                                       fmaf(m, fluid ? acc.ay : 0.f, d.gy),
                                       fmaf(m, fluid ? acc.az : 0.f, d.gz), m * acc.dr);
        const uint32_t npairs = valid ? acc.np - 1u : 0u;   // without the pair (i, i)
        if (valid) {
            a.ace[i] = out;
            if (COUNTS) a.nnb[i] = npairs;
        }
        // this instance's CFL maxima (non-negative floats order like their bits)
        float am = (valid && fluid) ? out.x * out.x + out.y * out.y + out.z * out.z : 0.f;
        if (!(am == am)) am = 0.f;
        float cm = valid ? ci : 0.f;
        float mm = (valid && fluid) ? acc.mu : 0.f;
        am = warp_max(am);
        cm = warp_max(cm);
        mm = warp_max(mm);
        if (lane == 0 && act) {
            atomicMax(d.is.terms + 3 * q + 0, __float_as_uint(am));
            atomicMax(d.is.terms + 3 * q + 1, __float_as_uint(cm));
            atomicMax(d.is.terms + 3 * q + 2, __float_as_uint(mm));
        }
        const bool bad = valid && !(isfinite(out.x) && isfinite(out.y) && isfinite(out.z) &&
                                    isfinite(out.w));
        const uint32_t tf = __reduce_add_sync(kFull, fluid ? npairs : 0u);
        const uint32_t tb = __reduce_add_sync(kFull, fluid ? 0u : npairs);
        if (__any_sync(kFull, bad) && lane == 0) s_ru[w][2] = kStatusNonFinite;
        if (lane == 0) {
            s_ru[w][0] += tf;
            s_ru[w][3] += tb;
        }
    }
    sb ^= 1;
    }
    // (a wait that gave up: the next unit's record may still be on its way)
    asm volatile("cp.async.wait_all;" ::: "memory");
    // the last block to finish rearms the unit counter for the next launch
    // (every block's last take precedes its finish ticket)
    __threadfence();
    if (tid == 0 && atomicAdd(a.sched + 1, 1u) == gridDim.x - 1u) {
        a.sched[0] = 0u;
        a.sched[1] = 0u;
    }

    sur::tc_fence_before();
    __syncthreads();
    if (w == 0) sur::tmem_dealloc(tmem, PIECE);
    if (tid == 0) {
        uint4 u = make_uint4(0u, 0u, 0u, 0u);
        for (int k = 0; k < NW; ++k) {
            u.x += s_ru[k][0];
            u.y += s_ru[k][1];
            u.z |= s_ru[k][2];
            u.w += s_ru[k][3];
        }
        a.part_u[blockIdx.x] = u;
    }
    if (a.ticket) {
        // the last block to finish runs the Sec. 3.3 reductions (every
        // thread's maxima atomics and thread 0's partials fenced first)
        __shared__ bool s_lastblk;
        __threadfence();
        __syncthreads();
        if (tid == 0) s_lastblk = atomicAdd(a.ticket, 1u) == gridDim.x - 1u;
        __syncthreads();
        if (s_lastblk) {
            __threadfence();
            reduce_counters_and_dt(d, a.red, a.set_dt);
            if (tid == 0) *a.ticket = 0u;
        }
    }
}

template <int W, int SPLIT, int STAGE, int WCAP, int PIECE, int MINB>
Variant tc_variant() {
    Variant v{};
    v.warps = W;
    v.split = SPLIT;
    v.stage = STAGE;
    v.fn[0][0] = k_interact_tc<W, SPLIT, STAGE, WCAP, PIECE, MINB, false, 0>;
    v.fn[0][1] = k_interact_tc<W, SPLIT, STAGE, WCAP, PIECE, MINB, true, 0>;
    v.fn[1][0] = k_interact_tc<W, SPLIT, STAGE, WCAP, PIECE, MINB, false, 1>;
    v.fn[1][1] = k_interact_tc<W, SPLIT, STAGE, WCAP, PIECE, MINB, true, 1>;
    v.smem = TcShape<W, SPLIT, STAGE, WCAP, PIECE>::smem;
    v.max_per_sm = 512 / PIECE;
    return v;
}

}  // namespace

// Large systems run best in 128-particle units on two blocks per SM, small
// ones and ensembles of small ones in 64-particle units on four (sph_autotune
// times them all; ms per launch on one GB300, 128 / 64: 35.4M particles 18.4 /
// 24.2, 1.39M 0.701 / 0.865, 60k 0.072 / 0.077, 256 dam breaks 3.20 / 3.15, 17k
// 0.0212 / 0.0196).  Between the first and the third, fourth and seventh,
// shared memory moves from staged candidates to hit words, for larger h/dp (more
// hits per particle); 200k particles, variants 0 / 2 / 3 / 6: h/dp 1.3 0.118 / 0.118 /
// 0.119 / 0.126, 1.5 0.161 / 0.146 / 0.142 / 0.157, 1.7 0.291 / 0.253 / 0.218 / 0.250,
// 1.8 0.363 / 0.371 / 0.345 / 0.318 (beyond 1.8 the shapes with 2,048 slots, 0.325 and
// less).  Variant 5 is for a spray: 300k particles at random, one in three cells
// 0.90 ms (variant 0 1.69, variant 1 1.12), one per cell 0.198 (0.347, 0.242).
Variant tc_variant_n(int k) {
    switch (k) {
        case 0: return tc_variant<4, 2, 1760, 16, 256, 2>();
        case 1: return tc_variant<2, 2, 896, 16, 128, 4>();
        case 2: return tc_variant<4, 2, 1664, 18, 256, 2>();
        case 3: return tc_variant<4, 2, 1536, 20, 256, 2>();
        case 4: return tc_variant<2, 2, 832, 18, 128, 4>();
        case 5: return tc_variant<1, 4, 768, 14, 128, 4>();
        default: return tc_variant<4, 2, 1408, 22, 256, 2>();
    }
}

}  // namespace sph
