// Device helpers shared by the interaction kernels (sph_kernels.cu and
// sph_interact_tc.cu): mbarrier and bulk-copy wrappers, the pair terms of
// Eqs. 7 and 9 (scalar and packed FP32) and the Sec. 3.3 reductions that the
// last interaction block runs.
#pragma once
#include "sph_internal.cuh"

namespace sph {

namespace {

constexpr uint32_t kFull = 0xffffffffu;

__device__ __forceinline__ float sqrt_approx(float x) {
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Index q with base[q] <= v < base[q + 1] (base has n + 1 ascending entries).
__device__ __forceinline__ uint32_t find_instance(const uint32_t* __restrict__ base, uint32_t n,
                                                  uint32_t v) {
    uint32_t lo = 0, hi = n;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (__ldg(base + mid) <= v) lo = mid;
        else hi = mid;
    }
    return lo;
}

constexpr uint32_t kIdxMask = (1u << 26) - 1;
constexpr uint32_t kWaitLimit = 1u << 22;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
                 : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}

// 1-D bulk copy global -> shared (TMA engine), completion counted on bar.
// Both addresses 16-byte aligned, bytes a multiple of 16.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
            "r"(smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// This thread's plain stores to the staging area before the bulk copies that
// another unit issues into it behind the next block barrier (the copies are of
// the asynchronous proxy, which a barrier alone does not order after them).
__device__ __forceinline__ void fence_staging() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}" : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}

// Bounded wait for phase `parity` of bar; false if it gave up.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity) {
    for (uint32_t k = 0; k < kWaitLimit; ++k)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

struct PairAcc {
    float ax, ay, az, dr, mu;
    uint32_t np;
};

// Pair terms of Eqs. 7 and 9 for i (pi, vi) and a neighbour j (pj, vj) at
// offset (dx, dy, dz) = r_i - r_j.  The momentum terms are accumulated for
// every particle; the caller keeps them only for fluid particles, since
// boundary particles never move (Sec. 2.3).
// KERN: 0 Wendland C2, 1 cubic spline (Sec. 2.2).
template <int KERN>
__device__ __forceinline__ void pair_terms(const Dev& d, float c0, const float4& pi,
                                           const float4& vi, float ci, float dx, float dy, float dz,
                                           const float4& pj, const float4& vj, PairAcc& s) {
    const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    // grad_i W = F r_ij.  Wendland C2: F = -5 aD/h^2 (1 - q/2)^3.  Cubic
    // spline: F = aD/h^2 (9/4 q - 3) for q < 1, -3/4 aD/h^2 (2 - q)^2 / q
    // for 1 <= q < 2 (a select: the outer piece is infinite at q = 0).
    const float q = sqrt_approx(d2) * d.inv_h;
    float shape;
    if (KERN == 1) {
        const float wo = 2.0f - q;
        const float outer = -0.75f * (wo * wo) * rcp_approx(q);
        const float inner = fmaf(2.25f, q, -3.0f);
        shape = q < 1.0f ? inner : outer;
    } else {
        const float wq = fmaf(-0.5f, q, 1.0f);
        shape = wq * wq * wq;
    }
    const float F = d.fc * shape;
    const float dvx = vi.x - vj.x, dvy = vi.y - vj.y, dvz = vi.z - vj.z;
    const float vr = fmaf(dvx, dx, fmaf(dvy, dy, dvz * dz));
    s.dr = fmaf(vr, F, s.dr);                                  // Eq. 7
    const float nu = d.h * vr * rcp_approx(d2 + d.eta2);       // Sec. 2.2
    const float rrj = vj.w * d.inv_rho0;
    const float cj = c0 * rrj * rrj * rrj;
    // Pi_ij only for approaching pairs (v_ij . r_ij < 0, the sign of nu)
    const float visc = -d.alpha * (ci + cj) * fminf(nu, 0.f) * rcp_approx(vi.w + vj.w);
    const float f = (pi.w + pj.w + visc) * F;                  // Eq. 9
    s.ax = fmaf(-f, dx, s.ax);
    s.ay = fmaf(-f, dy, s.ay);
    s.az = fmaf(-f, dz, s.az);
    s.mu = fmaxf(s.mu, fabsf(nu));
}

// Sec. 3.3 reductions, by one block once every interaction block has
// published its counters (pairs, candidates, status bits) and atomically
// raised the per-instance maxima: the counters are summed (integer sums and
// maxima do not depend on the order), then per instance
//   dt = CFL min( sqrt(h / max|a|), h / (max c + max mu) )
// (0 for instances that are done), and the maxima are cleared for the next
// evaluation.  Loads bypass L1 (the partials may come from the same kernel).
// Run by a block of at most 256 threads (an interaction block).
__device__ void reduce_counters_and_dt(const Dev& d, const ReduceArgs& a, int set_dt) {
    __shared__ unsigned long long s_u[8][3];
    __shared__ uint32_t s_b[8];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    unsigned long long pf = 0, pb = 0, nc = 0;
    uint32_t bad = 0;
    for (uint32_t i = threadIdx.x; i < a.nparts; i += blockDim.x) {
        const uint4 u = __ldcg(a.part_u + i);
        pf += u.x;
        nc += u.y;
        bad |= u.z;
        pb += u.w;
    }
    for (int o = 16; o; o >>= 1) {
        pf += __shfl_xor_sync(kFull, pf, o);
        pb += __shfl_xor_sync(kFull, pb, o);
        nc += __shfl_xor_sync(kFull, nc, o);
        bad |= __shfl_xor_sync(kFull, bad, o);
    }
    if (lane == 0) {
        s_u[w][0] = pf;
        s_u[w][1] = pb;
        s_u[w][2] = nc;
        s_b[w] = bad;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long qf = 0, qb = 0, qc = 0;
        uint32_t bb = 0;
        for (int k = 0; k < nw; ++k) {
            qf += s_u[k][0];
            qb += s_u[k][1];
            qc += s_u[k][2];
            bb |= s_b[k];
        }
        a.counters[0] += qf + qb;
        a.counters[1] += qc;
        a.counters[2] = qf + qb;
        a.counters[3] = qc;
        a.counters[4] = qf;
        a.counters[5] = qb;
        a.counters[6] += qf;
        a.counters[7] += qb;
        if (bb) atomicOr(a.status, bb);
    }
    for (uint32_t q = threadIdx.x; q < d.n_inst; q += blockDim.x) {
        uint32_t* tm = d.is.terms + 3 * q;
        const float fa = __uint_as_float(__ldcg(tm + 0));
        const float fc = __uint_as_float(__ldcg(tm + 1));
        const float fm = __uint_as_float(__ldcg(tm + 2));
        const double amax = sqrt((double)fa);
        if (set_dt) {
            double dt = 0.0;
            if (!d.is.done[q]) {
                if (d.dt_fixed > 0.0) {
                    dt = d.dt_fixed;
                } else {
                    const double dtf = amax > 0.0 ? sqrt(d.h_d / amax) : INFINITY;
                    const double dtc = d.h_d / ((double)fc + (double)fm);
                    dt = d.cfl * (dtf < dtc ? dtf : dtc);
                }
            }
            d.is.dt[q] = dt;
            d.is.last[3 * q + 0] = (float)amax;
            d.is.last[3 * q + 1] = fc;
            d.is.last[3 * q + 2] = fm;
        }
        tm[0] = 0u;
        tm[1] = 0u;
        tm[2] = 0u;
    }
}

// Packed accumulators of two pair streams (the two pairs a lane evaluates
// per step of the pair phase), one in each half of a float2.  The momentum
// sums hold +sum f r_ij (negated once by add_pairs2, which is exact).
struct PairAcc2 {
    float2 ax, ay, az, dr, npf;
    float mu;
};

__device__ __forceinline__ float2 ff2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }

// pair_terms for two candidates of a conservative pre-filter at once, with
// the Blackwell packed FP32 operations (__ffma2_rn, __fadd2_rn, __fmul2_rn:
// two FP32 results per instruction, each rounded as the scalar operation);
// the square roots, reciprocals, min/max and the support test stay scalar.
// The FP32 neighbour test decides and counts a pair: use = [d2 < (2h)^2], the
// saturated sign of 2^100 ((2h)^2 - d2), exact (power-of-two scaling).  A
// candidate far outside the support contributes exactly nothing and is not
// counted, which lets lane work be padded with one.  Masks are products with
// 0 or 1 rather than selects, keeping the integer/logic pipe free.  MOM:
// evaluate the momentum terms (a warp-uniform choice).
// Same arithmetic per pair as pair_terms, factor by factor: with the constant
// factors pulled out of the sums a launch is 0.5 to 1% faster (1.39M particles
// 0.697 against 0.701 ms), but every term is rounded differently, and after 30
// steps the positions are 1.2e-9 instead of 0.9e-9 from those of another order of
// the same sums.
template <int KERN, bool MOM>
__device__ __forceinline__ void pair_terms2(const Dev& d, float c0, const float4& pi,
                                            const float4& vi, float ci, float2 dx, float2 dy,
                                            float2 dz, const float4& pa, const float4& va,
                                            const float4& pb, const float4& vb, PairAcc2& s) {
    const float2 d2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
    const float r2s = d.r2max * 0x1p100f;
    const float2 use = ff2(__saturatef(fmaf(d2.x, -0x1p100f, r2s)),
                           __saturatef(fmaf(d2.y, -0x1p100f, r2s)));
    s.npf = __fadd2_rn(s.npf, use);
    const float2 q = __fmul2_rn(ff2(sqrt_approx(d2.x), sqrt_approx(d2.y)), dup2(d.inv_h));
    float2 shape;
    if (KERN == 1) {
        const float2 wo = __ffma2_rn(q, dup2(-1.0f), dup2(2.0f));
        const float2 outer =
            __fmul2_rn(__fmul2_rn(dup2(-0.75f), __fmul2_rn(wo, wo)), ff2(rcp_approx(q.x), rcp_approx(q.y)));
        const float2 inner = __ffma2_rn(dup2(2.25f), q, dup2(-3.0f));
        shape = ff2(q.x < 1.0f ? inner.x : outer.x, q.y < 1.0f ? inner.y : outer.y);
    } else {
        const float2 wq = __ffma2_rn(dup2(-0.5f), q, dup2(1.0f));
        shape = __fmul2_rn(__fmul2_rn(wq, wq), wq);
    }
    // (the mask before the shape: exact, and fc, 1e35 at h = 0.1 um, does not
    // overflow on the shape of a pad 32 cells away)
    const float2 F = __fmul2_rn(__fmul2_rn(dup2(d.fc), use), shape);
    const float2 m1 = dup2(-1.0f);
    const float2 dvx = __ffma2_rn(ff2(va.x, vb.x), m1, dup2(vi.x));
    const float2 dvy = __ffma2_rn(ff2(va.y, vb.y), m1, dup2(vi.y));
    const float2 dvz = __ffma2_rn(ff2(va.z, vb.z), m1, dup2(vi.z));
    const float2 vr = __ffma2_rn(dvx, dx, __ffma2_rn(dvy, dy, __fmul2_rn(dvz, dz)));
    s.dr = __ffma2_rn(vr, F, s.dr);                                 // Eq. 7
    if (MOM) {
        const float2 de = __fadd2_rn(d2, dup2(d.eta2));
        const float2 nu = __fmul2_rn(__fmul2_rn(dup2(d.h), vr), ff2(rcp_approx(de.x), rcp_approx(de.y)));
        const float2 rrj = __fmul2_rn(ff2(va.w, vb.w), dup2(d.inv_rho0));
        const float2 cj = __fmul2_rn(__fmul2_rn(__fmul2_rn(dup2(c0), rrj), rrj), rrj);
        const float2 rs = __fadd2_rn(dup2(vi.w), ff2(va.w, vb.w));
        const float2 nmin = ff2(fminf(nu.x, 0.f), fminf(nu.y, 0.f));
        const float2 visc = __fmul2_rn(
            __fmul2_rn(__fmul2_rn(dup2(-d.alpha), __fadd2_rn(dup2(ci), cj)), nmin),
            ff2(rcp_approx(rs.x), rcp_approx(rs.y)));
        const float2 f = __fmul2_rn(__fadd2_rn(__fadd2_rn(dup2(pi.w), ff2(pa.w, pb.w)), visc), F);
        s.ax = __ffma2_rn(f, dx, s.ax);                              // Eq. 9 (sign later)
        s.ay = __ffma2_rn(f, dy, s.ay);
        s.az = __ffma2_rn(f, dz, s.az);
        s.mu = fmaxf(s.mu, fmaxf(fabsf(nu.x) * use.x, fabsf(nu.y) * use.y));
    }
}

// The two streams' sums, in a fixed order.
__device__ __forceinline__ void add_pairs2(const PairAcc2& s, PairAcc& acc) {
    acc.ax -= s.ax.x + s.ax.y;
    acc.ay -= s.ay.x + s.ay.y;
    acc.az -= s.az.x + s.az.y;
    acc.dr += s.dr.x + s.dr.y;
    acc.mu = fmaxf(acc.mu, s.mu);
}

}  // namespace

}  // namespace sph
