// pg_device.cuh -- device-side building blocks shared by the pg kernels:
// packed FP32x2 arithmetic, the MUFU reciprocal square root, mbarriers with
// time-limited waits, bulk global->shared copies, and the status word the
// kernels report errors through. sm_100-family only (f32x2 needs sm_100+).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "pg_internal.h"

namespace pg {

typedef unsigned long long u64;

// ---------------------------------------------------------------- f32x2
// A u64 holds two FP32 lanes {lo, hi}; one instruction processes both.
__device__ __forceinline__ u64 pk2(float lo, float hi)
{
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void up2(u64 v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ u64 f2fma(u64 a, u64 b, u64 c)
{
    u64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ u64 f2add(u64 a, u64 b)
{
    u64 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 f2sub(u64 a, u64 b)
{
    u64 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 f2mul(u64 a, u64 b)
{
    u64 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// MUFU reciprocal square root, the hardware approximation (the GPU's
// counterpart of the paper's VRSQRTPS); flushes subnormals.
__device__ __forceinline__ float rsq(float x)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Knuth's TwoSum: s + e == a + b exactly (round-to-nearest, no overflow).
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// Packed TwoSum on both lanes.
__device__ __forceinline__ void two_sum2(u64 a, u64 b, u64 &s, u64 &e)
{
    s = f2add(a, b);
    u64 bb = f2sub(s, a);
    e = f2add(f2sub(a, f2sub(s, bb)), f2sub(b, bb));
}

// Fold a tile partial p into the running compensated pair (hi, lo).
__device__ __forceinline__ void fold2(u64 &hi, u64 &lo, u64 p)
{
    u64 s, e;
    two_sum2(hi, p, s, e);
    hi = s;
    lo = f2add(lo, e);
}

// ---------------------------------------------------------------- timers
__device__ __forceinline__ u64 global_ns()
{
    u64 t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// first error wins; the host reads the word after the launch sequence
__device__ __forceinline__ void report(int *status, int code, int where)
{
    if (status) {
        if (atomicCAS(status, 0, code) == 0) atomicExch(status + 1, where);
    }
}

// ---------------------------------------------------------------- mbarrier
// one {A, G1} table entry for s in [2, s_max]: byte offset from the FP32
// bits of s by shift and mask, then a shared load (no integer multiply);
// tbase = the table's shared address minus 8 times the index of s = 2
__device__ __forceinline__ float2 tab_at(unsigned tbase, unsigned bits, int shift3)
{
    float2 v;
    const unsigned addr = tbase + ((bits >> shift3) & ~7u);
    asm("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr));
    return v;
}

// the same for a table with a potential half: {A, G1, A_p, P1} per knot,
// 16 bytes; tbase = the table's shared address minus 16 times the index of
// s = 2
__device__ __forceinline__ float4 tab4_at(unsigned tbase, unsigned bits, int shift4)
{
    float4 v;
    const unsigned addr = tbase + ((bits >> shift4) & ~15u);
    asm("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
        : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
    return v;
}

// min(s, s_max) for s > 0 as the integer minimum of the FP32 bit patterns
// (positive floats order like their bits; a NaN also maps to s_max): the
// clamp then runs on the ALU pipe instead of the busier FMA pipe
__device__ __forceinline__ float clamp_pos(float s, unsigned smax_bits)
{
    return __uint_as_float(min(__float_as_uint(s), smax_bits));
}

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

__device__ __forceinline__ void mbar_fence_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_inval(uint64_t *bar)
{
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// arrive once and announce `bytes` of transaction for the current phase
__device__ __forceinline__ void mbar_arrive_tx(uint64_t *bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                 ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint64_t *bar, unsigned parity)
{
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n"
                 " mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                 " selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}

// Wait for the phase with the given parity to complete, giving up after
// `limit_ns` nanoseconds of wall time. Returns false on time-out.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, unsigned parity, u64 limit_ns)
{
    if (mbar_try(bar, parity)) return true;
    u64 t0 = global_ns();
    for (unsigned it = 0;; ++it) {
        if (mbar_try(bar, parity)) return true;
        if ((it & 63u) == 63u && global_ns() - t0 > limit_ns) return false;
    }
}

// make prior generic-proxy accesses to shared memory ordered before later
// async-proxy (bulk copy) accesses
__device__ __forceinline__ void fence_proxy_async()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Bulk copy of `bytes` (multiple of 16, both addresses 16-byte aligned)
// from global to this CTA's shared memory, completing on `bar`.
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, unsigned bytes, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
        ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

// ---------------------------------------------------------------- misc
__device__ __forceinline__ double4 ldg_d4(const double4 *p)
{
    double4 r;
    const double2 *q = reinterpret_cast<const double2 *>(p);
    double2 a = __ldg(q), b = __ldg(q + 1);
    r.x = a.x; r.y = a.y; r.z = b.x; r.w = b.y;
    return r;
}

// record i as a double-float pair: (hi, w) then (lo, w), lo = x - hi, w the
// record's fourth value (the mass of a j record; eps^2 of an i record with
// per-i softening, else 0)
__device__ __forceinline__ void pack_hilo_one(const double4 *__restrict__ in, long long i,
                                              float4 *__restrict__ out)
{
    double4 v = in[i];
    float hx = (float)v.x, hy = (float)v.y, hz = (float)v.z;
    out[2 * i] = make_float4(hx, hy, hz, (float)v.w);
    out[2 * i + 1] = make_float4((float)(v.x - (double)hx), (float)(v.y - (double)hy),
                                 (float)(v.z - (double)hz), (float)v.w);
}

// ---------------------------------------------------------------- narrow path
// FP64 centre of each group: midpoint of its i-particles' bounding box
// group g holds i_off[g] .. i_off[g + 1], or without offsets the chunk
// g chunk .. min((g + 1) chunk, ni)
__device__ __forceinline__ void group_ctr_warp(const double4 *__restrict__ xi,
                                               const long long *__restrict__ i_off, long long g,
                                               long long chunk, long long ni, int lane,
                                               double4 *__restrict__ ctr)
{
    const long long ib = i_off ? i_off[g] : g * chunk;
    const long long ie = i_off ? i_off[g + 1] : min((g + 1) * chunk, ni);
    double lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (long long i = ib + lane; i < ie; i += 32) {
        double4 v = xi[i];
        lo[0] = fmin(lo[0], v.x); lo[1] = fmin(lo[1], v.y); lo[2] = fmin(lo[2], v.z);
        hi[0] = fmax(hi[0], v.x); hi[1] = fmax(hi[1], v.y); hi[2] = fmax(hi[2], v.z);
    }
    for (int c = 0; c < 3; ++c)
        for (int o = 16; o; o >>= 1) {
            lo[c] = fmin(lo[c], __shfl_xor_sync(0xffffffffu, lo[c], o));
            hi[c] = fmax(hi[c], __shfl_xor_sync(0xffffffffu, hi[c], o));
        }
    if (lane == 0) {
        bool empty = !(lo[0] <= hi[0]);
        ctr[g] = empty ? make_double4(0, 0, 0, 0)
                       : make_double4(0.5 * (lo[0] + hi[0]), 0.5 * (lo[1] + hi[1]),
                                      0.5 * (lo[2] + hi[2]), 0.0);
    }
}

// The narrow path's preparation, block blk of narrow_prep_blocks: one warp a
// chunk centre in the first of them, then one thread an i record
constexpr int kNarrowPrepThreads = 128;
__host__ __device__ __forceinline__ long long narrow_prep_blocks(long long ni, const NarrowPrep &np)
{
    return (np.nic + kNarrowPrepThreads / 32 - 1) / (kNarrowPrepThreads / 32) +
           (ni + kNarrowPrepThreads - 1) / kNarrowPrepThreads;
}
__device__ __forceinline__ void narrow_prep_block(const double4 *__restrict__ xi, long long ni, const NarrowPrep &np,
                                                  long long blk)
{
    constexpr int kWarps = kNarrowPrepThreads / 32;
    const long long cb = (np.nic + kWarps - 1) / kWarps;
    if (blk == 0 && threadIdx.x < 2) np.queue[threadIdx.x] = 0;
    if (blk < cb) {
        const long long g = blk * kWarps + (threadIdx.x >> 5);
        if (g < np.nic) group_ctr_warp(xi, nullptr, g, np.chunk, ni, threadIdx.x & 31, np.ctr);
        return;
    }
    const long long i = (blk - cb) * kNarrowPrepThreads + threadIdx.x;
    if (i < ni) pack_hilo_one(xi, i, np.ihl);
}

// ---------------------------------------------------------------- tensor cores
// The differences come out short (the tensor cores round them toward zero),
// so the unit they are read in is longer by this. Fitted to the signed errors
// of forces (2 kTcShort) and potentials (kTcShort) against 64 bits, 12 sets
// of 112 to 2080 i against 3e5 to 1e6 j: +4.7e-8 and +2.6e-8 without it. (The
// differences themselves, all weighted alike, are 3.2e-8 short.)
constexpr double kTcShort = 2.5e-8;

__host__ __device__ __forceinline__ long long tc_owner(long long u, long long grid, long long W)
{
    return ((u + 1) * grid - 1) / W;
}

// i-particle i of a tensor-core run, by one warp: the partial sums of its tile
// over the CTAs, the own pair's potential, the units
__device__ __forceinline__ void tc_combine_one(const TcArgs &a, int grid, int self, long long self_off,
                                               double *__restrict__ acc, double *__restrict__ pot, long long i)
{
    const int lane = threadIdx.x & 31;
    const long long t = i / kTcBi, li = i % kTcBi;
    const long long bf = tc_owner(t * a.njt, grid, a.W), bl = tc_owner((t + 1) * a.njt - 1, grid, a.W);
    double s[4] = {0, 0, 0, 0};
    for (long long k = lane; k <= bl - bf; k += 32) {
        const double4 v = a.part[((size_t)t * a.slots + k) * kTcBi + li];
        s[0] += v.x; s[1] += v.y; s[2] += v.z; s[3] += v.w;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
        for (int o = 16; o; o >>= 1) s[q] += __shfl_xor_sync(0xffffffffu, s[q], o);
    if (lane != 0) return;
    const TcGeo &g = *a.geo;
    // the own pair as the loop added it: d = 0 exactly
    if (self) s[3] += (double)__fmul_rn(a.mass[i + self_off], rsq(g.e2));
    const double fa = ldexp((1.0 - kTcShort) * (1.0 - kTcShort), 2 * (23 - g.e) - g.mexp),
                 fp = ldexp(1.0 - kTcShort, 23 - g.e - g.mexp);
    acc[3 * i] = s[0] * fa;
    acc[3 * i + 1] = s[1] * fa;
    acc[3 * i + 2] = s[2] * fa;
    if (pot) pot[i] = s[3] * fp;
}

// ---------------------------------------------------------------- near pairs
// a loss weight that is not finite in FP32 (or nearly so)
__device__ __forceinline__ bool odd_weight(const double4 w)
{
    return !(fabsf((float)w.x) + fabsf((float)w.y) + fabsf((float)w.z) < 3.0e38f);
}

// Of a near-pair run: the CTAs that hold units of [u, v), asked for by all
// threads of the block: b0 the last that starts at or before u, b1 past the
// last that starts before v (CTAs without units in between). w: two words of
// shared memory.
__device__ __forceinline__ void plan_ctas(const long long *start, int grid, long long u, long long v, int *w,
                                            int &b0, int &b1)
{
    if (threadIdx.x < 2) w[threadIdx.x] = 0;
    __syncthreads();
    int n0 = 0, n1 = 0;
#pragma unroll 8
    for (int b = threadIdx.x; b < grid; b += blockDim.x) {
        const long long s = start[b];
        n0 += s <= u;
        n1 += s < v;
    }
    n0 = __reduce_add_sync(0xffffffffu, n0);
    n1 = __reduce_add_sync(0xffffffffu, n1);
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&w[0], n0);
        atomicAdd(&w[1], n1);
    }
    __syncthreads();
    b0 = w[0] > 0 ? w[0] - 1 : 0;
    b1 = w[1];
}

// The sum of a tile's partials for the 64 i-particles of a 256-thread block,
// i-particle li of its tile: four threads an i take the CTAs in turn and
// are added in order; the tiles of a dense core have most of the CTAs.
// The sum is valid on the first 64 threads.
constexpr int kNearCombineI = 64;
__device__ __forceinline__ double4 near_sum(const long long *start, int grid, int nch, const double4 *part, int Bi,
                                            long long t, int li, bool in)
{
    __shared__ int w[2];
    __shared__ double4 seg[3][kNearCombineI];
    int b0, b1;
    plan_ctas(start, grid, t * nch, (t + 1) * nch, w, b0, b1);
    const int q = threadIdx.x / kNearCombineI, k = threadIdx.x % kNearCombineI;
    double4 s = make_double4(0, 0, 0, 0);
#pragma unroll 4
    for (int b = b0 + q; b < b1; b += 4) {
        if (!in || start[b + 1] <= start[b]) continue;
        const double4 v = ldg_d4(part + (size_t)(t + b) * Bi + li);
        s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
    }
    if (q > 0) seg[q - 1][k] = s;
    __syncthreads();
    if (q == 0)
        for (int g = 0; g < 3; ++g) {
            s.x += seg[g][k].x; s.y += seg[g][k].y; s.z += seg[g][k].z; s.w += seg[g][k].w;
        }
    return s;
}

// The potential term i's own pair added in the loop (d = 0 exactly; i-particle
// k is j record k + self_off), as the
// loop computed it, so that subtracting it leaves no cancellation error:
// Newton -m_k rsqrt(eps^2) (eps of the global setting or of i itself; at
// eps = 0 the pair added nothing); table with a potential m_k psi~(s = 2),
// knot 0's value A_p + 2 P1.
__device__ __forceinline__ double self_potential(const CombineArgs &c, long long k)
{
    const float mk = (float)c.jrec[k + c.self_off].w;
    if (c.newton) {
        const float e2 = c.epsi ? (float)c.xi[k].w : c.eps2;
        return e2 > 0.0f ? -(double)__fmul_rn(mk, rsq(e2)) : 0.0;
    }
    if (c.tabpot) {
        const float4 t0 = c.agp[0];
        return (double)__fmul_rn(mk, __fmaf_rn(2.0f, t0.w, t0.z));
    }
    return 0.0;
}

}  // namespace pg
