// pg_tc.cu -- Newton all pairs with the pair differences on the tensor cores.
//
// The double-float paths spend 9 of their 19 FP32-pipe operations per pair on
// the difference x_j - x_i. A difference is a matrix product with an inner
// dimension of two, [x_j, 1] [1, -x_i]^T, so the 5th-generation tensor cores
// form it exactly and the FP32 pipe keeps the ten operations of the pair term
// (r^2, m/r, m/r^3, the four sums; MUFU rsqrt beside them).
//
// Positions are quantised once to 48-bit fixed point in the cube of the
// j-set (lsb = R 2^-47, R the cube's half side rounded up to a power of two)
// and split into four signed 12-bit digits per axis, each exact in FP16. A
// j record is 16 FP16 values (12 digits and 4 constants), a tile of 128 of
// them the A operand (M = 128 TMEM lanes); the B operand has one row per
// (i, axis) with the place values at that axis's digits and the negated
// digits of x_i at the constants. One MMA (K = 16, FP32 accumulation) gives
// the difference of the upper 24 bits, an integer below 2^24 and so exact;
// a second adds the lower 24 bits' difference, cut off by the tensor core
// near the last place of the result, mostly toward zero: d has an error
// relative to |d|, however far the i-particles are spread (measured against
// 64 bits: 3.2e-8 short on average, at most 1.5e-7, a little over one place).
// What that leaves in forces and potentials is taken out by the unit of the
// differences (kTcShort); they are then as near to 64 bits as the
// double-float kernel's (1048 i, 563704 j: 4.8e-8 and 2.3e-8 against 5.8e-8
// and 2.5e-8; i at 0.5 to 2 eps from a j, eps = 1e-3, median 1.3e-7 and 1.9e-7
// for 300 i, both 1.9e-7 for 1000).
//
// A CTA owns units (tile of 64 i, tile of 128 j), an equal contiguous
// range of them. One thread copies the j tiles in (cp.async.bulk), two issue
// the MMAs of alternate tiles (tcgen05.mma, cta_group::1; barrier tries,
// copies, MMAs and commits each take a thread 70 to 90 clocks, so one
// producer thread bounded a tile at 840 clocks), eight warps read the
// differences from TMEM (tcgen05.ld, four columns ahead) and evaluate: lane
// = j, 32 i per warp in registers, no shared-memory read in the pair loop.
// Every 128 tiles the lanes are added by a transposed butterfly into
// compensated sums. Eight warps of 32 i beat sixteen of 16 i (the barrier
// and address work per tile is paid once for twice the pairs): 2.41 against
// 2.28e12 pairs/s on 131072^2 pairs.
//
// Bound: the FP32 pipe with MUFU beside it. The ten operations alone, from
// registers, run at 9.6 pairs per SM-clock (3.0e12/s), the kernel at 7.4
// (2.3e12); the double-float kernel it replaces ran at 1.24e12.
#include <algorithm>

#include <cuda_fp16.h>

#include "pg_device.cuh"

namespace pg {

namespace {

constexpr int kTcWarps = 8;            // compute warps, two per SM sub-partition
constexpr int kIW = 32;                // i-particles of a warp
constexpr int kTcThreads = kTcWarps * 32 + 128;
constexpr int kTcJ = 128;              // j per tile (TMEM lanes)
constexpr int kDigBytes = kTcJ * 32;   // digits of a j tile
constexpr int kSlotBytes = kDigBytes + kTcJ * 4;   // and its masses
constexpr int kSums = 4 * kIW, kLaneSums = kSums / 32;
constexpr int kFoldTiles = 128;        // j tiles per FP32 partial sum of a lane

// two groups of kIW i per CTA tile; the groups' warps (four each, one per
// TMEM quadrant) share every j tile
constexpr int kBi = kTcBi;
static_assert(kTcBi == 2 * kIW, "two groups");
constexpr int kN = 3 * kBi;            // MMA N: (group, axis, i)
constexpr int kStages = 2;             // TMEM stages of kN columns
constexpr int kSlots = 8;              // staged j tiles
constexpr size_t kTcSmem = (size_t)kSlots * kSlotBytes + 2 * kN * 32 + kTcWarps * 2 * kSums * sizeof(float) +
                           (2 * kSlots + 2 * kStages) * 8 + 48;

// ---------------------------------------------------------------- PTX
// shared-memory operand, K-major without swizzle: core matrices of 8 rows x
// 16 bytes, the two K halves 128 bytes apart, groups of 8 rows 256 apart
__device__ __forceinline__ u64 operand(uint32_t addr)
{
    return (u64)((addr >> 4) & 0x3FFF) | ((u64)(128 >> 4) << 16) | ((u64)(256 >> 4) << 32) | (1ull << 46);
}

__device__ __forceinline__ void mma_f16(uint32_t d, u64 a, u64 b, uint32_t idesc, uint32_t accumulate)
{
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
                 " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}"
                 ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}

// four columns of this warp's lanes
__device__ __forceinline__ void tmem_ld4(uint32_t t, float (&r)[4])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]) : "r"(t));
}
// the loads above done; the registers pass through so that no use moves up
__device__ __forceinline__ void tmem_wait(float (&x)[4], float (&y)[4], float (&z)[4])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(x[0]), "+f"(x[1]), "+f"(x[2]), "+f"(x[3]), "+f"(y[0]), "+f"(y[1]), "+f"(y[2]), "+f"(y[3]),
                   "+f"(z[0]), "+f"(z[1]), "+f"(z[2]), "+f"(z[3])::"memory");
}

__device__ __forceinline__ uint32_t try_wait(uint32_t bar, unsigned parity, unsigned hint)
{
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
                 " selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok) : "r"(bar), "r"(parity), "r"(hint) : "memory");
    return ok;
}

// Wait for a phase, up to the time limit. A failure is recorded once for the
// CTA and ends all its later waits; the caller's control flow does not depend
// on it (loop counters and TMEM addresses stay uniform over the warp).
__device__ __forceinline__ void wait_or_fail(uint32_t bar, unsigned parity, volatile int *failed, int *status,
                                             int where)
{
    if (try_wait(bar, parity, 0u)) return;
    const u64 t0 = global_ns();
    for (;;) {
        if (try_wait(bar, parity, 100000u) || *failed) return;
        if (global_ns() - t0 > kWaitLimitNs) {
            *failed = 1;
            report(status, kStatusTimeout, where);
            return;
        }
    }
}

__device__ __forceinline__ void arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void copy_in(uint32_t dst, const void *src, unsigned bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

// ---------------------------------------------------------------- the kernel
__global__ void __launch_bounds__(kTcThreads, 1) k_tc(const __grid_constant__ TcArgs a)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    const uint32_t sA = smem_u32(sm);                                    // [slots][digits, masses]
    unsigned char *bh = sm + kSlots * kSlotBytes, *bl = bh + kN * 32;   // B, upper and lower digits
    float *red = reinterpret_cast<float *>(bl + kN * 32);             // [warps][hi, lo][kSums]
    uint64_t *bars = reinterpret_cast<uint64_t *>(red + kTcWarps * 2 * kSums);
    const uint32_t bFull = smem_u32(bars), bDone = bFull + 8 * kSlots, bEmpty = bDone + 8 * kStages,
                   bFree = bEmpty + 8 * kStages;
    volatile int *seg = reinterpret_cast<volatile int *>(bars + 2 * kSlots + 2 * kStages);   // i tile, j tiles, last
    volatile int *failed = seg + 4;
    uint32_t *tptr = reinterpret_cast<uint32_t *>(bars + 2 * kSlots + 2 * kStages + 3);

    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const long long G = gridDim.x, b = blockIdx.x;
    const long long u0 = b * a.W / G, u1 = (b + 1) * a.W / G;
    if (*a.ok == 0) {
        if (a.jhl && !a.geo->hl)
#pragma unroll 4
            for (long long k = b * kTcThreads + tid; k < a.nj; k += G * kTcThreads) pack_hilo_one(a.jrec, k, a.jhl);
        return;
    }
    if (u0 >= u1) return;
    if (tid == 0) {
        *failed = 0;
        for (int k = 0; k < kSlots; ++k) {
            mbar_init(bars + k, 1);
            mbar_init(bars + kSlots + 2 * kStages + k, 1);
        }
        for (int k = 0; k < kStages; ++k) {
            mbar_init(bars + kSlots + k, 1);
            mbar_init(bars + kSlots + kStages + k, kTcWarps);
        }
        mbar_fence_init();
    }
    if (warp == kTcWarps) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tptr)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tm = __shfl_sync(0xffffffffu, *tptr, 0);
    constexpr uint32_t idesc = (1u << 4) | ((uint32_t)(kN / 8) << 17) | ((kTcJ / 16u) << 24);   // FP32 += FP16 x FP16
    const int njt = a.njt;

    if (warp >= kTcWarps) {
        // 4 x 32 x (2 x 224 + 56) = the 12 warps' 168 registers at launch
        asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
        const int role = warp - kTcWarps;  // 0: segments, 1: copies, 2 and 3: MMAs of even and odd tiles
        int sl = role == 3 ? 1 : 0;        // slot of the next tile
        int n = 0, q0 = sl;                // tiles so far (up to what the first waits need); issuers: next segment's first
        unsigned par = 0;                  // parity of the slot's use
        for (long long u = u0; u < u1;) {
            const int t = (int)(u / njt), s0 = (int)(u - (long long)t * njt);
            const int nt = (int)min(u1 - u, (long long)(njt - s0));
            if (role == 0 && lane == 0) {
                seg[0] = t;
                seg[1] = nt;
                seg[2] = u + nt >= u1;
            }
            __syncthreads();
            __syncthreads();
            if (role == 1 && lane == 0) {
                const unsigned char *gd = a.dig + (size_t)s0 * kDigBytes;
                const float *gm = a.mass + (size_t)s0 * kTcJ;
                for (int q = 0; q < nt; ++q) {
                    const uint32_t bar = bFull + 8 * sl, dst = sA + sl * kSlotBytes;
                    if (n >= kSlots) {
                        wait_or_fail(bFree + 8 * sl, par ^ 1u, failed, a.status, 20);
                        if (*failed) break;
                    }
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(kSlotBytes) : "memory");
                    copy_in(dst, gd + (size_t)q * kDigBytes, kDigBytes, bar);
                    copy_in(dst + kDigBytes, gm + (size_t)q * kTcJ, kTcJ * 4, bar);
                    if (n < kSlots) ++n;
                    if (++sl == kSlots) { sl = 0; par ^= 1u; }
                }
                // after a failure, copies in flight land before the CTA's shared memory goes
                if (*failed)
                    for (int k = 0; k < n; ++k) mbar_wait(bars + k, k < sl ? par : par ^ 1u, kWaitLimitNs / 4);
            }
            if (role >= 2 && lane == 0) {
                const u64 dh = operand(smem_u32(bh)), dl = operand(smem_u32(bl));
                int q = q0;
                for (; q < nt; q += 2) {
                    const int st = sl % kStages;
                    if (n >= kStages / 2) {
                        // the stage's previous tile is read, so the slot it came from is free
                        wait_or_fail(bEmpty + 8 * st, ((sl / kStages) & 1) ^ 1u, failed, a.status, 21);
                        if (*failed) break;
                        arrive(bFree + 8 * ((sl + kSlots - kStages) % kSlots));
                    }
                    wait_or_fail(bFull + 8 * sl, par, failed, a.status, 22);
                    if (*failed) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const u64 da = operand(sA + sl * kSlotBytes);
                    mma_f16(tm + st * kN, da, dh, idesc, 0);
                    mma_f16(tm + st * kN, da, dl, idesc, 1);
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bDone + 8 * st) : "memory");
                    if (n < kStages / 2) ++n;
                    sl += 2;
                    if (sl >= kSlots) { sl -= kSlots; par ^= 1u; }
                }
                q0 = q - nt;
                // after a failure, the MMAs issued last end before the CTA's memory goes
                if (*failed && n > 0) {
                    const int ls = (sl + kSlots - 2) % kSlots;
                    mbar_wait(bars + kSlots + ls % kStages, (ls / kStages) & 1, kWaitLimitNs / 4);
                }
            }
            __syncthreads();
            u += nt;
            if (__syncthreads_or(*failed || u >= u1)) break;
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
        // (% 2: with the range of grp known the addresses stay in uniform registers; 2 % of the run)
        const int quad = warp & 3, grp = (warp >> 2) % 2;
        const float e2s = a.geo->e2;
        const u64 e2 = pk2(e2s, e2s);
        unsigned pos = 0;                  // the next tile, counted over the CTA's tiles
        const uint32_t tb0 = tm + ((uint32_t)(quad * 32) << 16) + grp * 3 * kIW;
        const uint32_t ms0 = sA + kDigBytes + (quad * 32 + lane) * 4;
        float *mine = red + warp * 2 * kSums + lane * kLaneSums;
        for (;;) {
            __syncthreads();
            const int t = __shfl_sync(0xffffffffu, seg[0], 0), nt = __shfl_sync(0xffffffffu, seg[1], 0);
            // B: row (group, axis, i); digits as FP16 pairs {upper 0, 1}, {lower 0, 1}
            for (int r = tid; r < kN; r += kTcWarps * 32) {
                const int g = r / (3 * kIW), axis = (r % (3 * kIW)) / kIW, ii = r % kIW;
                const long long i = (long long)t * kBi + g * kIW + ii;
                uint2 d = make_uint2(0u, 0u);
                if (i < a.ni)
                    d = *reinterpret_cast<const uint2 *>(a.idig + (i / 8) * 256 + (axis >> 1) * 128 + (i % 8) * 16 + (axis & 1) * 8);
                d.x ^= 0x80008000u;                                      // -x_i
                d.y ^= 0x80008000u;
                const unsigned wh = 0x3C006C00u, wl = 0x08000C00u;       // {4096, 1}, {2^-12, 2^-13}
                const size_t at = (r / 8) * 256 + (r % 8) * 16;
                *reinterpret_cast<uint4 *>(bh + at) = make_uint4(axis == 0 ? wh : 0, 0, axis == 1 ? wh : 0, 0);
                *reinterpret_cast<uint4 *>(bh + at + 128) = make_uint4(axis == 2 ? wh : 0, 0, d.x, 0);
                *reinterpret_cast<uint4 *>(bl + at) = make_uint4(0, axis == 0 ? wl : 0, 0, axis == 1 ? wl : 0);
                *reinterpret_cast<uint4 *>(bl + at + 128) = make_uint4(0, axis == 2 ? wl : 0, 0, d.y);
            }
#pragma unroll
            for (int k = 0; k < kLaneSums; ++k) mine[k] = mine[kSums + k] = 0.0f;
            fence_proxy_async();
            __syncthreads();

            int rem = nt;
            u64 ax[kIW / 2], ay[kIW / 2], az[kIW / 2], ph[kIW / 2];
            while (rem > 0) {
#pragma unroll
                for (int k = 0; k < kIW / 2; ++k) ax[k] = ay[k] = az[k] = ph[k] = 0ull;
                int c = min(rem, kFoldTiles);
                rem -= c;
#pragma unroll 1
                for (; c; --c) {
                    const unsigned st = pos % kStages;
                    wait_or_fail(bDone + 8 * st, (pos / kStages) & 1u, failed, a.status, 23);
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    float m;
                    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(m) : "r"(ms0 + (pos % kSlots) * kSlotBytes));
                    const u64 m2 = pk2(m, m);
                    const uint32_t tb = tb0 + st * kN;
                    ++pos;
                    float xb[2][4], yb[2][4], zb[2][4];
                    tmem_ld4(tb, xb[0]);
                    tmem_ld4(tb + kIW, yb[0]);
                    tmem_ld4(tb + 2 * kIW, zb[0]);
#pragma unroll
                    for (int h = 0; h < kIW / 4; ++h) {
                        float (&x)[4] = xb[h & 1], (&y)[4] = yb[h & 1], (&z)[4] = zb[h & 1];
                        tmem_wait(x, y, z);
                        if (h < kIW / 4 - 1) {
                            tmem_ld4(tb + 4 * h + 4, xb[(h + 1) & 1]);
                            tmem_ld4(tb + kIW + 4 * h + 4, yb[(h + 1) & 1]);
                            tmem_ld4(tb + 2 * kIW + 4 * h + 4, zb[(h + 1) & 1]);
                        } else {           // all read: the stage and the masses may be overwritten
                            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                            __syncwarp();
                            if (lane == 0) arrive(bEmpty + 8 * st);
                        }
#pragma unroll
                        for (int k = 0; k < 2; ++k) {
                            const int p = 2 * h + k;
                            const u64 dx = pk2(x[2 * k], x[2 * k + 1]), dy = pk2(y[2 * k], y[2 * k + 1]),
                                      dz = pk2(z[2 * k], z[2 * k + 1]);
                            u64 r2 = f2fma(dx, dx, e2);
                            r2 = f2fma(dy, dy, r2);
                            r2 = f2fma(dz, dz, r2);
                            float ra, rb;
                            up2(r2, ra, rb);
                            const u64 q = pk2(rsq(ra), rsq(rb));
                            const u64 mq = f2mul(m2, q);
                            const u64 mq3 = f2mul(mq, f2mul(q, q));
                            ph[p] = f2sub(ph[p], mq);
                            ax[p] = f2fma(mq3, dx, ax[p]);
                            ay[p] = f2fma(mq3, dy, ay[p]);
                            az[p] = f2fma(mq3, dz, az[p]);
                        }
                    }
                }
                // the lanes' sums: lane l ends with values kLaneSums l ... of (component, i)
                float v[kSums];
#pragma unroll
                for (int k = 0; k < kIW / 2; ++k) {
                    up2(ax[k], v[2 * k], v[2 * k + 1]);
                    up2(ay[k], v[kIW + 2 * k], v[kIW + 2 * k + 1]);
                    up2(az[k], v[2 * kIW + 2 * k], v[2 * kIW + 2 * k + 1]);
                    up2(ph[k], v[3 * kIW + 2 * k], v[3 * kIW + 2 * k + 1]);
                }
#pragma unroll
                for (int o = 16; o; o >>= 1) {
                    const bool up = lane & o;
#pragma unroll
                    for (int k = 0; k < kLaneSums * o; ++k) {
                        const float x = v[k], y = v[k + kLaneSums * o];
                        v[k] = __fadd_rn(up ? y : x, __shfl_xor_sync(0xffffffffu, up ? x : y, o));
                    }
                }
#pragma unroll
                for (int k = 0; k < kLaneSums; ++k) {
                    float s, e;
                    two_sum(mine[k], v[k], s, e);
                    mine[k] = s;
                    mine[kSums + k] = __fadd_rn(mine[kSums + k], e);
                }
            }
            __syncthreads();
            {
                // the segment's sums over quadrants, in order
                const long long slot = b - tc_owner((long long)t * njt, G, a.W);
                double *dst = reinterpret_cast<double *>(a.part + ((size_t)t * a.slots + slot) * kBi);
                for (int e = tid; e < 4 * kBi; e += kTcWarps * 32) {
                    const int i = e / 4, comp = e % 4, g = i / kIW, ii = i % kIW;
                    double s = 0.0;
                    for (int w = 4 * g; w < 4 * g + 4; ++w)
                        s += (double)red[w * 2 * kSums + comp * kIW + ii] + (double)red[w * 2 * kSums + kSums + comp * kIW + ii];
                    dst[e] = s;
                }
            }
            if (__syncthreads_or(*failed || seg[2])) break;
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == kTcWarps) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tm));
    }
}

// ---------------------------------------------------------------- digits
// a coordinate's four digits as FP16, lower digit 1 scaled by 2^-11 (its
// place value 2^-24 is below FP16's normal range)
// (x scale is exact, a power of two, so y is (x - c) scale, rounded once, with
// cs = c scale; adding 1.5 2^52 rounds it to an integer, the low bits of the
// sum. The packing of 2^20 records takes 21 us; a subtraction, a product and
// a conversion to 64-bit integers a coordinate took 25.)
__device__ __forceinline__ void digits(double x, double cs, double scale, __half *h)
{
    const double y = fma(x, scale, -cs);
    const long long X = __double_as_longlong(y + 0x1.8p52) - __double_as_longlong(0x1.8p52);
    const long long hi = (X + (1ll << 23)) >> 24, lo = X - (hi << 24);
    const int h0 = (int)((hi + 2048) >> 12), h1 = (int)(hi - ((long long)h0 << 12));
    const int l0 = (int)((lo + 2048) >> 12), l1 = (int)(lo - ((long long)l0 << 12));
    h[0] = __int2half_rn(h0);
    h[1] = __int2half_rn(h1);
    h[2] = __int2half_rn(l0);
    h[3] = __float2half_rn((float)l1 * (1.0f / 2048.0f));
}

__device__ __forceinline__ void write_digits(const double4 v, const TcGeo &g, unsigned char *dig, long long k)
{
    __align__(16) __half h[16];
    digits(v.x, g.sx, g.scale, h);
    digits(v.y, g.sy, g.scale, h + 4);
    digits(v.z, g.sz, g.scale, h + 8);
    h[12] = __float2half_rn(4096.0f);
    h[13] = __float2half_rn(1.0f);
    h[14] = __float2half_rn(1.0f / 4096.0f);
    h[15] = __float2half_rn(1.0f / 8192.0f);
    unsigned char *d = dig + (k / 8) * 256 + (k % 8) * 16;
    *reinterpret_cast<uint4 *>(d) = *reinterpret_cast<uint4 *>(h);
    *reinterpret_cast<uint4 *>(d + 128) = *reinterpret_cast<uint4 *>(h + 8);
}

__device__ __forceinline__ u64 ord64(double v)
{
    const u64 b = (u64)__double_as_longlong(v);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
// (on the integer pipe: a comparison in FP64 takes a warp 16 clocks of the SM)
__device__ __forceinline__ bool finite64(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }
__device__ __forceinline__ double unord64(u64 u)
{
    return __longlong_as_double((long long)((u >> 63) ? (u & 0x7fffffffffffffffull) : ~u));
}

// The j-set's cube, largest and smallest nonzero mass; the last block to
// finish sets the geometry and clears the words for the next call. words: 3
// minima (stored inverted, so that zero starts them all), 3 maxima, largest
// |m| (as bits, all ones with a non-finite value), smallest nonzero |m|
// (inverted bits), ticket. seen (may be null): the host's copy. PACK: from
// the caller's arrays, with the records written as k_pack_j writes them.
// Bound: the latency of the records; kBoxRec of them in flight a thread, at
// most kBoxBlocks blocks at the words. 2^20 from the caller's arrays: 18 us,
// k_pack_j alone 11 (tests of isfinite, comparisons in FP64, made it 33).
constexpr int kBoxRec = 2;
constexpr long long kBoxBlocks = 608;
template <bool PACK>
__global__ void __launch_bounds__(256) k_tc_box(const double *__restrict__ x, const double *__restrict__ m,
                                                double4 *__restrict__ jrec, long long nj, u64 *words, TcGeo *geo,
                                                TcSeen *seen, long long gen)
{
    __shared__ u64 sh[8][8];
    u64 v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    const long long stride = gridDim.x * 256ll;
    for (long long k0 = blockIdx.x * 256ll + threadIdx.x; k0 < nj; k0 += kBoxRec * stride) {
        double4 rec[kBoxRec];
#pragma unroll
        for (int q = 0; q < kBoxRec; ++q) {
            const long long k = k0 + q * stride;
            if (k < nj) rec[q] = PACK ? make_double4(x[3 * k], x[3 * k + 1], x[3 * k + 2], m[k]) : jrec[k];
        }
#pragma unroll
        for (int q = 0; q < kBoxRec; ++q) {
            const long long k = k0 + q * stride;
            if (k >= nj) break;
            const double4 r = rec[q];
            if (PACK) jrec[k] = r;
            const u64 o[3] = {ord64(r.x), ord64(r.y), ord64(r.z)};
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                v[d] = max(v[d], ~o[d]);
                v[3 + d] = max(v[3 + d], o[d]);
            }
            const u64 mb = (u64)__double_as_longlong(r.w) & ~(1ull << 63);
            v[6] = max(v[6], finite64(r.x) && finite64(r.y) && finite64(r.z) && finite64(r.w) ? mb : ~0ull);
            v[7] = max(v[7], mb ? ~mb : 0ull);
        }
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        for (int o = 16; o; o >>= 1) v[q] = max(v[q], __shfl_xor_sync(0xffffffffu, v[q], o));
        if (lane == 0) sh[q][w] = v[q];
    }
    __syncthreads();
    if (threadIdx.x < 8) {
        u64 m = 0;
        for (int q = 0; q < 8; ++q) m = max(m, sh[threadIdx.x][q]);
        if (m > __ldcg(words + threadIdx.x)) atomicMax(words + threadIdx.x, m);
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x != 0 || atomicAdd(words + 8, 1ull) != gridDim.x - 1) return;
    __threadfence();
    double lo[3], hi[3];
    for (int d = 0; d < 3; ++d) {
        lo[d] = unord64(~__ldcg(words + d));
        hi[d] = unord64(__ldcg(words + 3 + d));
    }
    const u64 mb = __ldcg(words + 6), ms = __ldcg(words + 7);
    TcGeo g{};
    g.ok = 0;
    if (mb != ~0ull) {
        g.cx = 0.5 * lo[0] + 0.5 * hi[0];
        g.cy = 0.5 * lo[1] + 0.5 * hi[1];
        g.cz = 0.5 * lo[2] + 0.5 * hi[2];
        const double half = fmax(fmax(hi[0] - lo[0], hi[1] - lo[1]), hi[2] - lo[2]) * 0.5;
        // R = 2^e >= 5/4 half: i-particles a little outside still fit
        int e = half > 0.0 ? ilogb(1.25 * half) + 1 : 0;
        g.e = e;
        g.scale = ldexp(1.0, 47 - e);
        g.sx = g.cx * g.scale;
        g.sy = g.cy * g.scale;
        g.sz = g.cz * g.scale;
        const int em = mb ? ilogb(__longlong_as_double((long long)mb)) : 0;
        g.mscale = ldexp(1.0, 20 - em);        // masses enter at most 2^21
        g.mexp = 20 - em;
        g.mmin = ms ? __longlong_as_double((long long)~ms) * g.mscale : 0.0;
        g.ok = half < 1e300 && e > -900 && e < 900 && em > -900 && em < 900 &&
               fabs(g.sx) < 1e300 && fabs(g.sy) < 1e300 && fabs(g.sz) < 1e300;
    }
    *geo = g;
    for (int q = 0; q < kTcBoxWords; ++q) words[q] = 0;
    if (seen) {
        seen->mmin = g.mmin;
        seen->e = g.e;
        seen->ok = g.ok;
        __threadfence_system();
        *(volatile long long *)&seen->gen = gen;
    }
}

// the j records' digits and scaled masses, padded with massless records
__global__ void __launch_bounds__(256) k_tc_pack(const double4 *__restrict__ jrec, long long nj, long long npad,
                                                 float eps2, const TcGeo *__restrict__ geo,
                                                 unsigned char *__restrict__ dig, float *__restrict__ mass)
{
    __shared__ int go;
    const TcGeo g = *geo;
    if (threadIdx.x == 0) go = !g.packed && tc_fits(g.ok, g.e, g.mmin, eps2);
    __syncthreads();
    if (!go) return;
    for (long long k = blockIdx.x * 256ll + threadIdx.x; k < npad; k += gridDim.x * 256ll) {
        double4 v = make_double4(g.cx, g.cy, g.cz, 0.0);
        if (k < nj) v = jrec[k];
        write_digits(v, g, dig, k);
        mass[k] = (float)(v.w * g.mscale);
    }
}

// The i-particles' digits, and whether this call can use them: the j-set and
// eps fit and every i lies within the cube. The last block writes the verdict.
// The first tb blocks; those behind them prepare the narrow path.
constexpr int kPrepThreads = kTcJ;
static_assert(kPrepThreads == kNarrowPrepThreads, "one launch");
__global__ void __launch_bounds__(kPrepThreads) k_tc_prep(const double4 *__restrict__ xi, long long ni, int tb,
                                                          float eps2, TcGeo *geo, unsigned char *__restrict__ idig,
                                                          unsigned *words, int *ok, NarrowPrep np)
{
    if (blockIdx.x >= tb) {
        narrow_prep_block(xi, ni, np, blockIdx.x - tb);
        return;
    }
    const long long k = blockIdx.x * (long long)kPrepThreads + threadIdx.x;    // of whole tiles of kTcJ
    const TcGeo g = *geo;
    bool bad = false;
    double4 v = make_double4(g.cx, g.cy, g.cz, 0.0);
    if (k < ni && g.ok) {
        const double4 r = xi[k];
        const double lim = ldexp(1.0, g.e) * (1.0 - 0x1p-20);
        bad = !(fabs(r.x - g.cx) < lim && fabs(r.y - g.cy) < lim && fabs(r.z - g.cz) < lim);
        if (!bad) v = r;
    }
    write_digits(v, g, idig, k);
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(words, 1u);
    if (threadIdx.x != 0) return;
    __threadfence();
    if (atomicAdd(words + 1, 1u) != tb - 1) return;
    __threadfence();
    const bool far = __ldcg(words) != 0, fits = tc_fits(g.ok, g.e, g.mmin, eps2);
    // eps in units of the upper digits' last place, u = R 2^-23
    geo->e2 = (float)(ldexp((double)eps2, 2 * (23 - g.e)) * ((1.0 - kTcShort) * (1.0 - kTcShort)));
    geo->packed = g.packed || fits;
    geo->hl = g.stood_in;
    geo->stood_in = g.stood_in || far || !fits;
    *ok = fits && !far;
    words[0] = words[1] = 0;
}

__global__ void __launch_bounds__(256) k_tc_combine(TcArgs a, int grid, int self, long long self_off,
                                                    double *__restrict__ acc, double *__restrict__ pot)
{
    if (*a.ok == 0) return;
    const long long i = blockIdx.x * 8ll + (threadIdx.x >> 5);
    if (i < a.ni) tc_combine_one(a, grid, self, self_off, acc, pot, i);
}

}  // namespace

size_t tc_dig_bytes(long long n) { return (size_t)((n + kTcJ - 1) / kTcJ) * kDigBytes; }
int tc_jtiles(long long nj) { return (int)((nj + kTcJ - 1) / kTcJ); }
int tc_slots(long long ntiles, int njt, long long W, int grid)
{
    int s = 1;
    for (long long t = 0; t < ntiles; ++t)
        s = std::max<int>(s, (int)(tc_owner((t + 1) * njt - 1, grid, W) - tc_owner(t * njt, grid, W) + 1));
    return s;
}

static unsigned box_blocks(long long nj)
{
    return (unsigned)std::min<long long>((nj + 256 * kBoxRec - 1) / (256 * kBoxRec), kBoxBlocks);
}

cudaError_t launch_tc_box(const double4 *jrec, long long nj, unsigned long long *words, TcGeo *geo, TcSeen *seen,
                          long long gen, cudaStream_t st)
{
    if (nj <= 0) return cudaErrorInvalidValue;
    k_tc_box<false><<<box_blocks(nj), 256, 0, st>>>(nullptr, nullptr, const_cast<double4 *>(jrec), nj, words, geo, seen,
                                                    gen);
    return cudaGetLastError();
}

cudaError_t launch_tc_pack_box(const double *x, const double *m, double4 *jrec, long long nj, unsigned long long *words,
                               TcGeo *geo, TcSeen *seen, long long gen, cudaStream_t st)
{
    if (nj <= 0) return cudaErrorInvalidValue;
    k_tc_box<true><<<box_blocks(nj), 256, 0, st>>>(x, m, jrec, nj, words, geo, seen, gen);
    return cudaGetLastError();
}

cudaError_t launch_tc_pack(const double4 *jrec, long long nj, float eps2, const TcGeo *geo, unsigned char *dig,
                           float *mass, cudaStream_t st)
{
    if (nj <= 0) return cudaErrorInvalidValue;
    const long long npad = (long long)tc_jtiles(nj) * kTcJ;
    k_tc_pack<<<(unsigned)std::min<long long>((npad + 255) / 256, 1216), 256, 0, st>>>(jrec, nj, npad, eps2, geo, dig,
                                                                                        mass);
    return cudaGetLastError();
}

cudaError_t launch_tc_prep(const double4 *xi, long long ni, float eps2, TcGeo *geo, unsigned char *idig,
                           unsigned *words, int *ok, const NarrowPrep &np, cudaStream_t st)
{
    if (ni <= 0) return cudaErrorInvalidValue;
    const int tb = tc_jtiles(ni);
    const long long nb = tb + (np.nic > 0 ? narrow_prep_blocks(ni, np) : 0);
    k_tc_prep<<<(unsigned)nb, kPrepThreads, 0, st>>>(xi, ni, tb, eps2, geo, idig, words, ok, np);
    return cudaGetLastError();
}

cudaError_t launch_tc(const TcArgs &a, int grid, cudaStream_t st)
{
    if (grid <= 0 || a.W <= 0) return cudaErrorInvalidValue;
    static bool done[kMaxDevices] = {};
    const cudaError_t e = once_per_device(done, [] {
        return cudaFuncSetAttribute(k_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTcSmem);
    });
    if (e != cudaSuccess) return e;
    k_tc<<<grid, kTcThreads, kTcSmem, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_tc_combine(const TcArgs &a, int grid, int self, long long self_off, double *acc, double *pot,
                              cudaStream_t st)
{
    k_tc_combine<<<(unsigned)((a.ni + 7) / 8), 256, 0, st>>>(a, grid, self, self_off, acc, pot);
    return cudaGetLastError();
}

}  // namespace pg
