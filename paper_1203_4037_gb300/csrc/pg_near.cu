// pg_near.cu -- the tabulated force on compact i-tiles, near pairs only.
//
// The table's g is exactly 0 at and beyond r_cut (so is its potential), and
// an i-tile that is one run of the Morton order needs only the j-particles
// within r_cut of its box. All pairs beyond that add exact zeros, which is
// what the all-pairs kernels spend nearly all their time on when r_cut is
// small against the system.
//
// A CTA streams the j records in FP32 (16 bytes each, kNearJ per unit, bulk
// copies in two buffers), keeps those near its tile's box in a list, and
// whenever the list holds kTJ converts that many from their FP64 records
// (the all-pairs kernels' conversion) and evaluates them: each warp first
// leaves out the records beyond r_cut of its own run of i-particles, then
// runs the all-pairs pair term on the rest. Converting from a list keeps the
// FP64 work on full warps (GB300 issues FP64 at about two lanes per SM-clock
// whatever lanes are active).
//
// Bound: the tests, about 12 instructions per (i-tile, j), and the latency
// of a unit (copy, two barriers, list) and of a batch (gather, conversion,
// barrier); the pair terms are a few per cent of n^2. Measured (kernels, one
// Plummer sphere of 65536, r_cut = 0.1 scale lengths, against the all-pairs
// kernels): forward 2.72 -> 0.36 ms, backward 5.96 -> 0.67 ms; how well the
// sampled costs split the units depends on the set (262144, six spheres:
// forward 2.0 to 3.7 ms, all pairs 43 ms). With equal unit counts instead of
// the split by cost the forward kernel took 0.56 ms (an earlier form),
// converting records in place instead of from a list about 8000 clocks per
// 256 j.
#include <type_traits>

#include "pg_device.cuh"

namespace pg {

namespace {

constexpr int kList = kTJ + kNearJ;            // kept records waiting, at most kTJ - 1 from before a unit
constexpr int kPadIdx = 4;                     // a warp's record numbers are padded to this
constexpr int kIdx = kTJ + kPadIdx;
constexpr int kTests = kNearJ / kNT;           // records a thread tests per unit
static_assert(kNearJ % kNT == 0 && kIdx % 4 == 0, "whole rounds and whole words");

// A tile's box as the test uses it, in units of the table's s (lengths times
// sc; the cutoff is R = sqrt(s_max - 2)): FP32 squares in the caller's unit
// would leave the range for an r_cut below 1e-19 or above 1e19. Positions are
// taken from tile 0's centre o: FP32 has no room for a cutoff 1e7 times
// smaller than the distance to the caller's origin. Its centre in
// FP32 and half extents grown past every rounding of the test: for a j in
// range, |x_j| <= |c| + h + R, so its FP32 coordinate, the FP32 centre and
// half extent, their difference and the growth are together within 6 2^-24 of
// that sum per axis; R^2 is grown by 1e-5, past the roundings of the squares.
struct TileBox {
    float cx, cy, cz, hx, hy, hz, lim;
};

__device__ __forceinline__ TileBox tile_box(const double4 c, const double4 h, const double4 o, double sc, float R)
{
    constexpr float u = 3.6e-7f;   // just above 6 2^-24
    TileBox b;
    b.cx = (float)((c.x - o.x) * sc);
    b.cy = (float)((c.y - o.y) * sc);
    b.cz = (float)((c.z - o.z) * sc);
    const float hx = (float)(h.x * sc), hy = (float)(h.y * sc), hz = (float)(h.z * sc);
    b.hx = hx + u * (fabsf(b.cx) + hx + R);
    b.hy = hy + u * (fabsf(b.cy) + hy + R);
    b.hz = hz + u * (fabsf(b.cz) + hz + R);
    b.lim = R * R * (1.0f + 1e-5f);
    return b;
}

// whether a record with squared distance d2 to a box is kept; one with a
// non-finite value always is, as it makes its pairs non-finite at any distance
__device__ __forceinline__ bool keep_it(float d2, float lim, const float4 j)
{
    const bool fin = fabsf(j.x) + fabsf(j.y) + fabsf(j.z) + fabsf(j.w) < 3.0e38f;   // false for NaN
    return !(d2 > lim && fin);
}

__device__ __forceinline__ bool tile_keep(const TileBox &b, const float4 j)
{
    const float dx = fmaxf(fabsf(j.x - b.cx) - b.hx, 0.0f);
    const float dy = fmaxf(fabsf(j.y - b.cy) - b.hy, 0.0f);
    const float dz = fmaxf(fabsf(j.z - b.cz) - b.hz, 0.0f);
    return keep_it(dx * dx + dy * dy + dz * dz, b.lim, j);
}

// The same against one warp's own i-particles, on the converted scaled
// offsets: a tile in a sparse halo spans a box that can hold the whole core,
// its warps' runs of the order are smaller. R: the cutoff in scaled units.
struct WarpBox {
    float lx, ly, lz, hx, hy, hz, lim;

    __device__ __forceinline__ void clear()
    {
        lx = ly = lz = __int_as_float(0x7f800000);
        hx = hy = hz = -__int_as_float(0x7f800000);
    }
    __device__ __forceinline__ void add(float x, float y, float z)
    {
        lx = fminf(lx, x); hx = fmaxf(hx, x);
        ly = fminf(ly, y); hy = fmaxf(hy, y);
        lz = fminf(lz, z); hz = fmaxf(hz, z);
    }
    // over the warp; `all`: keep everything (a non-finite i-particle)
    __device__ __forceinline__ void close(float R, bool all)
    {
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            lx = fminf(lx, __shfl_xor_sync(0xffffffffu, lx, o));
            ly = fminf(ly, __shfl_xor_sync(0xffffffffu, ly, o));
            lz = fminf(lz, __shfl_xor_sync(0xffffffffu, lz, o));
            hx = fmaxf(hx, __shfl_xor_sync(0xffffffffu, hx, o));
            hy = fmaxf(hy, __shfl_xor_sync(0xffffffffu, hy, o));
            hz = fmaxf(hz, __shfl_xor_sync(0xffffffffu, hz, o));
        }
        constexpr float u = 2.4e-7f;           // both offsets' roundings and the difference's
        const float gx = u * (fabsf(lx) + fabsf(hx) + R), gy = u * (fabsf(ly) + fabsf(hy) + R),
                    gz = u * (fabsf(lz) + fabsf(hz) + R);
        lx -= gx; ly -= gy; lz -= gz;
        hx += gx; hy += gy; hz += gz;
        lim = all ? __int_as_float(0x7f800000) : R * R * (1.0f + 1e-5f);
    }
    __device__ __forceinline__ bool keep(const float4 j) const
    {
        const float dx = fmaxf(fmaxf(lx - j.x, j.x - hx), 0.0f);
        const float dy = fmaxf(fmaxf(ly - j.y, j.y - hy), 0.0f);
        const float dz = fmaxf(fmaxf(lz - j.z, j.z - hz), 0.0f);
        return keep_it(dx * dx + dy * dy + dz * dz, lim, j);
    }
};

// The numbers of the n staged records (x, y, z, m given by at(e)) that this
// warp keeps (`all`: every one), in order, in idx; padded to whole groups of
// kPadIdx with `pad`. Returns the padded count.
template <typename At>
__device__ __forceinline__ int warp_list(const WarpBox &b, bool all, int n, unsigned short *idx, int pad, At at)
{
    const int lane = threadIdx.x & 31;
    int k = 0;
    for (int e0 = 0; e0 < n; e0 += 32) {
        const int e = e0 + lane;
        const bool kp = e < n && (all || b.keep(at(e)));
        const unsigned m = __ballot_sync(0xffffffffu, kp);
        if (kp) idx[k + __popc(m & ((1u << lane) - 1u))] = (unsigned short)e;
        k += __popc(m);
    }
    const int kp = (k + kPadIdx - 1) / kPadIdx * kPadIdx;
    if (lane < kp - k) idx[k + lane] = (unsigned short)pad;
    __syncwarp();
    return kp;
}

// the shared memory both kernels use beside their own
struct NearShared {
    float4 *raw;               // [2][kNearJ]
    int *list;                 // [kList] kept records' indices
    int *cnt;                  // [kNearJ / 32]
    unsigned short *idx;       // this warp's [kIdx]
    uint64_t *bar;             // [2]
    int *flag;
};
constexpr size_t kNearShared = 2 * kNearJ * sizeof(float4) + kList * sizeof(int) + kNearJ / 32 * sizeof(int) +
                               (kNT / 32) * kIdx * sizeof(unsigned short) + 4 * sizeof(uint64_t);
static_assert(kNearShared % 16 == 0, "what follows stays aligned");

__device__ __forceinline__ NearShared near_shared(unsigned char *p)
{
    NearShared s;
    s.raw = reinterpret_cast<float4 *>(p);
    s.bar = reinterpret_cast<uint64_t *>(s.raw + 2 * kNearJ);
    s.flag = reinterpret_cast<int *>(s.bar + 2);
    s.list = reinterpret_cast<int *>(s.bar + 4);
    s.cnt = s.list + kList;
    s.idx = reinterpret_cast<unsigned short *>(s.cnt + kNearJ / 32) + (threadIdx.x >> 5) * kIdx;
    return s;
}

// The stream of one CTA: begin(t) and end(t) around each tile's units,
// eval(list, n) on n <= kTJ kept records. Returns false if a wait ran out.
// eval may end without a barrier; the next use of its staging comes after one.
template <typename Begin, typename Eval, typename End>
__device__ __forceinline__ bool near_stream(const NearArgs &a, const NearShared &sm, Begin begin, Eval eval, End end)
{
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const long long b = blockIdx.x, u0 = a.start[b], u1 = a.start[b + 1];
    if (u0 >= u1 || !*a.near) return true;
    auto sub = [&](long long u) { return (long long)(u % a.nch) * a.sstride % a.nch; };
    auto issue = [&](long long u, int buf) {
        const long long j0 = sub(u) * a.unit;
        const unsigned bytes = (unsigned)(min(a.nj - j0, (long long)a.unit) * sizeof(float4));
        mbar_arrive_tx(&sm.bar[buf], bytes);
        bulk_g2s(sm.raw + buf * kNearJ, a.jf + j0, bytes, &sm.bar[buf]);
    };
    if (tid == 0) {
        mbar_init(&sm.bar[0], 1);
        mbar_init(&sm.bar[1], 1);
        mbar_fence_init();
    }
    __syncthreads();
    unsigned pending = 0, phase = 0;
    if (tid == 0) {
        issue(u0, 0);
        pending = 1u;
        if (u0 + 1 < u1) {
            issue(u0 + 1, 1);
            pending |= 2u;
        }
    }
    TileBox box = {};
    long long cur = -1;
    int held = 0;
    for (long long u = u0; u < u1; ++u) {
        const long long t = u / a.nch;
        const int buf = (int)((u - u0) & 1);
        if (t != cur) {
            if (cur >= 0) {
                if (held) eval(sm.list, held);
                end(cur);
            }
            cur = t;
            held = 0;
            box = tile_box(a.ctr[t], a.ext[t], a.ctr[0], a.tab.scale, sqrtf(a.tab.s_max - 2.0f));
            begin(t);
        }
        if (tid == 0) {
            const bool ok = mbar_wait(&sm.bar[buf], (phase >> buf) & 1u, kWaitLimitNs);
            if (ok) pending &= ~(1u << buf);
            *sm.flag = ok ? 1 : 0;
        }
        __syncthreads();               // the records are here; the list's last readers are done
        if (*sm.flag == 0) {
            // let copies still in flight land before the CTA's shared memory goes
            if (tid == 0) {
                report(a.status, kStatusTimeout, 5);
                for (int k = 0; k < 2; ++k)
                    if (pending & (1u << k)) mbar_wait(&sm.bar[k], (phase >> k) & 1u, kWaitLimitNs / 4);
            }
            return false;
        }
        phase ^= 1u << buf;
        const long long j0 = sub(u) * a.unit;
        const int nu = (int)min(a.nj - j0, (long long)a.unit);
        unsigned m[kTests];
#pragma unroll
        for (int r = 0; r < kTests; ++r) {
            const int e = r * kNT + tid;
            const bool k = e < nu && tile_keep(box, sm.raw[buf * kNearJ + e]);
            m[r] = __ballot_sync(0xffffffffu, k);
            if (lane == 0) sm.cnt[r * (kNT / 32) + w] = __popc(m[r]);
        }
        __syncthreads();
        if (tid == 0 && u + 2 < u1) {  // the buffer is read: refill it
            fence_proxy_async();
            issue(u + 2, buf);
            pending |= 1u << buf;
        }
        // where this warp's kept records go: a scan of the 32 counts
        static_assert(kNearJ / 32 == 32, "one count per lane");
        int c = sm.cnt[lane], x = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        const int total = __shfl_sync(0xffffffffu, x, 31);
#pragma unroll
        for (int r = 0; r < kTests; ++r) {
            const int at = held + __shfl_sync(0xffffffffu, x - c, r * (kNT / 32) + w);
            if (m[r] >> lane & 1u) sm.list[at + __popc(m[r] & ((1u << lane) - 1u))] = (int)(j0 + r * kNT + tid);
        }
        held += total;
        if (held < kTJ) continue;
        __syncthreads();               // the list is written
        while (held >= kTJ) {
            held -= kTJ;
            eval(sm.list + held, kTJ);
        }
    }
    __syncthreads();
    if (held) eval(sm.list, held);
    end(cur);
    return true;
}

// ---------------------------------------------------------------- forward

template <bool DF> struct NearWords { static constexpr int value = DF ? 8 : 4; };

// CTAs per SM the register budget is sized for
template <int NP> struct NearBlocks { static constexpr int value = NP == 1 ? 6 : NP == 2 ? 4 : 2; };

template <int NP, bool EXT, bool DF>
__global__ void __launch_bounds__(kNT, NearBlocks<NP>::value) k_near(NearArgs a)
{
    constexpr int Bi = kNT * 2 * NP, kW = NearWords<DF>::value, kComp = EXT ? 4 : 3;
    extern __shared__ __align__(128) unsigned char smem[];
    const NearShared sm = near_shared(smem);
    u64 *cvt = reinterpret_cast<u64 *>(smem + kNearShared);                 // [kTJ + 1][kW], the last a pad
    u64 *run = cvt + (kTJ + 1) * kW;                                        // [2 kComp NP][kNT]
    float2 *tab = reinterpret_cast<float2 *>(run + 2 * kComp * NP * kNT);
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    if (EXT)
        for (int k = tid; k < a.tab.n; k += kNT) reinterpret_cast<float4 *>(tab)[k] = a.tab.AGP[k];
    else
        for (int k = tid; k < a.tab.n; k += kNT) tab[k] = a.tab.AG1[k];

    // per-thread state, as in the all-pairs kernel; each warp's i are one run of the order
    u64 xi[NP], yi[NP], zi[NP], exi[DF ? NP : 1], eyi[DF ? NP : 1], ezi[DF ? NP : 1];
    u64 ax[NP], ay[NP], az[NP], ph[NP];
    auto RH = [&](int p, int k) -> u64 & { return run[(2 * kComp * p + k) * kNT + tid]; };
    auto RL = [&](int p, int k) -> u64 & { return run[(2 * kComp * p + kComp + k) * kNT + tid]; };
    auto LI = [&](int p, int q) { return (w * 2 * NP + 2 * p + q) * 32 + lane; };
    double cx = 0, cy = 0, cz = 0;
    const double sc = a.tab.scale;
    const float R = sqrtf(a.tab.s_max - 2.0f);
    const u64 c0v = pk2(2.0f, 2.0f);
    const unsigned smax_bits = __float_as_uint(a.tab.s_max);
    const int sh3 = a.tab.shift - (EXT ? 4 : 3);
    const unsigned tb0 = smem_u32(tab) - (a.tab.base << (EXT ? 4 : 3));
    WarpBox wb;
    bool dense = false;

    auto begin = [&](long long t) {
        const double4 c = a.ctr[t];
        cx = c.x; cy = c.y; cz = c.z;
        dense = a.dense[t] != 0;
        wb.clear();
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            float f[3][2], e[3][2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const long long i = t * Bi + LI(p, q);
#pragma unroll
                for (int k = 0; k < 3; ++k) f[k][q] = e[k][q] = 0.0f;
                if (i >= a.ni) continue;
                const double4 v = a.xi[i];
                const double o[3] = {(v.x - cx) * sc, (v.y - cy) * sc, (v.z - cz) * sc};
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    f[k][q] = (float)o[k];
                    e[k][q] = (float)(o[k] - (double)f[k][q]);
                }
                wb.add(f[0][q], f[1][q], f[2][q]);
            }
            xi[p] = pk2(f[0][0], f[0][1]); yi[p] = pk2(f[1][0], f[1][1]); zi[p] = pk2(f[2][0], f[2][1]);
            if (DF) {
                exi[p] = pk2(e[0][0], e[0][1]); eyi[p] = pk2(e[1][0], e[1][1]); ezi[p] = pk2(e[2][0], e[2][1]);
            }
#pragma unroll
            for (int k = 0; k < kComp; ++k) RH(p, k) = RL(p, k) = 0ull;
        }
        wb.close(R, isinf(a.ext[t].x));
    };

    auto pair = [&](int e) {
        const ulonglong2 xy = reinterpret_cast<const ulonglong2 *>(cvt)[(kW / 2) * e];
        const ulonglong2 zm = reinterpret_cast<const ulonglong2 *>(cvt)[(kW / 2) * e + 1];
        ulonglong2 rxy = make_ulonglong2(0ull, 0ull), rz0 = rxy;
        if (DF) {
            rxy = reinterpret_cast<const ulonglong2 *>(cvt)[(kW / 2) * e + 2];
            rz0 = reinterpret_cast<const ulonglong2 *>(cvt)[(kW / 2) * e + 3];
        }
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            u64 dx = f2sub(xy.x, xi[p]), dy = f2sub(xy.y, yi[p]), dz = f2sub(zm.x, zi[p]);
            if (DF) {
                dx = f2add(dx, f2sub(rxy.x, exi[p]));
                dy = f2add(dy, f2sub(rxy.y, eyi[p]));
                dz = f2add(dz, f2sub(rz0.x, ezi[p]));
            }
            u64 r2 = f2fma(dx, dx, c0v);
            r2 = f2fma(dy, dy, r2);
            r2 = f2fma(dz, dz, r2);
            float ra, rb;
            up2(r2, ra, rb);
            ra = clamp_pos(ra, smax_bits);
            rb = clamp_pos(rb, smax_bits);
            u64 g;
            if (EXT) {
                const float4 ta = tab4_at(tb0, __float_as_uint(ra), sh3);
                const float4 tb = tab4_at(tb0, __float_as_uint(rb), sh3);
                g = pk2(__fmaf_rn(ra, ta.y, ta.x), __fmaf_rn(rb, tb.y, tb.x));
                ph[p] = f2fma(zm.y, pk2(__fmaf_rn(ra, ta.w, ta.z), __fmaf_rn(rb, tb.w, tb.z)), ph[p]);
            } else {
                const float2 ta = tab_at(tb0, __float_as_uint(ra), sh3);
                const float2 tb = tab_at(tb0, __float_as_uint(rb), sh3);
                g = pk2(__fmaf_rn(ra, ta.y, ta.x), __fmaf_rn(rb, tb.y, tb.x));
            }
            const u64 mg = f2mul(zm.y, g);
            ax[p] = f2fma(mg, dx, ax[p]);
            ay[p] = f2fma(mg, dy, ay[p]);
            az[p] = f2fma(mg, dz, az[p]);
        }
    };

    auto eval = [&](const int *list, int n) {
        __syncthreads();               // the staging's last readers are done; the list is written
        for (int k = tid; k < n; k += kNT) {
            const double4 v = ldg_d4(a.jrec + list[k]);
            const double o[3] = {(v.x - cx) * sc, (v.y - cy) * sc, (v.z - cz) * sc};
            u64 *q = cvt + kW * k;
            const float m = (float)v.w;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const float f = (float)o[d];
                q[d] = pk2(f, f);
                if (DF) {
                    const float r = (float)(o[d] - (double)f);
                    q[4 + d] = pk2(r, r);
                }
            }
            q[3] = pk2(m, m);
            if (DF) q[7] = 0ull;
        }
        if (tid == 0) {                // the pad: zero mass far away adds exactly 0
            u64 *q = cvt + kW * n;
            q[0] = q[1] = q[2] = pk2(1.0e4f, 1.0e4f);
#pragma unroll
            for (int k = 3; k < kW; ++k) q[k] = 0ull;
        }
        __syncthreads();
#pragma unroll
        for (int p = 0; p < NP; ++p) ax[p] = ay[p] = az[p] = ph[p] = 0ull;
        if (dense && n == kTJ) {       // hardly a record to leave out
#pragma unroll 16
            for (int e = 0; e < kTJ; ++e) pair(e);
        } else {
            const int nw = warp_list(wb, false, n, sm.idx, n, [&](int e) {
                const u64 *q = cvt + kW * e;
                return make_float4(__uint_as_float((unsigned)q[0]), __uint_as_float((unsigned)q[1]),
                                   __uint_as_float((unsigned)q[2]), __uint_as_float((unsigned)q[3]));
            });
            if (nw == 0) return;
#pragma unroll 1
            for (int e = 0; e < nw; e += kPadIdx) {
                const ushort4 id = *reinterpret_cast<const ushort4 *>(sm.idx + e);
                pair(id.x);
                pair(id.y);
                pair(id.z);
                pair(id.w);
            }
        }
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            fold2(RH(p, 0), RL(p, 0), ax[p]);
            fold2(RH(p, 1), RL(p, 1), ay[p]);
            fold2(RH(p, 2), RL(p, 2), az[p]);
            if (EXT) fold2(RH(p, 3), RL(p, 3), ph[p]);
        }
    };

    auto end = [&](long long t) {
        double4 *dst = a.part + (size_t)(t + blockIdx.x) * Bi;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            float h[8] = {0, 0, 0, 0, 0, 0, 0, 0}, l[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
            for (int k = 0; k < kComp; ++k) {
                up2(RH(p, k), h[2 * k], h[2 * k + 1]);
                up2(RL(p, k), l[2 * k], l[2 * k + 1]);
            }
#pragma unroll
            for (int q = 0; q < 2; ++q)
                if (t * Bi + LI(p, q) < a.ni)
                    dst[LI(p, q)] = make_double4((double)h[q] + (double)l[q], (double)h[2 + q] + (double)l[2 + q],
                                                 (double)h[4 + q] + (double)l[4 + q], (double)h[6 + q] + (double)l[6 + q]);
        }
    };

    near_stream(a, sm, begin, eval, end);
}

// ---------------------------------------------------------------- backward
// The table's gradients (pg_backward.cu states them), scalar FP32, kBwKI i
// per thread, the knot gradient through a shared-memory histogram.
constexpr int kBiN = kNT * kBwKI;

__global__ void __launch_bounds__(kNT) k_near_backward(NearArgs a)
{
    constexpr int KI = kBwKI;
    extern __shared__ __align__(128) unsigned char smem[];
    const NearShared sm = near_shared(smem);
    float4 *cv = reinterpret_cast<float4 *>(smem + kNearShared);            // [kTJ + 1][2], the last a pad
    float2 *tab = reinterpret_cast<float2 *>(cv + 2 * kTJ + 2);
    float *hist = reinterpret_cast<float *>(tab + a.tab.n);
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    for (int k = tid; k < a.tab.n; k += kNT) {
        tab[k] = a.tab.AG1[k];
        hist[k] = 0.0f;
    }
    float xk[KI], yk[KI], zk[KI], mk[KI], wx[KI], wy[KI], wz[KI];
    float h[KI][4], l[KI][4];                  // compensated sums of dL/dx (3), dL/dm
    auto LI = [&](int q) { return (w * KI + q) * 32 + lane; };
    double cx = 0, cy = 0, cz = 0;
    const double sc = a.tab.scale;
    const float R = sqrtf(a.tab.s_max - 2.0f);
    WarpBox wb;

    auto begin = [&](long long t) {
        const double4 c = a.ctr[t];
        cx = c.x; cy = c.y; cz = c.z;
        wb.clear();
#pragma unroll
        for (int q = 0; q < KI; ++q) {
            const long long i = t * kBiN + LI(q);
            xk[q] = yk[q] = zk[q] = mk[q] = wx[q] = wy[q] = wz[q] = 0.0f;
            if (i < a.ni) {
                const double4 v = a.xi[i], ww = a.wi[i];
                xk[q] = (float)((v.x - cx) * sc);
                yk[q] = (float)((v.y - cy) * sc);
                zk[q] = (float)((v.z - cz) * sc);
                mk[q] = (float)v.w;
                wx[q] = (float)ww.x; wy[q] = (float)ww.y; wz[q] = (float)ww.z;
                wb.add(xk[q], yk[q], zk[q]);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) h[q][k] = l[q][k] = 0.0f;
        }
        wb.close(R, isinf(a.ext[t].x));
    };

    auto eval = [&](const int *list, int n) {
        __syncthreads();               // the staging's last readers are done; the list is written
        bool odd = false;              // a non-finite weight: its pairs are, near or far
        for (int k = tid; k < n; k += kNT) {
            const double4 v = ldg_d4(a.jrec + list[k]), ww = ldg_d4(a.jw + list[k]);
            odd |= odd_weight(ww);
            cv[2 * k] = make_float4((float)((v.x - cx) * sc), (float)((v.y - cy) * sc), (float)((v.z - cz) * sc),
                                    (float)v.w);
            cv[2 * k + 1] = make_float4((float)ww.x, (float)ww.y, (float)ww.z, 0.0f);
        }
        if (tid == 0) {
            cv[2 * n] = make_float4(1.0e4f, 1.0e4f, 1.0e4f, 0.0f);
            cv[2 * n + 1] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
        odd = __syncthreads_or(odd);
        const int nw = warp_list(wb, odd, n, sm.idx, n, [&](int e) { return cv[2 * e]; });
        if (nw == 0) return;
        float g[KI][4];
#pragma unroll
        for (int q = 0; q < KI; ++q) g[q][0] = g[q][1] = g[q][2] = g[q][3] = 0.0f;
#pragma unroll 2
        for (int e0 = 0; e0 < nw; ++e0) {
            const int e = sm.idx[e0];
            const float4 p = cv[2 * e], wj = cv[2 * e + 1];
#pragma unroll
            for (int q = 0; q < KI; ++q) {
                const float dx = p.x - xk[q], dy = p.y - yk[q], dz = p.z - zk[q];
                const float r2 = fmaf(dx, dx, fmaf(dy, dy, fmaf(dz, dz, 2.0f)));
                // u = m_k w_j - m_j w_k with separate roundings: exactly 0 for j = k
                const float ux = __fsub_rn(__fmul_rn(mk[q], wj.x), __fmul_rn(p.w, wx[q]));
                const float uy = __fsub_rn(__fmul_rn(mk[q], wj.y), __fmul_rn(p.w, wy[q]));
                const float uz = __fsub_rn(__fmul_rn(mk[q], wj.z), __fmul_rn(p.w, wz[q]));
                const float du = fmaf(dx, ux, fmaf(dy, uy, dz * uz));
                const float wd = fmaf(dx, wj.x, fmaf(dy, wj.y, dz * wj.z));
                const float sv = fminf(r2, a.tab.s_max);
                const unsigned bits = __float_as_uint(sv);
                const unsigned at = (bits >> a.tab.shift) - a.tab.base;
                const float2 ag = tab[at];
                const float K = fmaf(sv, ag.y, ag.x);
                const float c2 = 2.0f * ag.y * du;
                if (sv < a.tab.s_max) {
                    // hat weights of the bin's two knots; the knot spacing
                    // is 2^(exponent of s_k - F)
                    const unsigned kb = bits & ~((1u << a.tab.shift) - 1u);
                    const float sk = __uint_as_float(kb);
                    const float ds = __uint_as_float((kb & 0x7f800000u) - ((unsigned)(23 - a.tab.shift) << 23));
                    const float tt = (sv - sk) / ds;
                    const float pw = p.w * fmaf(dx, wx[q], fmaf(dy, wy[q], dz * wz[q]));
                    atomicAdd(&hist[at], pw * (1.0f - tt));
                    atomicAdd(&hist[at + 1], pw * tt);
                }
                g[q][0] = fmaf(K, ux, fmaf(c2, dx, g[q][0]));
                g[q][1] = fmaf(K, uy, fmaf(c2, dy, g[q][1]));
                g[q][2] = fmaf(K, uz, fmaf(c2, dz, g[q][2]));
                g[q][3] = fmaf(-K, wd, g[q][3]);
            }
        }
#pragma unroll
        for (int q = 0; q < KI; ++q)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                float s, er;
                two_sum(h[q][k], g[q][k], s, er);
                h[q][k] = s;
                l[q][k] += er;
            }
    };

    auto end = [&](long long t) {
        double4 *dst = a.part + (size_t)(t + blockIdx.x) * kBiN;
#pragma unroll
        for (int q = 0; q < KI; ++q)
            if (t * kBiN + LI(q) < a.ni)
                dst[LI(q)] = make_double4((double)h[q][0] + l[q][0], (double)h[q][1] + l[q][1],
                                          (double)h[q][2] + l[q][2], (double)h[q][3] + l[q][3]);
    };

    if (!near_stream(a, sm, begin, eval, end)) return;
    if (a.dv) {
        __syncthreads();
        for (int k = tid; k < a.tab.n; k += kNT)
            if (hist[k] != 0.0f) atomicAdd(&a.dv[k], (double)hist[k]);
    }
}

// ---------------------------------------------------------------- split
// One CTA per tile, one warp per run of `run` i-particles: each warp takes its
// run's box, then every thread counts its sampled j records within r_cut of
// each box.
constexpr int kCostSample = 2048;      // records sampled: 1 % of the j kept is then 20 +- 4.5
constexpr int kCostWarps = 4;

__global__ void __launch_bounds__(32 * kCostWarps) k_near_cost(NearArgs a, int Bi, int run, float pair_cost,
                                                               float unit_cost, unsigned *__restrict__ cost,
                                                               unsigned char *__restrict__ dense)
{
    __shared__ float box[kCostWarps][6];
    __shared__ int hits[kCostWarps];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const long long t = blockIdx.x;
    const float inf = __int_as_float(0x7f800000);
    const double sc = a.tab.scale;
    const double4 org = a.ctr[0];
    float l[3] = {inf, inf, inf}, h[3] = {-inf, -inf, -inf};
    for (int k = lane; k < run; k += 32) {
        const long long i = t * Bi + (long long)w * run + k;
        if (i >= a.ni) break;
        const double4 v = a.xi[i];
        const float f[3] = {(float)((v.x - org.x) * sc), (float)((v.y - org.y) * sc), (float)((v.z - org.z) * sc)};
        for (int c = 0; c < 3; ++c) { l[c] = fminf(l[c], f[c]); h[c] = fmaxf(h[c], f[c]); }
    }
    for (int c = 0; c < 3; ++c)
        for (int o = 16; o; o >>= 1) {
            l[c] = fminf(l[c], __shfl_xor_sync(0xffffffffu, l[c], o));
            h[c] = fmaxf(h[c], __shfl_xor_sync(0xffffffffu, h[c], o));
        }
    if (lane == 0) {
        for (int c = 0; c < 3; ++c) { box[w][c] = l[c]; box[w][3 + c] = h[c]; }
        hits[w] = 0;
    }
    __syncthreads();
    const bool all = isinf(a.ext[t].x);
    const long long step = (a.nj + kCostSample - 1) / kCostSample, ns = (a.nj + step - 1) / step;
    const float lim = a.tab.s_max - 2.0f;      // the cutoff, squared
    int n[kCostWarps] = {};
#pragma unroll 4
    for (long long q = tid; q < ns; q += 32 * kCostWarps) {
        const float4 j = a.jf[q * step];
#pragma unroll
        for (int k = 0; k < kCostWarps; ++k) {
            const float dx = fmaxf(fmaxf(box[k][0] - j.x, j.x - box[k][3]), 0.0f);
            const float dy = fmaxf(fmaxf(box[k][1] - j.y, j.y - box[k][4]), 0.0f);
            const float dz = fmaxf(fmaxf(box[k][2] - j.z, j.z - box[k][5]), 0.0f);
            if (all || !(dx * dx + dy * dy + dz * dz > lim)) ++n[k];
        }
    }
#pragma unroll
    for (int k = 0; k < kCostWarps; ++k) {
        const int v = __reduce_add_sync(0xffffffffu, n[k]);
        if (lane == 0) atomicAdd(&hits[k], v);
    }
    __syncthreads();
    if (tid == 0) {
        // the CTA's barriers make its slowest warp set the time
        int m = 0;
        for (int k = 0; k < kCostWarps; ++k) m = max(m, hits[k]);
        const float f = ns > 0 ? (float)m / (float)ns : 0.0f;
        cost[t] = (unsigned)(unit_cost + f * (float)a.unit * pair_cost) + 1u;
        dense[t] = f > 0.8f;
    }
}

// Scans the tiles' costs (per unit, times nch units) into prefix, then places
// the CTAs' first units: CTA b starts at cost b C / grid, in the tile that
// holds it at the unit it falls in.
__global__ void __launch_bounds__(1024) k_near_split(const unsigned *__restrict__ cost, int ntiles, int nch, int grid,
                                                     double all_near, u64 *prefix, long long *__restrict__ start,
                                                     int *__restrict__ near)
{
    __shared__ u64 wsum[32];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    u64 base = 0;
    for (int t0 = 0; t0 < ntiles; t0 += 1024) {
        const u64 c = t0 + tid < ntiles ? (u64)cost[t0 + tid] * nch : 0ull;
        u64 x = c;
        for (int o = 1; o < 32; o <<= 1) {
            const u64 y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[w] = x;
        __syncthreads();
        const u64 mine = wsum[lane];
        u64 y = mine;
        for (int o = 1; o < 32; o <<= 1) {
            const u64 z = __shfl_up_sync(0xffffffffu, y, o);
            if (lane >= o) y += z;
        }
        const u64 before = __shfl_sync(0xffffffffu, y - mine, w), total = __shfl_sync(0xffffffffu, y, 31);
        if (t0 + tid < ntiles) prefix[t0 + tid] = base + before + x - c;
        base += total;
        __syncthreads();
    }
    const u64 C = base;
    if (tid == 0) {
        *near = (double)C < kNearShare * all_near;
        start[grid] = (long long)ntiles * nch;
    }
    for (int b = tid; b < grid; b += 1024) {
        const u64 at = (u64)b * C / (unsigned)grid;
        int lo = 0, hi = ntiles - 1;           // the last tile that starts at or before `at`
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (prefix[mid] <= at) lo = mid;
            else hi = mid - 1;
        }
        start[b] = (long long)lo * nch + (long long)((at - prefix[lo]) / cost[lo]);
    }
}

}  // namespace

cudaError_t launch_near_plan(const NearArgs &a, int Bi, int run, float pair_cost, float unit_cost, int grid,
                             unsigned *cost, u64 *prefix, unsigned char *dense, long long *start, int *near,
                             cudaStream_t st)
{
    if (a.ntiles <= 0 || grid <= 0) return cudaSuccess;
    if (Bi != run * kCostWarps) return cudaErrorInvalidValue;
    k_near_cost<<<a.ntiles, 32 * kCostWarps, 0, st>>>(a, Bi, run, pair_cost, unit_cost, cost, dense);
    // the cost if every warp kept everything
    const double all = (double)a.ntiles * a.nch * ((double)a.unit * pair_cost + unit_cost);
    k_near_split<<<1, 1024, 0, st>>>(cost, a.ntiles, a.nch, grid, all, prefix, start, near);
    return cudaGetLastError();
}

int near_stride(int nch)
{
    auto gcd = [](int a, int b) {
        while (b) { const int t = a % b; a = b; b = t; }
        return a;
    };
    int s = (int)(nch * 0.6180339887);          // the golden section spreads any run of steps
    if (s < 1) s = 1;
    while (gcd(s, nch) != 1) ++s;
    return s;
}

// ------------------------------------------------------------------ host

namespace {

template <int NP, bool EXT, bool DF>
cudaError_t configure_near()
{
    static bool done[kMaxDevices] = {};
    return once_per_device(done, [] {
        return cudaFuncSetAttribute(k_near<NP, EXT, DF>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)near_smem(NP, 2 << 13, EXT, DF));
    });
}

cudaError_t configure_near_backward()
{
    static bool done[kMaxDevices] = {};
    return once_per_device(done, [] {
        return cudaFuncSetAttribute(k_near_backward, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)near_backward_smem(1 << 13));
    });
}

// f(NP, EXT, DF) with the run's choice as types
template <typename F>
auto near_pick(int np, bool ext, bool df, F f)
{
    auto e = [&](auto n) {
        if (ext) return df ? f(n, std::true_type{}, std::true_type{}) : f(n, std::true_type{}, std::false_type{});
        return df ? f(n, std::false_type{}, std::true_type{}) : f(n, std::false_type{}, std::false_type{});
    };
    return np == 1 ? e(std::integral_constant<int, 1>{})
         : np == 4 ? e(std::integral_constant<int, 4>{}) : e(std::integral_constant<int, 2>{});
}

}  // namespace

size_t near_smem(int np, int ntab, bool ext, bool df)
{
    return kNearShared + (size_t)(kTJ + 1) * (df ? 8 : 4) * sizeof(u64) +
           (size_t)2 * (ext ? 4 : 3) * np * kNT * sizeof(u64) + (size_t)ntab * sizeof(float2);
}

int near_max_blocks_per_sm(int np, int ntab, bool ext, bool df)
{
    return near_pick(np, ext, df, [&](auto n, auto e, auto d) {
        int nb = 0;
        if (configure_near<n(), e(), d()>() != cudaSuccess) return 1;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_near<n(), e(), d()>, kNT,
                                                          near_smem(n(), ntab, e(), d())) != cudaSuccess)
            return 1;
        return nb > 0 ? nb : 1;
    });
}

cudaError_t launch_near(const NearArgs &a, int grid, int np, bool ext, bool df, size_t smem, cudaStream_t st)
{
    if (grid <= 0) return cudaSuccess;
    return near_pick(np, ext, df, [&](auto n, auto e, auto d) {
        const cudaError_t rc = configure_near<n(), e(), d()>();
        if (rc != cudaSuccess) return rc;
        k_near<n(), e(), d()><<<grid, kNT, smem, st>>>(a);
        return cudaGetLastError();
    });
}

size_t near_backward_smem(int ntab)
{
    return kNearShared + (size_t)(2 * kTJ + 2) * sizeof(float4) + (size_t)ntab * (sizeof(float2) + sizeof(float));
}

int near_backward_max_blocks_per_sm(int ntab)
{
    int nb = 0;
    if (configure_near_backward() != cudaSuccess) return 1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_near_backward, kNT, near_backward_smem(ntab)) !=
        cudaSuccess)
        return 1;
    return nb > 0 ? nb : 1;
}

cudaError_t launch_near_backward(const NearArgs &a, int grid, size_t smem, cudaStream_t st)
{
    if (grid <= 0) return cudaSuccess;
    const cudaError_t rc = configure_near_backward();
    if (rc != cudaSuccess) return rc;
    k_near_backward<<<grid, kNT, smem, st>>>(a);
    return cudaGetLastError();
}

}  // namespace pg
