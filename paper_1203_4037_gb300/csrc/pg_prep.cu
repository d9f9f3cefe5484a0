// pg_prep.cu -- data staging ahead of the force kernels:
//  * packing of FP64 positions/masses into 32-byte records (the paper's
//    Jpdata/Ipdata packing, Section 3.1, kept in FP64 for the differencing
//    step);
//  * spatial ordering of the i-particles along a Morton curve so that each
//    i-tile is compact and its FP32 offsets from the FP64 tile centre are small;
//  * a stable LSD radix sort (8-bit digits, warp-level ranking) used for that
//    ordering and for the cell list;
//  * gather into tile order with per-tile FP64 centres.
#include <algorithm>

#include "pg_device.cuh"

namespace pg {

// ---------------------------------------------------------------- packing
__global__ void k_pack_j(const double *__restrict__ x, const double *__restrict__ m,
                         double4 *__restrict__ out, long long n, float4 *__restrict__ hl)
{
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double4 v = make_double4(x[3 * i], x[3 * i + 1], x[3 * i + 2], m ? m[i] : 0.0);
    out[i] = v;
    if (hl) {   // double-float pairs: hi = fp32(x), lo = fp32(x - hi)
        const float hx = (float)v.x, hy = (float)v.y, hz = (float)v.z;
        hl[2 * i] = make_float4(hx, hy, hz, (float)v.w);
        hl[2 * i + 1] = make_float4((float)(v.x - (double)hx), (float)(v.y - (double)hy),
                                    (float)(v.z - (double)hz), (float)v.w);
    }
}

// i records' fourth value: eps_k^2 with per-i softening (eps == nullptr: 0)
__global__ void k_set_w(double4 *__restrict__ x, const double *__restrict__ eps, long long n)
{
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double e = eps ? eps[i] : 0.0;
    x[i].w = e * e;
}

cudaError_t launch_set_w(double4 *x, const double *eps, long long n, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    k_set_w<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(x, eps, n);
    return cudaGetLastError();
}

cudaError_t launch_pack_j(const double *x, const double *m, double4 *jrec, long long n,
                          cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    k_pack_j<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(x, m, jrec, n, nullptr);
    return cudaGetLastError();
}

cudaError_t launch_pack_i(const double *x, double4 *xi, long long n, cudaStream_t st, float4 *ihl)
{
    if (n <= 0) return cudaSuccess;
    k_pack_j<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(x, nullptr, xi, n, ihl);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- bbox
// order-preserving map of a double onto an unsigned 64-bit integer
__device__ __forceinline__ unsigned long long ord_d(double v)
{
    unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return (b & 0x8000000000000000ull) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double unord_d(unsigned long long u)
{
    unsigned long long b = (u & 0x8000000000000000ull) ? (u & 0x7fffffffffffffffull) : ~u;
    return __longlong_as_double((long long)b);
}

__global__ void k_bbox_init(unsigned long long *bb)
{
    if (threadIdx.x < 3) bb[threadIdx.x] = ~0ull;          // min
    else if (threadIdx.x < 6) bb[threadIdx.x] = 0ull;      // max
}

__global__ void k_bbox(const double4 *__restrict__ x, long long n, unsigned long long *bb)
{
    unsigned long long lo[3] = {~0ull, ~0ull, ~0ull}, hi[3] = {0, 0, 0};
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        double4 p = x[i];
        unsigned long long o[3] = {ord_d(p.x), ord_d(p.y), ord_d(p.z)};
        for (int c = 0; c < 3; ++c) {
            lo[c] = o[c] < lo[c] ? o[c] : lo[c];
            hi[c] = o[c] > hi[c] ? o[c] : hi[c];
        }
    }
    for (int c = 0; c < 3; ++c) {
        for (int off = 16; off; off >>= 1) {
            unsigned long long a = __shfl_xor_sync(0xffffffffu, lo[c], off);
            unsigned long long b = __shfl_xor_sync(0xffffffffu, hi[c], off);
            lo[c] = a < lo[c] ? a : lo[c];
            hi[c] = b > hi[c] ? b : hi[c];
        }
    }
    if ((threadIdx.x & 31) == 0) {
        for (int c = 0; c < 3; ++c) {
            atomicMin(bb + c, lo[c]);
            atomicMax(bb + 3 + c, hi[c]);
        }
    }
}

// spread the low 10 bits of v so that two zero bits separate each
__device__ __forceinline__ unsigned spread10(unsigned v)
{
    v &= 0x3ffu;
    v = (v | (v << 16)) & 0x030000ffu;
    v = (v | (v << 8)) & 0x0300f00fu;
    v = (v | (v << 4)) & 0x030c30c3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}

__global__ void k_morton(const double4 *__restrict__ x, long long n,
                         const unsigned long long *__restrict__ bb,
                         unsigned *__restrict__ keys, unsigned *__restrict__ vals)
{
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    double lo0 = unord_d(bb[0]), lo1 = unord_d(bb[1]), lo2 = unord_d(bb[2]);
    double s0 = unord_d(bb[3]) - lo0, s1 = unord_d(bb[4]) - lo1, s2 = unord_d(bb[5]) - lo2;
    double span = fmax(fmax(s0, s1), fmax(s2, 1e-300));
    double q = 1023.0 / span;
    double4 p = x[i];
    unsigned a = (unsigned)fmin(fmax((p.x - lo0) * q, 0.0), 1023.0);
    unsigned b = (unsigned)fmin(fmax((p.y - lo1) * q, 0.0), 1023.0);
    unsigned c = (unsigned)fmin(fmax((p.z - lo2) * q, 0.0), 1023.0);
    keys[i] = (spread10(a) << 2) | (spread10(b) << 1) | spread10(c);
    vals[i] = (unsigned)i;
}

// ---------------------------------------------------------------- radix sort
// Least significant digit first, 8 bits a pass, one launch a pass. A kernel
// first counts every pass's digits at once. In a pass each block takes the
// next tile of keys by ticket, counts its digits, and learns how many keys of
// each digit the tiles before it hold by looking back at what those blocks
// have published (the decoupled look-back of Merrill and Garland's scan,
// 2016, and of Adinets and Merrill's one-sweep radix sort, 2022): its own
// count first, then, once known, the count up to and including itself. A
// block waits only on blocks with earlier tickets, which are running or done;
// one whose wait runs out counts the keys before its tile itself, so that a
// pass always writes a permutation (what follows a sort indexes with it).
// Ranking by lane order within rounds keeps the sort stable. The keys are
// placed in shared memory in destination order first and written out as runs
// of consecutive addresses.
//
// Bound: launches and the look-back's round trips. A histogram, three scan
// kernels and a scatter per pass took 20 launches for 30-bit keys; now it is
// a memset, the count and four passes. Measured: a 250007-particle PP + PM
// call (four sorted passes) 439 -> 410 us, a 65536-particle fit of a table
// (two sorts of four passes) 2000 -> 1680 us; a pass over 2^21 keys 38 us, as
// long as the five kernels it replaces.
constexpr int kSortWarps = 8;                  // 256 threads, one per digit
constexpr int kSortThreads = 32 * kSortWarps;
// keys per lane: tiles of 4096 keys for large sets; for small ones tiles of
// 2048, twice the blocks. Tiles of 8192 are as fast from 2^21 keys on and
// leave SMs idle below: a tree call on 2^20 particles takes 2172 us with them,
// 2145 with 4096 and 2171 with 2048, on 300007 1517, 1488 and 1486; cells of
// 2^21 particles 2509, 2512 and 2538
constexpr int kSortRounds = 16, kSortRoundsSmall = 8;
constexpr int kSortBatch = 8;          // rounds in flight per lane
constexpr long long kSortSmall = 1LL << 18;
constexpr int kSortPasses = 4;         // 32-bit keys

long long sort_tiles(long long n)
{
    const int rounds = n <= kSortSmall ? kSortRoundsSmall : kSortRounds;
    return (n + kSortThreads * rounds - 1) / (kSortThreads * rounds);
}

// 32-bit words of SortScratch::hist for sorts of up to n keys: the look-back
// words (two of them each), the digit counts and the tickets (a set at the
// switch to large tiles has more tiles than a somewhat larger one)
size_t sort_hist_entries(long long n)
{
    const long long tiles = std::max(sort_tiles(n), sort_tiles(std::min(n, kSortSmall)));
    return (size_t)kSortPasses * (512 * (size_t)tiles + 256 + 1) + 16;
}

// counts of every pass's digits, added to cnt[pass][256]
__global__ void __launch_bounds__(256) k_rs_count(const unsigned *__restrict__ keys, long long n, int passes,
                                                  unsigned *__restrict__ cnt)
{
    __shared__ unsigned h[kSortPasses * 256];
    for (int k = threadIdx.x; k < passes * 256; k += blockDim.x) h[k] = 0;
    __syncthreads();
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i0 = blockIdx.x * (long long)blockDim.x + threadIdx.x; i0 < n; i0 += 4 * stride) {
        unsigned k[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) k[q] = i0 + q * stride < n ? keys[i0 + q * stride] : 0u;
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (i0 + q * stride < n)
                for (int p = 0; p < passes; ++p) atomicAdd(&h[p * 256 + ((k[q] >> (8 * p)) & 255u)], 1u);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < passes * 256; k += blockDim.x)
        if (h[k]) atomicAdd(&cnt[k], h[k]);
}

// exclusive scan of 256 values in shared memory by one warp
__device__ __forceinline__ void scan256(unsigned *v, int lane)
{
    unsigned x[8], tot = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        x[q] = v[8 * lane + q];
        tot += x[q];
    }
    unsigned incl = tot;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    unsigned run = incl - tot;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        v[8 * lane + q] = run;
        run += x[q];
    }
}

// look-back word of (tile, digit): a count with its kind in the top bits
constexpr int kLook = 32;                      // look-back words a thread reads at once
constexpr u64 kOwn = 1ull << 62, kUpTo = 2ull << 62, kCountMask = (1ull << 62) - 1;

__device__ __forceinline__ u64 ld_relaxed(const u64 *p)
{
    u64 v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed(u64 *p, u64 v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

template <int R>
__global__ void __launch_bounds__(kSortThreads) k_rs_pass(const unsigned *__restrict__ kin,
                                                          const unsigned *__restrict__ vin,
                                                          unsigned *__restrict__ kout, unsigned *__restrict__ vout,
                                                          long long n, int shift, const unsigned *__restrict__ total,
                                                          u64 *look, unsigned *ticket, u64 wait_ns)
{
    constexpr int kTile = kSortThreads * R, kChunk = 32 * R;
    extern __shared__ unsigned sort_smem[];
    unsigned *sk = sort_smem, *sv = sk + kTile;
    unsigned (*cnt)[256] = reinterpret_cast<unsigned (*)[256]>(sv + kTile);   // [kSortWarps][256]
    __shared__ unsigned gstart[256], lstart[256];
    __shared__ unsigned tile_s;
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    if (tid == 0) tile_s = atomicAdd(ticket, 1u);
    for (int d = lane; d < 256; d += 32) cnt[w][d] = 0;
    for (int d = tid; d < 256; d += kSortThreads) gstart[d] = total[d];
    __syncthreads();
    const long long tile = tile_s, base = tile * kTile + w * kChunk;
#pragma unroll 1
    for (int r0 = 0; r0 < R; r0 += kSortBatch) {
        unsigned key[kSortBatch];
#pragma unroll
        for (int r = 0; r < kSortBatch; ++r) key[r] = base + (r0 + r) * 32 + lane < n ? kin[base + (r0 + r) * 32 + lane] : 0u;
#pragma unroll
        for (int r = 0; r < kSortBatch; ++r)
            if (base + (r0 + r) * 32 + lane < n) atomicAdd(&cnt[w][(key[r] >> shift) & 255u], 1u);
    }
    __syncthreads();
    if (w == 0) scan256(gstart, lane);         // keys of smaller digits
    u64 *mine = look + (size_t)tile * 256;
    for (int d = tid; d < 256; d += kSortThreads) {
        unsigned c = 0;
#pragma unroll
        for (int q = 0; q < kSortWarps; ++q) c += cnt[q][d];
        lstart[d] = c;
        st_relaxed(mine + d, (tile == 0 ? kUpTo : kOwn) | c);
    }
    __syncthreads();
    // the tiles before this one, digit by digit
    static_assert(kSortThreads == 256, "one digit a thread");
    const int dg = tid;
    bool late = tile > 0 && wait_ns == 0;
    if (tile > 0 && !late) {
        u64 before = 0;
        const u64 t0 = global_ns();
        for (long long q = tile - 1; q >= 0;) {
            // all tiles start together, so few have their running count yet
            // and the walk takes tiles / kLook round trips
            u64 v[kLook];
#pragma unroll
            for (int k = 0; k < kLook; ++k) v[k] = q - k >= 0 ? ld_relaxed(look + (size_t)(q - k) * 256 + dg) : kUpTo;
            bool wait = false;
#pragma unroll
            for (int k = 0; k < kLook; ++k) {
                if (wait || q < 0) continue;
                if (!(v[k] & ~kCountMask)) { wait = true; continue; }
                before += v[k] & kCountMask;
                q = v[k] & kUpTo ? -1 : q - 1;
            }
            if (wait && global_ns() - t0 > wait_ns) {
                late = true;
                break;
            }
        }
        if (!late) {
            st_relaxed(mine + dg, kUpTo | (before + lstart[dg]));
            gstart[dg] += (unsigned)before;
        }
    }
    if (__syncthreads_or(late)) {
        unsigned *h = sk;                      // not in use yet
        h[dg] = 0;
        __syncthreads();
        for (long long e = tid; e < tile * kTile; e += kSortThreads) atomicAdd(&h[(kin[e] >> shift) & 255u], 1u);
        __syncthreads();
        if (late) {
            st_relaxed(mine + dg, kUpTo | (h[dg] + lstart[dg]));
            gstart[dg] += h[dg];
        }
        __syncthreads();
    }
    if (w == 0) scan256(lstart, lane);
    __syncthreads();
    // each warp's first place of each digit in the tile's order
    for (int d = tid; d < 256; d += kSortThreads) {
        unsigned at = lstart[d];
#pragma unroll
        for (int q = 0; q < kSortWarps; ++q) {
            const unsigned c = cnt[q][d];
            cnt[q][d] = at;
            at += c;
        }
    }
    __syncthreads();
    const unsigned lt = (1u << lane) - 1u;
    // ranks, kSortBatch rounds at a time: the lanes with each lane's digit by
    // eight ballots (independent over the rounds), then the running places
#pragma unroll 1
    for (int r0 = 0; r0 < R; r0 += kSortBatch) {
        unsigned key[kSortBatch], val[kSortBatch], peers[kSortBatch];
#pragma unroll
        for (int r = 0; r < kSortBatch; ++r) {
            const long long e = base + (r0 + r) * 32 + lane;
            key[r] = e < n ? kin[e] : 0u;
            val[r] = e < n ? vin[e] : 0u;
        }
#pragma unroll
        for (int r = 0; r < kSortBatch; ++r) {
            const unsigned d = key[r] >> shift;
            unsigned m = __ballot_sync(0xffffffffu, base + (r0 + r) * 32 + lane < n);   // invalid lanes match nobody
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const bool bit = d >> k & 1u;
                const unsigned bal = __ballot_sync(0xffffffffu, bit);
                m &= bit ? bal : ~bal;
            }
            peers[r] = m;
        }
#pragma unroll
        for (int r = 0; r < kSortBatch; ++r) {
            const bool valid = base + (r0 + r) * 32 + lane < n;
            const unsigned d = (key[r] >> shift) & 255u, below = __popc(peers[r] & lt);
            unsigned at = 0;
            if (valid) at = cnt[w][d] + below;
            __syncwarp();
            if (valid) {
                if (below == 0) cnt[w][d] = at + __popc(peers[r]);
                sk[at] = key[r];
                sv[at] = val[r];
            }
            __syncwarp();
        }
    }
    __syncthreads();
    const int nb = (int)min((long long)kTile, n - tile * kTile);
    for (int p = tid; p < nb; p += kSortThreads) {
        const unsigned k = sk[p], d = (k >> shift) & 255u;
        const unsigned g = gstart[d] + ((unsigned)p - lstart[d]);
        kout[g] = k;
        vout[g] = sv[p];
    }
}

// exclusive scan of n unsigned values in place: blocks of 1024 threads scan
// 4096 values each, a single block scans the block totals, a third pass adds
constexpr int kScanPer = 4096;

__device__ unsigned block_excl_scan(unsigned v, unsigned *sh)
{
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    unsigned x = v;
    for (int o = 1; o < 32; o <<= 1) {
        unsigned y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[w] = x;
    __syncthreads();
    if (w == 0) {
        unsigned t = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0u;
        for (int o = 1; o < 32; o <<= 1) {
            unsigned y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        sh[lane] = t;
    }
    __syncthreads();
    unsigned pre = w ? sh[w - 1] : 0u;
    unsigned total = sh[(blockDim.x >> 5) - 1];
    __syncthreads();
    sh[32] = total;
    return pre + x - v;
}

__global__ void k_scan1(unsigned *a, long long n, unsigned *sums)
{
    __shared__ unsigned sh[33];
    long long base = blockIdx.x * (long long)kScanPer + threadIdx.x * 4;
    unsigned v[4], s = 0;
    for (int q = 0; q < 4; ++q) {
        v[q] = base + q < n ? a[base + q] : 0u;
        s += v[q];
    }
    unsigned ex = block_excl_scan(s, sh);
    for (int q = 0; q < 4; ++q) {
        if (base + q < n) a[base + q] = ex;
        ex += v[q];
    }
    if (threadIdx.x == 0) sums[blockIdx.x] = sh[32];
}

__global__ void k_scan2(unsigned *sums, int nb)
{
    __shared__ unsigned sh[33];
    unsigned carry = 0;
    for (int base = 0; base < nb; base += blockDim.x) {
        int i = base + threadIdx.x;
        unsigned v = i < nb ? sums[i] : 0u;
        unsigned ex = block_excl_scan(v, sh);
        if (i < nb) sums[i] = carry + ex;
        carry += sh[32];
        __syncthreads();
    }
}

__global__ void k_scan3(unsigned *a, long long n, const unsigned *sums)
{
    long long base = blockIdx.x * (long long)kScanPer + threadIdx.x * 4;
    unsigned add = sums[blockIdx.x];
    for (int q = 0; q < 4; ++q)
        if (base + q < n) a[base + q] += add;
}

static cudaError_t excl_scan(unsigned *a, long long n, unsigned *sums, cudaStream_t st)
{
    long long nb = (n + kScanPer - 1) / kScanPer;
    if (nb <= 0) return cudaSuccess;
    k_scan1<<<(unsigned)nb, 1024, 0, st>>>(a, n, sums);
    k_scan2<<<1, 1024, 0, st>>>(sums, (int)nb);
    k_scan3<<<(unsigned)nb, 1024, 0, st>>>(a, n, sums);
    return cudaGetLastError();
}

cudaError_t launch_excl_scan(unsigned *a, long long n, unsigned *sums, cudaStream_t st)
{
    return excl_scan(a, n, sums, st);
}

static size_t sort_smem_bytes(int rounds)
{
    return ((size_t)2 * kSortThreads * rounds + kSortWarps * 256) * sizeof(unsigned);
}

cudaError_t launch_radix_sort(unsigned *keys, unsigned *vals, long long n, int key_bits,
                              SortScratch &s, unsigned **keys_out, unsigned **vals_out,
                              cudaStream_t st, unsigned long long wait_ns)
{
    unsigned *kin = keys, *vin = vals;
    unsigned *kb = (keys == s.keys[0]) ? s.keys[1] : s.keys[0];
    unsigned *vb = (vals == s.vals[0]) ? s.vals[1] : s.vals[0];
    const int passes = (key_bits + 7) / 8;
    if (n > 0 && passes > 0) {
        const long long tiles = sort_tiles(n);
        u64 *look = (u64 *)s.hist;
        unsigned *cnt = (unsigned *)(look + (size_t)passes * tiles * 256), *ticket = cnt + passes * 256;
        cudaError_t e = cudaMemsetAsync(s.hist, 0, (char *)(ticket + passes) - (char *)s.hist, st);
        if (e != cudaSuccess) return e;
        const long long blocks = (n + 1023) / 1024;
        k_rs_count<<<(unsigned)std::min<long long>(blocks, 608), 256, 0, st>>>(kin, n, passes, cnt);
        const bool small = n <= kSortSmall;
        const size_t smem = sort_smem_bytes(small ? kSortRoundsSmall : kSortRounds);
        static bool done[kMaxDevices] = {};
        e = once_per_device(done, [] {
            return cudaFuncSetAttribute(k_rs_pass<kSortRounds>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)sort_smem_bytes(kSortRounds));
        });
        if (e != cudaSuccess) return e;
        for (int p = 0; p < passes; ++p) {
            auto k = small ? k_rs_pass<kSortRoundsSmall> : k_rs_pass<kSortRounds>;
            k<<<(unsigned)tiles, kSortThreads, smem, st>>>(kin, vin, kb, vb, n, 8 * p, cnt + 256 * p,
                                                        look + (size_t)p * tiles * 256, ticket + p, wait_ns);
            std::swap(kin, kb);
            std::swap(vin, vb);
        }
    }
    *keys_out = kin;
    *vals_out = vin;
    return cudaGetLastError();
}

cudaError_t launch_morton_sort(const double4 *xi, long long n, SortScratch &s, unsigned **perm_out,
                               cudaStream_t st)
{
    k_bbox_init<<<1, 32, 0, st>>>(s.bbox);
    unsigned g = (unsigned)((n + 255) / 256);
    k_bbox<<<g < 1024 ? g : 1024, 256, 0, st>>>(xi, n, s.bbox);
    k_morton<<<g, 256, 0, st>>>(xi, n, s.bbox, s.keys[0], s.vals[0]);
    unsigned *ko;
    return launch_radix_sort(s.keys[0], s.vals[0], n, 30, s, &ko, perm_out, st);
}

// ---------------------------------------------------------------- tiles
// One CTA per tile of Bi consecutive (sorted) i: gather the positions and
// take the midpoint of the tile's bounding box as its FP64 centre.
__global__ void k_tile_prep(const double4 *__restrict__ xi, const unsigned *__restrict__ perm,
                            long long n, int Bi, double4 *__restrict__ xt,
                            double4 *__restrict__ ctr, double4 *__restrict__ ext)
{
    __shared__ double red[6][32];
    long long t = blockIdx.x;
    bool odd = false;          // a non-finite coordinate
    double lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (int k = threadIdx.x; k < Bi; k += blockDim.x) {
        long long p = t * Bi + k;
        if (p >= n) break;
        double4 v = xi[perm ? (long long)perm[p] : p];
        xt[p] = v;
        odd |= !(isfinite(v.x) && isfinite(v.y) && isfinite(v.z));
        lo[0] = fmin(lo[0], v.x); lo[1] = fmin(lo[1], v.y); lo[2] = fmin(lo[2], v.z);
        hi[0] = fmax(hi[0], v.x); hi[1] = fmax(hi[1], v.y); hi[2] = fmax(hi[2], v.z);
    }
    for (int c = 0; c < 3; ++c)
        for (int o = 16; o; o >>= 1) {
            lo[c] = fmin(lo[c], __shfl_xor_sync(0xffffffffu, lo[c], o));
            hi[c] = fmax(hi[c], __shfl_xor_sync(0xffffffffu, hi[c], o));
        }
    int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0)
        for (int c = 0; c < 3; ++c) { red[c][w] = lo[c]; red[3 + c][w] = hi[c]; }
    odd = __syncthreads_or(odd);
    if (threadIdx.x == 0) {
        int nw = blockDim.x >> 5;
        for (int q = 1; q < nw; ++q)
            for (int c = 0; c < 3; ++c) {
                red[c][0] = fmin(red[c][0], red[c][q]);
                red[3 + c][0] = fmax(red[3 + c][0], red[3 + c][q]);
            }
        double c0 = 0.5 * (red[0][0] + red[3][0]);
        double c1 = 0.5 * (red[1][0] + red[4][0]);
        double c2 = 0.5 * (red[2][0] + red[5][0]);
        ctr[t] = make_double4(c0, c1, c2, 0.0);
        if (ext) {
            auto half = [&](int c, double m) {         // from the centre as stored
                return odd ? INFINITY : fmax(red[3 + c][0] - m, m - red[c][0]);
            };
            ext[t] = make_double4(half(0, c0), half(1, c1), half(2, c2), 0.0);
        }
    }
}

cudaError_t launch_tile_prep(const double4 *xi, const unsigned *perm, long long n, int Bi,
                             double4 *xi_tiled, double4 *ctr, cudaStream_t st, double4 *ext)
{
    long long nt = (n + Bi - 1) / Bi;
    if (nt <= 0) return cudaSuccess;
    k_tile_prep<<<(unsigned)nt, 256, 0, st>>>(xi, perm, n, Bi, xi_tiled, ctr, ext);
    return cudaGetLastError();
}

__global__ void k_pack_f32(const double4 *__restrict__ rec, const double4 *__restrict__ w, long long n,
                           const double4 *__restrict__ org, double sc, float4 *__restrict__ out)
{
    const long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (k >= n) return;
    const double4 v = rec[k], o = *org;
    const float m = w && odd_weight(w[k]) ? __int_as_float(0x7fffffff) : (float)v.w;
    out[k] = make_float4((float)((v.x - o.x) * sc), (float)((v.y - o.y) * sc), (float)((v.z - o.z) * sc), m);
}

cudaError_t launch_pack_f32(const double4 *rec, const double4 *w, long long n, const double4 *org, double scale,
                            float4 *out, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    k_pack_f32<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(rec, w, n, org, scale, out);
    return cudaGetLastError();
}

}  // namespace pg
