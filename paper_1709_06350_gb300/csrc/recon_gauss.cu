// recon_gauss.cu -- 1-point Gaussianisation of a field (Sec. III: the paper
// tried it on delta_r), read as the rank mapping
//     g_i = mean + std * Phi^-1((rank_i + 1/2) / n),
// rank_i the position of value i in ascending order, ties broken by
// position; mean and std (population) of the input.
//
// Ranks come from buckets: the values are mapped by a monotone function to
// ~n/11 buckets of nearly equal occupancy, counted and scattered in one pass
// each, and a value's rank is its bucket's start plus the bucket's smaller
// (key, index) pairs.  The map takes 52 bits linear in the value (the
// significand of v + c, one rounded addition), their top 12 as a cell, and in
// each cell a power of two of sub-buckets by its share of a 1/16 sample.
// Fields that defeat it (heavy ties: the sum of squared occupancies says what
// the comparisons would cost) take a least-significant-digit radix sort of
// (key, index) pairs instead, 8 passes of 8-bit digits; both paths are
// enqueued and the device decides, so the call stays asynchronous.
//
// The quantile is FP64 and was half of the time (normcdfinv, ~67 FP64
// operations per value at one per 64 FP32 ones): it is evaluated once per 128
// ranks and continued by its Taylor series (five FP64 operations per value).
// What bounds it: the sector traffic of the scatters and the FP64 pipe.
// Measured (GB300): 256^3 4.24 -> 1.35 to 1.50 ms (GPUs differ; scatter 0.43 to
// 0.52, ranks 0.38 to 0.44, places 0.16), 512^3 36.9 -> 12.1 to 12.7 ms; a 256^3 field of
// rounded values (radix path) 3.5 -> 1.8 ms.  Fields that take the radix path are
// 3 to 5% slower than by it alone at 64^3 and 80^3, and faster at other sides.
#include <climits>
#include <cmath>

#include "dfloat.cuh"
#include "internal.cuh"

namespace recon {

#define CK(expr)                                \
    do {                                        \
        const cudaError_t ck_e = (expr);        \
        if (ck_e != cudaSuccess) return ck_e;   \
    } while (0)

constexpr int kRadixThreads = 256;
constexpr int kRadixItems = 16;                        // items per thread per tile
constexpr int kTile = kRadixThreads * kRadixItems;     // 4096
constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanSeg = kScanThreads * kScanItems;    // 4096 counts per scan block

// the value's bits as an order-preserving unsigned integer (-0 as +0), and back
__device__ __forceinline__ unsigned long long order_key(double v)
{
    unsigned long long b = (unsigned long long)__double_as_longlong(v);
    if ((b << 1) == 0) b = 0;
    return (b >> 63) ? ~b : (b | (1ull << 63));
}
__device__ __forceinline__ double key_value(unsigned long long k)
{
    return __longlong_as_double((long long)((k >> 63) ? (k ^ (1ull << 63)) : ~k));
}

// ---- what the device decides and shares (one per handle)
constexpr int kCells = 4096;                 // top 12 of the 52 linear bits
constexpr int kCellBits = 40;                // bits within a cell
constexpr int kPerBucket = 16;               // values per bucket: 8 to 16 where the sample is right
constexpr int kSampleRun = 256, kSampleStep = 16 * kSampleRun;
constexpr unsigned long long kMaxWork = 128; // comparisons per value above which the radix sort runs
struct GaussPlan {
    double mean, sd;
    double shift;                            // c: v + c lies in [2^e, 2^(e+1))
    unsigned long long base;                 // bits of 2^e
    unsigned long long squares;              // sum of squared bucket occupancies
    int bad;                                 // no usable range
    unsigned cell[kCells];                   // sampled counts, then first bucket
    unsigned char down[kCells];              // bits to drop within the cell
};
__device__ __forceinline__ bool use_radix(const GaussPlan *P, size_t n) { return P->bad || P->squares > kMaxWork * n; }

__device__ __forceinline__ unsigned long long linear_bits(const GaussPlan *P, double v)
{
    const long long u = __double_as_longlong(v + P->shift) - (long long)P->base;
    return u < 0 ? 0ull : (u >= (1ll << 52) ? (1ull << 52) - 1 : (unsigned long long)u);
}

// mean, population std, the linear map; clears the cells (one block of kThreads)
__device__ __noinline__ void gauss_moments(const double *partials, int nb, double n, GaussPlan *P)
{
    __shared__ double sh[2 * 32];
    __shared__ unsigned long long smin[kThreads / 32], smax[kThreads / 32];
    double sums[2];
    total_columns<kThreads>(partials, nb, sh, sums);
    unsigned long long kmin = ~0ull, kmax = 0ull;
    for (int i = threadIdx.x; i < nb; i += kThreads) {
        const unsigned long long x = (unsigned long long)__double_as_longlong(__ldcg(partials + 4 * i + 2));
        const unsigned long long y = (unsigned long long)__double_as_longlong(__ldcg(partials + 4 * i + 3));
        kmin = x < kmin ? x : kmin;
        kmax = y > kmax ? y : kmax;
    }
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long x = __shfl_xor_sync(0xffffffffu, kmin, o), y = __shfl_xor_sync(0xffffffffu, kmax, o);
        kmin = x < kmin ? x : kmin;
        kmax = y > kmax ? y : kmax;
    }
    if ((threadIdx.x & 31) == 0) {
        smin[threadIdx.x >> 5] = kmin;
        smax[threadIdx.x >> 5] = kmax;
    }
    for (int c = threadIdx.x; c < kCells; c += kThreads) P->cell[c] = 0;
    __syncthreads();
    if (ltid() == 0) {
        for (int w = 1; w < kThreads / 32; ++w) {
            kmin = smin[w] < kmin ? smin[w] : kmin;
            kmax = smax[w] > kmax ? smax[w] : kmax;
        }
        const double m = sums[0] / n, var = sums[1] / n - m * m;
        P->mean = m;
        P->sd = var > 0.0 ? sqrt(var) : 0.0;
        const double lo = key_value(kmin), range = key_value(kmax) - lo;
        P->squares = 0;
        // (equal values, ranges that overflow or underflow the significand map)
        P->bad = !(range > 1e-290 && range < 1e290 && fabs(lo) < 1e290);
        int e = 0;
        frexp(range, &e);                    // range < 2^e
        const double top = ldexp(1.0, P->bad ? 0 : e);
        P->shift = top - lo;
        P->base = (unsigned long long)__double_as_longlong(top);
    }
}

// per-block sums of v and v^2, smallest and largest key; the last block makes
// the moments and the map of them
__global__ void __launch_bounds__(kThreads)
k_gauss_stats(const double *__restrict__ v, size_t n, double *__restrict__ partials, unsigned *__restrict__ counter,
              GaussPlan *__restrict__ P)
{
    __shared__ double sh[32];
    __shared__ unsigned long long smin[kThreads / 32], smax[kThreads / 32];
    double s1 = 0.0, s2 = 0.0;
    unsigned long long kmin = ~0ull, kmax = 0ull;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const double x = v[i];
        const unsigned long long k = order_key(x);
        kmin = k < kmin ? k : kmin;
        kmax = k > kmax ? k : kmax;
        s1 += x;
        s2 = fma(x, x, s2);
    }
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long a = __shfl_xor_sync(0xffffffffu, kmin, o), b = __shfl_xor_sync(0xffffffffu, kmax, o);
        kmin = a < kmin ? a : kmin;
        kmax = b > kmax ? b : kmax;
    }
    if ((threadIdx.x & 31) == 0) {
        smin[threadIdx.x >> 5] = kmin;
        smax[threadIdx.x >> 5] = kmax;
    }
    double t = block_sum<kThreads>(s1, sh);
    if (ltid() == 0) partials[4 * blockIdx.x + 0] = t;
    t = block_sum<kThreads>(s2, sh);
    if (ltid() == 0) {
        partials[4 * blockIdx.x + 1] = t;
        for (int w = 1; w < kThreads / 32; ++w) {
            kmin = smin[w] < kmin ? smin[w] : kmin;
            kmax = smax[w] > kmax ? smax[w] : kmax;
        }
        partials[4 * blockIdx.x + 2] = __longlong_as_double((long long)kmin);
        partials[4 * blockIdx.x + 3] = __longlong_as_double((long long)kmax);
    }
    if (last_block(counter)) gauss_moments(partials, gridDim.x, (double)n, P);
}

__device__ __forceinline__ unsigned block_excl_scan(unsigned v, unsigned *sh, unsigned *total);

// bucket of every value and its place among the bucket's arrivals.  Arrivals at
// one counter queue (2.3 ns each), so a warp takes the places of one bucket by one
// atomic, and a bucket that alone would take a sixteenth of kMaxWork (`most`
// values) ends the count: stored by the arrival that fills it, not by all after it
// (160^3, half of it zeros: 1.41 ms before the radix sort began).  The flag is read
// every fourth turn: read every turn, its one cache line took 0.15 ms at 256^3.
__global__ void __launch_bounds__(kThreads)
k_gauss_count(const double *__restrict__ v, size_t n, GaussPlan *__restrict__ P, unsigned *__restrict__ counts,
              uint2 *__restrict__ where, unsigned most)
{
    volatile int *bad = &P->bad;
    const unsigned lane = threadIdx.x & 31;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    int turn = 0;
    for (size_t first = (size_t)blockIdx.x * blockDim.x + (threadIdx.x - lane); first < n; first += stride) {
        if ((turn++ & 3) == 0 && __any_sync(0xffffffffu, *bad)) return;
        const size_t i = first + lane;
        const bool on = i < n;
        unsigned b = ~0u;
        if (on) {
            const unsigned long long u = linear_bits(P, __ldcs(v + i));
            const unsigned c = (unsigned)(u >> kCellBits);
            b = P->cell[c] + (unsigned)((u & ((1ull << kCellBits) - 1)) >> P->down[c]);
        }
        const unsigned peers = __match_any_sync(0xffffffffu, b);
        const int leader = __ffs(peers) - 1;
        unsigned at = 0;
        if (on && (int)lane == leader) at = atomicAdd(&counts[b], (unsigned)__popc(peers));
        at = __shfl_sync(0xffffffffu, at, leader) + __popc(peers & ((1u << lane) - 1u));
        if (on) {
            __stcs(where + i, make_uint2(b, at));
            if (at == most) *bad = 1;
        }
    }
}

// a value in its bucket: one 16-byte store per value
struct __align__(16) Member {
    unsigned long long key;
    unsigned index, bucket;
};
__global__ void __launch_bounds__(kThreads)
k_gauss_scatter(const double *__restrict__ v, size_t n, const GaussPlan *__restrict__ P,
                const unsigned *__restrict__ start, const uint2 *__restrict__ where, Member *__restrict__ out)
{
    if (use_radix(P, n)) return;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        // (streaming reads, so that the members being filled keep the L2)
        const uint2 w = __ldcs(where + i);
        Member m;
        m.key = order_key(__ldcs(v + i));
        m.index = (unsigned)i;
        m.bucket = w.x;
        *reinterpret_cast<int4 *>(out + start[w.x] + w.y) = *reinterpret_cast<const int4 *>(&m);
    }
}

// ---- quantiles: out = mean + std Phi^-1((r + 1/2) / n).  With z = Phi^-1(q)
// and D = dz/dr = sqrt(2 pi) exp(z^2/2) / n, the k-th derivative with respect
// to r is P_k(z) D^k, P_1 = 1, P_{k+1} = P_k' + k z P_k; the series about the
// middle of 128 ranks in terms of their offset is kept per anchor.  From rank
// kTail on an offset is below 2^-8 of the rank and six terms leave 2^-58; the
// terms from the fourth on are below 2^-32 and evaluated in FP32, for z itself:
// with std in them they left FP32's range (infinities from std 3e56 up, 2e-11
// of std lost below 1e-24).  The lower half is mirrored, so the two tails have
// the same precision.
constexpr int kAnchor = 128;
constexpr size_t kTail = 16384;
struct __align__(64) Anchor {
    double z, c1, c2, c3;
    float c4, c5, c6, unused[5];
};
__device__ __forceinline__ void make_anchor(size_t n, size_t a, Anchor *__restrict__ out)
{
    const double z = normcdfinv(((double)(a * kAnchor + kAnchor / 2) + 0.5) / (double)n), z2 = z * z;
    const double D = 2.5066282746310002 * exp(0.5 * z2) / (double)n;   // sqrt(2 pi)
    const double D2 = D * D, D3 = D2 * D;
    Anchor x;
    x.z = z;
    x.c1 = D;
    x.c2 = D2 * z * 0.5;
    x.c3 = D3 * (1.0 + 2.0 * z2) * (1.0 / 6.0);
    x.c4 = (float)(D2 * D2 * z * (7.0 + 6.0 * z2) * (1.0 / 24.0));
    x.c5 = (float)(D2 * D3 * (7.0 + z2 * (46.0 + 24.0 * z2)) * (1.0 / 120.0));
    x.c6 = (float)(D3 * D3 * z * (127.0 + z2 * (326.0 + 120.0 * z2)) * (1.0 / 720.0));
    out[a] = x;
}

// sub-buckets of every cell: a power of two above its share / kPerBucket
// (below n / 8 + kCells buckets in all); one block of kSampleRun threads
__device__ __noinline__ void gauss_plan(int weight, GaussPlan *P)
{
    __shared__ unsigned sh[32];
    constexpr int kPer = kCells / kSampleRun;
    unsigned lg[kPer], sum = 0;
    for (int i = 0; i < kPer; ++i) {
        const unsigned want = (__ldcg(&P->cell[threadIdx.x * kPer + i]) * (unsigned)weight) / kPerBucket;
        lg[i] = want ? 32 - __clz(want) - (__popc(want) == 1) : 0;   // ceil(log2(want))
        sum += 1u << lg[i];
    }
    unsigned total;
    unsigned run = block_excl_scan(sum, sh, &total);
    for (int i = 0; i < kPer; ++i) {
        P->cell[threadIdx.x * kPer + i] = run;
        P->down[threadIdx.x * kPer + i] = (unsigned char)(kCellBits - lg[i]);
        run += 1u << lg[i];
    }
}

// Cell counts of the sample (kSampleRun of every kSampleStep values, or all of a
// small field) by the first `blocks` blocks; the anchors by the others, hidden
// behind the sample; the plan by the last
__global__ void __launch_bounds__(kSampleRun)
k_gauss_sample(const double *__restrict__ v, size_t n, size_t step, unsigned blocks, int weight,
               GaussPlan *__restrict__ P, size_t anchors, Anchor *__restrict__ out, unsigned *__restrict__ counter)
{
    __shared__ unsigned c[kCells];
    const bool bad = P->bad;
    if (blockIdx.x >= blocks) {
        const size_t a = (size_t)(blockIdx.x - blocks) * kSampleRun + threadIdx.x;
        if (a < anchors) make_anchor(n, a, out);
    } else if (!bad) {
        for (int i = threadIdx.x; i < kCells; i += kSampleRun) c[i] = 0;
        __syncthreads();
        for (size_t b = (size_t)blockIdx.x * step; b < n; b += (size_t)blocks * step)
            if (b + threadIdx.x < n) atomicAdd(&c[linear_bits(P, v[b + threadIdx.x]) >> kCellBits], 1u);
        __syncthreads();
        for (int i = threadIdx.x; i < kCells; i += kSampleRun)
            if (c[i]) atomicAdd(&P->cell[i], c[i]);
    }
    __syncthreads();   // the block's counts before its ticket
    if (last_block(counter) && !bad) gauss_plan(weight, P);
}
__device__ __noinline__ double quantile_tail(size_t lo, bool low, size_t n, double m, double sd)
{
    const double z = normcdfinv(((double)lo + 0.5) / (double)n);
    return m + sd * (low ? z : -z);
}
__device__ __forceinline__ double quantile(size_t r, size_t n, const GaussPlan *P, const Anchor *anchors)
{
    const size_t lo = r < n - 1 - r ? r : n - 1 - r;
    if (lo < kTail) return quantile_tail(lo, r == lo, n, P->mean, P->sd);
    const Anchor &x = anchors[lo / kAnchor];
    const float f = (float)((int)(lo & (kAnchor - 1)) - kAnchor / 2);
    const double d = df_f2d_bits(f);
    const double p = df_f2d_bits(fmaf(fmaf(x.c6, f, x.c5), f, x.c4));
    const double z = fma(fma(fma(fma(p, d, x.c3), d, x.c2), d, x.c1), d, x.z);
    return fma(r == lo ? P->sd : -P->sd, z, P->mean);
}

// rank of every member within its bucket, and its quantile to its place
__global__ void __launch_bounds__(kThreads)
k_gauss_rank(const Member *__restrict__ mem, size_t n, const GaussPlan *__restrict__ P,
             const unsigned *__restrict__ start, const Anchor *__restrict__ anchors, double *__restrict__ g)
{
    if (use_radix(P, n)) return;
    for (size_t p = (size_t)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += (size_t)gridDim.x * blockDim.x) {
        const Member m = mem[p];
        const unsigned lo = start[m.bucket], hi = start[m.bucket + 1];
        unsigned r = lo;
        for (unsigned j = lo; j < hi; ++j) {
            const Member o = mem[j];
            r += o.key < m.key || (o.key == m.key && o.index < m.index);
        }
        g[m.index] = quantile(r, n, P, anchors);
    }
}

// ---- the radix sort (P: run only where the buckets do not serve).  The first
// pass (FIRST) takes the keys from the values v, with their positions as indices.
// counts[d * ntile + tile] = occurrences of digit d in the tile
template <bool FIRST>
__global__ void __launch_bounds__(kRadixThreads)
k_radix_hist(const unsigned long long *__restrict__ key, const double *__restrict__ v, size_t n, int shift, int ntile,
             unsigned *__restrict__ counts, const GaussPlan *__restrict__ P)
{
    __shared__ unsigned hist[256];
    if (!use_radix(P, n)) return;
    for (int tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
        hist[threadIdx.x] = 0;
        __syncthreads();
        const size_t base = (size_t)tile * kTile;
        for (int r = 0; r < kRadixItems; ++r) {
            const size_t e = base + (size_t)r * kRadixThreads + threadIdx.x;
            if (e < n) atomicAdd(&hist[(unsigned)((FIRST ? order_key(v[e]) : key[e]) >> shift) & 255u], 1u);
        }
        __syncthreads();
        counts[(size_t)threadIdx.x * ntile + tile] = hist[threadIdx.x];
    }
}

// block-wide exclusive scan of one value per thread (total in *total)
__device__ __forceinline__ unsigned block_excl_scan(unsigned v, unsigned *sh, unsigned *total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[warp] = x;
    __syncthreads();
    if (warp == 0) {
        unsigned w = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0u;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        sh[lane] = w;   // inclusive prefix over warps
    }
    __syncthreads();
    const unsigned before = warp ? sh[warp - 1] : 0u;
    *total = sh[(blockDim.x >> 5) - 1];
    __syncthreads();
    return before + x - v;
}

// The scans serve both paths: the buckets' unless the count was ended (k_scan_seg
// then adds up their squared counts), the radix sort's where it runs.
__device__ __forceinline__ bool scan_off(const GaussPlan *P, size_t n, bool buckets)
{
    return buckets ? P->bad != 0 : !use_radix(P, n);
}
// exclusive scan of each kScanSeg-long segment in place; segsum = its total
__global__ void __launch_bounds__(kScanThreads)
k_scan_seg(unsigned *__restrict__ a, size_t m, unsigned *__restrict__ segsum, GaussPlan *__restrict__ P, size_t n,
           bool buckets)
{
    __shared__ unsigned sh[32];
    if (scan_off(P, n, buckets)) return;
    const size_t base = (size_t)blockIdx.x * kScanSeg + (size_t)threadIdx.x * kScanItems;
    unsigned v[kScanItems], s = 0;
    unsigned long long sq = 0;
    for (int k = 0; k < kScanItems; ++k) {
        v[k] = base + k < m ? a[base + k] : 0u;
        s += v[k];
        sq += (unsigned long long)v[k] * v[k];
    }
    if (buckets) {
        for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
        if ((threadIdx.x & 31) == 0 && sq) atomicAdd(&P->squares, sq);
    }
    unsigned total;
    unsigned run = block_excl_scan(s, sh, &total);
    for (int k = 0; k < kScanItems; ++k) {
        if (base + k < m) a[base + k] = run;
        run += v[k];
    }
    if (threadIdx.x == 0) segsum[blockIdx.x] = total;
}

// exclusive scan of the segment totals (one block, any count)
__global__ void __launch_bounds__(kScanThreads)
k_scan_top(unsigned *__restrict__ segsum, int nseg, const GaussPlan *__restrict__ P, size_t n, bool buckets)
{
    __shared__ unsigned sh[32];
    if (scan_off(P, n, buckets)) return;
    unsigned carry = 0;
    for (int base = 0; base < nseg; base += kScanThreads) {
        const int i = base + threadIdx.x;
        const unsigned v = i < nseg ? segsum[i] : 0u;
        unsigned total;
        const unsigned ex = block_excl_scan(v, sh, &total);
        if (i < nseg) segsum[i] = carry + ex;
        carry += total;
    }
}

__global__ void __launch_bounds__(kScanThreads)
k_scan_add(unsigned *__restrict__ a, size_t m, const unsigned *__restrict__ segsum, const GaussPlan *__restrict__ P,
           size_t n, bool buckets)
{
    if (scan_off(P, n, buckets)) return;
    const size_t base = (size_t)blockIdx.x * kScanSeg + (size_t)threadIdx.x * kScanItems;
    const unsigned add = segsum[blockIdx.x];
    for (int k = 0; k < kScanItems; ++k)
        if (base + k < m) a[base + k] += add;
}

// The whole scan in one block, where that takes no longer than three launches
// (64^3: 16384 radix counts 9.7 us against 10.6; the buckets', once a call, pay up
// to 40960): a small field's time is its launches (8^3 with ties 250 us in 54,
// 176 us in 32)
constexpr size_t kScanOne[2] = {4 * kScanSeg, 10 * kScanSeg};   // radix, buckets
__global__ void __launch_bounds__(kScanThreads)
k_scan_one(unsigned *__restrict__ a, size_t m, GaussPlan *__restrict__ P, size_t n, bool buckets)
{
    __shared__ unsigned sh[32];
    if (scan_off(P, n, buckets)) return;
    unsigned carry = 0;
    unsigned long long sq = 0;
    for (size_t seg = 0; seg < m; seg += kScanSeg) {
        const size_t base = seg + (size_t)threadIdx.x * kScanItems;
        unsigned v[kScanItems], s = 0;
        for (int k = 0; k < kScanItems; ++k) {
            v[k] = base + k < m ? a[base + k] : 0u;
            s += v[k];
            sq += (unsigned long long)v[k] * v[k];
        }
        unsigned total;
        unsigned run = carry + block_excl_scan(s, sh, &total);
        for (int k = 0; k < kScanItems; ++k) {
            if (base + k < m) a[base + k] = run;
            run += v[k];
        }
        carry += total;
    }
    if (buckets) {
        for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
        if ((threadIdx.x & 31) == 0 && sq) atomicAdd(&P->squares, sq);
    }
}
// exclusive scan of m counts in place
void scan_counts(unsigned *a, size_t m, unsigned *segsum, GaussPlan *P, size_t n, bool buckets, cudaStream_t s)
{
    if (m <= kScanOne[buckets]) {
        note_launch();
        k_scan_one<<<1, kScanThreads, 0, s>>>(a, m, P, n, buckets);
        return;
    }
    const int nseg = (int)((m + kScanSeg - 1) / kScanSeg);
    note_launch(3);
    k_scan_seg<<<nseg, kScanThreads, 0, s>>>(a, m, segsum, P, n, buckets);
    k_scan_top<<<1, kScanThreads, 0, s>>>(segsum, nseg, P, n, buckets);
    k_scan_add<<<nseg, kScanThreads, 0, s>>>(a, m, segsum, P, n, buckets);
}

// stable scatter of one tile by the digit at `shift`; offs[d * ntile + tile]
// is where the tile's first element of digit d goes
template <bool FIRST>
__global__ void __launch_bounds__(kRadixThreads)
k_radix_scatter(const unsigned long long *__restrict__ kin, const unsigned *__restrict__ iin,
                const double *__restrict__ v, size_t n, int shift, int ntile, const unsigned *__restrict__ offs,
                unsigned long long *__restrict__ kout, unsigned *__restrict__ iout, const GaussPlan *__restrict__ P)
{
    if (!use_radix(P, n)) return;
    constexpr int kW = kRadixThreads / 32;
    __shared__ unsigned base[256], total[256];
    __shared__ unsigned wcnt[kW][256];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned lt = (1u << lane) - 1u;
    for (int it = blockIdx.x; it < ntile; it += gridDim.x) {
        __syncthreads();   // the previous tile's last reads of base
        base[tid] = offs[(size_t)tid * ntile + it];
        const size_t tile = (size_t)it * kTile;
        for (int r = 0; r < kRadixItems; ++r) {
            for (int w = 0; w < kW; ++w) wcnt[w][tid] = 0;
            const size_t e = tile + (size_t)r * kRadixThreads + tid;
            const bool valid = e < n;
            const unsigned long long k = !valid ? 0ull : (FIRST ? order_key(v[e]) : kin[e]);
            const unsigned d = valid ? ((unsigned)(k >> shift) & 255u) : 256u;
            const unsigned peers = __match_any_sync(0xffffffffu, d);
            const unsigned rank = __popc(peers & lt);
            __syncthreads();   // base / wcnt ready
            if (valid && rank == 0) wcnt[warp][d] = __popc(peers);
            __syncthreads();
            {   // per digit: exclusive prefix over the warps of this round
                unsigned run = 0;
                for (int w = 0; w < kW; ++w) {
                    const unsigned c = wcnt[w][tid];
                    wcnt[w][tid] = run;
                    run += c;
                }
                total[tid] = run;
            }
            __syncthreads();
            if (valid) {
                const unsigned pos = base[d] + wcnt[warp][d] + rank;
                kout[pos] = k;
                iout[pos] = FIRST ? (unsigned)e : iin[e];
            }
            __syncthreads();
            base[tid] += total[tid];
        }
    }
}

// g[idx[r]] = the quantile of rank r
__global__ void __launch_bounds__(kThreads)
k_gauss_out(const unsigned *__restrict__ idx, size_t n, const GaussPlan *__restrict__ P,
            const Anchor *__restrict__ anchors, double *__restrict__ g)
{
    if (!use_radix(P, n)) return;
    for (size_t r = (size_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (size_t)gridDim.x * blockDim.x)
        g[idx[r]] = quantile(r, n, P, anchors);
}

inline size_t bucket_slots(size_t n) { return n / 8 + 2 * kCells; }
inline size_t anchor_count(size_t n) { return n / (2 * kAnchor) + 1; }

cudaError_t gauss_alloc(recon_handle *H, size_t n)
{
    GaussWork &G = H->gauss;
    if (G.cap >= n) return cudaSuccess;
    gauss_free(H);
    const size_t ntile = (n + kTile - 1) / kTile, m = 256 * ntile > bucket_slots(n) ? 256 * ntile : bucket_slots(n);
    const size_t nseg = (m + kScanSeg - 1) / kScanSeg;
    // two key arrays and two index arrays, or the members and their places
    cudaError_t e = cudaMalloc(&G.pairs, 24 * n);
    if (e == cudaSuccess) e = cudaMalloc(&G.counts, sizeof(unsigned) * m);
    if (e == cudaSuccess) e = cudaMalloc(&G.segsum, sizeof(unsigned) * nseg);
    if (e == cudaSuccess) e = cudaMalloc(&G.anchors, sizeof(Anchor) * anchor_count(n));
    if (e == cudaSuccess) e = cudaMalloc(&G.plan, sizeof(GaussPlan));
    if (e != cudaSuccess) {
        gauss_free(H);
        return e;
    }
    G.cap = n;
    return cudaSuccess;
}

void gauss_free(recon_handle *H)
{
    GaussWork &G = H->gauss;
    if (G.pairs) cudaFree(G.pairs);
    if (G.counts) cudaFree(G.counts);
    if (G.segsum) cudaFree(G.segsum);
    if (G.anchors) cudaFree(G.anchors);
    if (G.plan) cudaFree(G.plan);
    G = GaussWork{};
}

cudaError_t gaussianise(recon_handle *H, const double *v, size_t n, double *g)
{
    cudaStream_t s = H->stream;
    CK(gauss_alloc(H, n));
    GaussWork &G = H->gauss;
    GaussPlan *P = static_cast<GaussPlan *>(G.plan);
    Anchor *anchors = static_cast<Anchor *>(G.anchors);
    const unsigned nb = stride_blocks(n) < (unsigned)kMaxRedBlocks ? stride_blocks(n) : (unsigned)kMaxRedBlocks;
    const unsigned sb = stride_blocks(n);
    // the map and the quantiles' anchors
    const size_t nanchor = anchor_count(n);
    const bool whole = n < 256 * (size_t)kSampleStep;   // small fields are counted in full
    const size_t step = whole ? kSampleRun : kSampleStep;
    const size_t sblocks = (n + step - 1) / step;
    note_launch(2);
    k_gauss_stats<<<nb, kThreads, 0, s>>>(v, n, H->partials, H->ticket, P);
    const unsigned sampling = (unsigned)(sblocks < 608 ? sblocks : 608);
    k_gauss_sample<<<sampling + (unsigned)((nanchor + kSampleRun - 1) / kSampleRun), kSampleRun, 0, s>>>(
        v, n, step, sampling, whole ? 1 : kSampleStep / kSampleRun, P, nanchor, anchors, H->ticket);
    // buckets
    Member *mem = static_cast<Member *>(G.pairs);
    uint2 *where = reinterpret_cast<uint2 *>(mem + n);
    const size_t slots = bucket_slots(n);
    CK(cudaMemsetAsync(G.counts, 0, sizeof(unsigned) * slots, s));
    note_launch(3);
    const unsigned most = (unsigned)std::sqrt((double)(kMaxWork / 16) * (double)n) + 1;
    k_gauss_count<<<sb, kThreads, 0, s>>>(v, n, P, G.counts, where, most);
    scan_counts(G.counts, slots, G.segsum, P, n, true, s);
    k_gauss_scatter<<<sb, kThreads, 0, s>>>(v, n, P, G.counts, where, mem);
    k_gauss_rank<<<sb, kThreads, 0, s>>>(mem, n, P, G.counts, anchors, g);
    // the radix sort, where the plan says so
    unsigned long long *key[2] = {static_cast<unsigned long long *>(G.pairs),
                                  static_cast<unsigned long long *>(G.pairs) + n};
    unsigned *idx[2] = {reinterpret_cast<unsigned *>(key[1] + n), reinterpret_cast<unsigned *>(key[1] + n) + n};
    const int ntile = (int)((n + kTile - 1) / kTile);
    const unsigned rb = ntile < 1216 ? ntile : 1216;
    const size_t m = 256 * (size_t)ntile;
    int cur = 0;
    for (int shift = 0; shift < 64; shift += 8) {
        note_launch(2);
        (shift ? k_radix_hist<false> : k_radix_hist<true>)<<<rb, kRadixThreads, 0, s>>>(key[cur], v, n, shift, ntile,
                                                                                   G.counts, P);
        scan_counts(G.counts, m, G.segsum, P, n, false, s);
        (shift ? k_radix_scatter<false> : k_radix_scatter<true>)<<<rb, kRadixThreads, 0, s>>>(
            key[cur], idx[cur], v, n, shift, ntile, G.counts, key[cur ^ 1], idx[cur ^ 1], P);
        cur ^= 1;
    }
    note_launch();
    k_gauss_out<<<nb, kThreads, 0, s>>>(idx[cur], n, P, anchors, g);
    return cudaGetLastError();
}

}  // namespace recon
