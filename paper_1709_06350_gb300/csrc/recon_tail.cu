// recon_tail.cu -- the small levels of a V-cycle in one thread-block cluster.
//
// From the first level that fits (tail_ok) down, the rest of a FAS V-cycle
// (Sec. II.A.3) or of a linear one runs in a single launch: the levels live in
// the shared memory of a cluster of kTailCtas thread blocks and every step of
// the multi-kernel cycle is a loop over cells between two barriers.
//
//  * A level whose side is at least dist_side<T>() is split into slabs of an
//    even number of planes, one slab per block; the smaller ones are held by
//    block 0, whose barriers are block barriers.  A coarse cell's children
//    are all in one slab.
//  * Stencil arrays of a split level carry one halo plane on each side.
//    Whoever stores a cell of a slab's first or last plane stores it into the
//    neighbour's halo as well (distributed shared memory), so all stencil
//    loads are local and one cluster barrier per step orders everything.
//  * The coarsest solve (Gauss-Seidel until the mean-free residual drops by
//    rtol, stops dropping, or a sweep cap) needs that residual after every
//    sweep.  A sweep's residual sums are taken by the pass that also relaxes
//    the red cells of the next one into another buffer, so a sweep costs two
//    barriers; if it was the last, the extra red pass is dropped.
//  * Sums are double-float (48 bits) for FP32 levels, FP64 for FP64 ones: an
//    FP64 addition holds a warp for 16 cycles of the SM's FP64 pipe, and the
//    block sums of the coarsest solve were most of its time.  The cycles of
//    mixed solves are bit for bit those with FP64 sums and a two-pass variance
//    (12 boxes, 64^3 to 448^3).
//  * The levels keep the arithmetic of the grid kernels (cell_update, det_IH;
//    jac_apply and the IEEE quotient of k_lin_pass) operation for operation: a
//    mixed solve's last digits follow the FP32 rounding of its cycles (1e-10 of
//    phi).  Paired instructions with an approximate reciprocal on the linear
//    levels, 2e-8 off in a correction's residual, were no faster (64^3 solve
//    1.68 ms either way; linear tail of 160^3 194 against 197 us).
//
// What bounds it: latency.  One pass over 32^3 takes ~3 us, one over 4^3 ~0.5;
// issue is active 11-12% of the time (160^3's tails, 20^3 and 10^3), and most
// stalls are at barriers, of the blocks and warps that wait for block 0's small
// levels.  16 blocks instead of 8 measured the same (32^3: 91 against 93 us
// per cycle) and a batch of solves slower.  Measured (GB300), against one
// thread block from 16^3 down and a dozen launches per level above it: mixed
// solves at 64^3 2.83 -> 1.77 ms, 160^3 (ends at 10^3) 8.78 -> 5.92 ms, FP64
// at 128^3 37.7 -> 31.8 ms; a 96^3 reconstruction 4.10 -> 2.87 ms.
#include <cooperative_groups.h>

#include "cellmath.cuh"
#include "dfloat.cuh"
#include "internal.cuh"

namespace cg = cooperative_groups;

namespace recon {
namespace {

constexpr int kMaxTail = 8;      // levels in a tail
constexpr int kTailCtas = 8;     // thread blocks of the cluster (the portable maximum)

// ---- sums in more than T's precision ---------------------------------------
__device__ __forceinline__ df acc_add(df a, df b) { return df_add(a, b); }
__device__ __forceinline__ double acc_add(double a, double b) { return a + b; }
__device__ __forceinline__ df acc_xor(df v, int o)
{
    return df_make(__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o));
}
__device__ __forceinline__ double acc_xor(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ df acc_lane(df v, int l)
{
    return df_make(__shfl_sync(0xffffffffu, v.hi, l), __shfl_sync(0xffffffffu, v.lo, l));
}
__device__ __forceinline__ double acc_lane(double v, int l) { return __shfl_sync(0xffffffffu, v, l); }

// V: the type of sums
template <typename T>
struct Math;
template <>
struct Math<float> {
    using V = df;
    static __host__ __device__ V of(double x) { return df_from_double(x); }
    static __device__ __forceinline__ V sum2(float a, float b)
    {
        df r;
        two_sum(a, b, r.hi, r.lo);
        return r;
    }
    static __device__ __forceinline__ V square(float x)
    {
        df r;
        two_prod(x, x, r.hi, r.lo);
        return r;
    }
    static __device__ __forceinline__ V mul(V a, V b) { return df_mul(a, b); }
    static __device__ __forceinline__ V sub(V a, V b) { return df_sub(a, b); }
    static __device__ __forceinline__ bool le(V a, V b) { return a.hi < b.hi || (a.hi == b.hi && a.lo <= b.lo); }
    static __device__ __forceinline__ float round(V a) { return a.hi; }
    static __device__ __forceinline__ double get(V a) { return (double)a.hi + (double)a.lo; }
};
template <>
struct Math<double> {
    using V = double;
    static __host__ __device__ V of(double x) { return x; }
    static __device__ __forceinline__ V sum2(double a, double b) { return a + b; }
    static __device__ __forceinline__ V square(double x) { return x * x; }
    static __device__ __forceinline__ V mul(V a, V b) { return a * b; }
    static __device__ __forceinline__ V sub(V a, V b) { return a - b; }
    static __device__ __forceinline__ bool le(V a, V b) { return a <= b; }
    static __device__ __forceinline__ double round(V a) { return a; }
    static __device__ __forceinline__ double get(V a) { return a; }
};

// the dynamic shared memory
template <typename T>
__device__ __forceinline__ T *smem()
{
    extern __shared__ __align__(16) unsigned char tail_smem[];
    return reinterpret_cast<T *>(tail_smem);
}

// ---- geometry ---------------------------------------------------------------
// slabs of a level of side N: number of blocks that hold one
__host__ __device__ inline int slab_blocks(int N, bool dist)
{
    const int pairs = N >> 1;
    return !dist ? 1 : (pairs < kTailCtas ? pairs : kTailCtas);
}
__host__ __device__ inline int first_pair(int N, int blocks, int r) { return r * (N >> 1) / blocks; }

template <typename T>
struct TailArgs {
    int nl;                     // levels in the tail (>= 1)
    int N[kMaxTail];
    int off[kMaxTail];          // first element of the level's arrays in shared memory
    int planes[kMaxTail];       // planes of a stencil array, halos included
    unsigned dist;              // bit l: level l is split over the cluster
    T ih2[kMaxTail], h2_6[kMaxTail];
    typename Math<T>::V rn[kMaxTail];   // 1 / cells
    T *t;                       // top level, global: theta (FAS) or e (linear), in and out
    const T *g;                 // top level, global: right side
    const float *cof[kMaxTail]; // linear: the colour-split cofactor arrays of every level
    const double *cptr;         // FAS: c of the top level (0 below)
    double *scal;               // FAS: the handle's device scalars; levels l0 .. are written
    int l0;
    int nu1, nu2, rule, cmax;
    T floor_;                   // FAS: scaled-defect floor (<= 0: off)
    typename Math<T>::V rtol2;  // coarsest solve: rtol^2 (0: fixed number of sweeps)
    int checked;                // rtol > 0
    int raw;                    // g is the restricted residual: FAS forms the right side from it,
                                // linear removes its mean
    int zero;                   // the iterate starts from 0 (t is not read)
};

// One level as a block sees it.
template <typename T>
struct Level {
    int l, N, NN, half;
    unsigned rN, rH;            // ceil(2^20 / .): exact quotients for indices below 2^13
    int blocks, first, np;      // blocks holding a slab; this block's first plane and plane count
    int npp;                    // planes of the slab below
    bool dist;
    int halo;                   // halo planes on each side: 1 if split, else 0 (planes wrap in place)
    int nth;                    // threads of a block that work on the level (a prefix)
    T *lo, *hi;                 // shared memory of the blocks holding the slabs below and above
};
// A cell row as stencils address it: offsets of its plane and the two beside
// it within an array, and of its row and the two beside it within a plane
struct Row {
    int c, m, p, r, rp, rm, ip;
};

template <typename T, int NT>
struct Tail {
    static constexpr int kW = NT / 32;
    using V = typename Math<T>::V;
    using M = Math<T>;
    struct Shared {
        V part[2][kTailCtas][kW][2];
        T pmin[2][kTailCtas][kW];
        double pscale[kMaxTail];
    };
    const TailArgs<T> &A;
    static __device__ __forceinline__ Shared &shared()
    {
        __shared__ Shared s;
        return s;
    }
    int rank, nctas, tid, lane, warp;
    int buf = 0;

    __device__ Tail(const TailArgs<T> &a) : A(a)
    {
        cg::cluster_group c = cg::this_cluster();
        rank = (int)c.block_rank();
        nctas = (int)c.num_blocks();
        tid = threadIdx.x;
        lane = tid & 31;
        warp = tid >> 5;
    }
    template <typename P>
    __device__ __forceinline__ P *at(P *p, int r) const { return cg::this_cluster().map_shared_rank(p, r); }
    __device__ __forceinline__ bool split(int l) const { return (A.dist >> l) & 1u; }
    // threads that work on level l: a block-held level takes one per pair of
    // cells, so the idle warps of the smallest levels stay off their barriers
    __device__ __forceinline__ int threads(int l) const
    {
        if (split(l)) return NT;
        const int N = A.N[l], t = (N * N * (N >> 1) + 31) & ~31;
        return t < NT ? t : NT;
    }
    __device__ __forceinline__ bool mine(int l) const { return split(l) || (rank == 0 && tid < threads(l)); }
    __device__ __forceinline__ void sync(const Level<T> &G) const
    {
        if (G.dist)
            cg::this_cluster().sync();
        else
            block_sync(G);
    }
    // barrier of the block's threads on the level (barrier 1 + level: the
    // threads above a smaller level's wait at their own level's barrier)
    __device__ __forceinline__ void block_sync(const Level<T> &G) const
    {
        if (G.nth == 32)
            __syncwarp();
        else
            asm volatile("bar.sync %0, %1;" ::"r"(1 + G.l), "r"(G.nth) : "memory");
    }

    __device__ Level<T> level(int l) const
    {
        Level<T> G;
        G.l = l;
        G.N = A.N[l];
        G.NN = G.N * G.N;
        G.half = G.N >> 1;
        G.rN = (1u << 20) / (unsigned)G.N + 1u;
        G.rH = (1u << 20) / (unsigned)G.half + 1u;
        G.dist = split(l);
        G.halo = G.dist ? 1 : 0;
        G.nth = threads(l);
        G.blocks = slab_blocks(G.N, G.dist);
        const int f = first_pair(G.N, G.blocks, rank);
        G.first = 2 * f;
        G.np = rank < G.blocks ? 2 * (first_pair(G.N, G.blocks, rank + 1) - f) : 0;
        const int below = rank == 0 ? G.blocks - 1 : rank - 1;
        const int above = rank + 1 >= G.blocks ? 0 : rank + 1;
        G.npp = 2 * (first_pair(G.N, G.blocks, below + 1) - first_pair(G.N, G.blocks, below));
        G.lo = at(smem<T>(), below < nctas ? below : 0);
        G.hi = at(smem<T>(), above);
        return G;
    }
    // arrays of a level, as element offsets: stencil arrays (with halos) first
    __device__ __forceinline__ int arr(const Level<T> &G, int x) const { return A.off[G.l] + x * A.planes[G.l] * G.NN; }
    // elements of an array without halos
    __device__ __forceinline__ int own(const Level<T> &G) const { return (A.planes[G.l] - 2 * G.halo) * G.NN; }

    // row j of local plane ip
    __device__ __forceinline__ Row row(const Level<T> &G, int ip, int j) const
    {
        Row w;
        w.ip = ip;
        w.c = (ip + G.halo) * G.NN;
        w.m = w.c - G.NN;
        w.p = w.c + G.NN;
        if (!G.dist) {
            if (ip == 0) w.m += G.np * G.NN;
            if (ip == G.np - 1) w.p = 0;
        }
        w.r = j * G.N;
        w.rp = w.r + G.N == G.NN ? 0 : w.r + G.N;
        w.rm = w.r == 0 ? G.NN - G.N : w.r - G.N;
        return w;
    }
    // store a cell and, in the first or last plane of a slab, into the neighbour's halo
    __device__ __forceinline__ void put(const Level<T> &G, int a, const Row &w, int o, T v) const
    {
        smem<T>()[a + w.c + o] = v;
        if (G.dist) {
            if (w.ip == 0) G.lo[a + (G.npp + 1) * G.NN + o] = v;
            if (w.ip == G.np - 1) G.hi[a + o] = v;
        }
    }
    // 19-point neighbourhood of cell k of a row in a stencil array
    __device__ __forceinline__ Nb19<T> nb(const Level<T> &G, int a, const Row &w, int k) const
    {
        const T *c = smem<T>() + a + w.c, *cm = smem<T>() + a + w.m, *cp = smem<T>() + a + w.p;
        const int kp = k + 1 == G.N ? 0 : k + 1, km = k == 0 ? G.N - 1 : k - 1;
        Nb19<T> v;
        v.c = c[w.r + k];
        v.xp = cp[w.r + k];
        v.xm = cm[w.r + k];
        v.yp = c[w.rp + k];
        v.ym = c[w.rm + k];
        v.zp = c[w.r + kp];
        v.zm = c[w.r + km];
        v.xpyp = cp[w.rp + k];
        v.xmym = cm[w.rm + k];
        v.xmyp = cm[w.rp + k];
        v.xpym = cp[w.rm + k];
        v.ypzp = c[w.rp + kp];
        v.ymzm = c[w.rm + km];
        v.ymzp = c[w.rm + kp];
        v.ypzm = c[w.rp + km];
        v.xpzp = cp[w.r + kp];
        v.xmzm = cm[w.r + km];
        v.xmzp = cm[w.r + kp];
        v.xpzm = cp[w.r + km];
        return v;
    }
    // the id-th pair of cells along k of this block's slab: its row and the k
    // of its red ((i + j + k) even; slabs start at an even plane) and black cell
    __device__ __forceinline__ Row pair(const Level<T> &G, int id, int &kr, int &kb) const
    {
        const int r = (int)(((unsigned)id * G.rH) >> 20), ip = (int)(((unsigned)r * G.rN) >> 20);
        const int m = id - r * G.half, j = r - ip * G.N, par = (ip + j) & 1;
        kr = 2 * m + par;
        kb = 2 * m + 1 - par;
        return row(G, ip, j);
    }
    __device__ __forceinline__ Row cell(const Level<T> &G, int id, int &k) const
    {
        const int r = (int)(((unsigned)id * G.rN) >> 20), ip = (int)(((unsigned)r * G.rN) >> 20);
        k = id - r * G.N;
        return row(G, ip, r - ip * G.N);
    }
    // f(a, b, first, second) over the indices below n, two per thread and
    // round (`first`, `second`: whether a and b are valid, else they repeat a
    // valid index).  Every thread of a working warp takes part, for the votes
    // of the paired update.
    template <class F>
    __device__ __forceinline__ void twos(const Level<T> &G, int n, F f) const
    {
        for (int base = 0; base + (tid & ~31) < n; base += 2 * G.nth) {
            const int a = base + tid, b = a + G.nth;
            f(a < n ? a : 0, b < n ? b : 0, a < n, b < n, base + (tid & ~31) + G.nth < n);
        }
    }
    // f(coarse plane I, J, K, fine local plane of the first child) over the
    // parents of this block's cells
    template <class F>
    __device__ __forceinline__ void parents(const Level<T> &G, F f) const
    {
        const int Nc = G.half, NcNc = Nc * Nc;
        for (int id = tid; id < (G.np >> 1) * NcNc; id += G.nth) {
            const int r = (int)(((unsigned)id * G.rH) >> 20), q = (int)(((unsigned)r * G.rH) >> 20);
            f((G.first >> 1) + q, r - q * Nc, id - r * Nc, 2 * q);
        }
    }
    // where plane I of level l lives
    struct Home {
        int r, lp, np, below, npp, above, halo;
    };
    __device__ __forceinline__ Home home(int l, int I) const
    {
        Home h;
        if (!split(l)) {
            h.r = h.below = h.above = h.halo = 0;
            h.lp = I;
            h.np = h.npp = A.N[l];
            return h;
        }
        const int N = A.N[l], B = slab_blocks(N, true), pr = I >> 1;
        h.r = ((pr + 1) * B - 1) / (N >> 1);
        const int f = first_pair(N, B, h.r);
        h.lp = I - 2 * f;
        h.np = 2 * (first_pair(N, B, h.r + 1) - f);
        h.below = h.r == 0 ? B - 1 : h.r - 1;
        h.npp = 2 * (first_pair(N, B, h.below + 1) - first_pair(N, B, h.below));
        h.above = h.r + 1 == B ? 0 : h.r + 1;
        h.halo = 1;
        return h;
    }
    __device__ __forceinline__ void put_home(const Home &h, int NN, int a, int o, T v) const
    {
        at(smem<T>(), h.r)[a + (h.lp + h.halo) * NN + o] = v;
        if (h.halo) {
            if (h.lp == 0) at(smem<T>(), h.below)[a + (h.npp + 1) * NN + o] = v;
            if (h.lp == h.np - 1) at(smem<T>(), h.above)[a + o] = v;
        }
    }

    // ---- reductions: push, a barrier, get (every thread).  Two sums at once:
    // the first exchange leaves one per half-warp.  The buffers alternate, so
    // a push only needs the previous get's barrier behind it.
    __device__ __forceinline__ void push(V a, V b, const Level<T> &G)
    {
        const bool second = lane & 16;
        V x = acc_add(second ? b : a, acc_xor(second ? a : b, 16));
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) x = acc_add(x, acc_xor(x, o));
        if (!G.dist) {
            if ((lane & 15) == 0) shared().part[buf][0][warp][second] = x;
        } else if ((lane & 15) < nctas) {
            at(&shared(), lane & 15)->part[buf][rank][warp][second] = x;
        }
    }
    // dist, nw: of the level that pushed
    __device__ __forceinline__ void get(V &a, V &b, bool dist, int nw)
    {
        V x = M::of(0.0);
        const int w = lane & 15;
        if (w < nw)
            for (int r = 0; r < (dist ? nctas : 1); ++r) x = acc_add(x, shared().part[buf][r][w][lane >> 4]);
        for (int o = nw > 8 ? 8 : (nw > 4 ? 4 : (nw > 1 ? 2 : 0)); o > 0; o >>= 1) x = acc_add(x, acc_xor(x, o));
        a = acc_lane(x, 0);
        b = acc_lane(x, 16);
        buf ^= 1;
    }
    __device__ __forceinline__ void push_min(T v, const Level<T> &G)
    {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const T u = __shfl_xor_sync(0xffffffffu, v, o);
            v = u < v ? u : v;
        }
        if (!G.dist) {
            if (lane == 0) shared().pmin[buf][0][warp] = v;
        } else if (lane < nctas) {
            at(&shared(), lane)->pmin[buf][rank][warp] = v;
        }
    }
    __device__ __forceinline__ T get_min(const Level<T> &G)
    {
        T v = T(INFINITY);
        if (lane < G.nth / 32)
            for (int r = 0; r < (G.dist ? nctas : 1); ++r) {
                const T u = shared().pmin[buf][r][lane];
                v = u < v ? u : v;
            }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const T u = __shfl_xor_sync(0xffffffffu, v, o);
            v = u < v ? u : v;
        }
        buf ^= 1;
        return v;
    }

    // global -> shared copy of n elements (a multiple of four), 16 bytes at a
    // time without waiting when the source is aligned; load_wait ends them
    __device__ __forceinline__ void copy_in(T *dst, const T *src, int n, int nth) const
    {
        constexpr int kE = 16 / (int)sizeof(T);
        if (((uintptr_t)src & 15) == 0) {
            const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
            for (int o = tid; o < n / kE; o += nth)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d + 16u * (unsigned)o),
                             "l"(src + o * kE));
        } else {
            for (int o = tid; o < n; o += nth) dst[o] = src[o];
        }
    }
    __device__ __forceinline__ void load_wait() const { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
    // the top level's arrays from global: with halos, and without
    __device__ void load_halo(const Level<T> &G, int a, const T *src) const
    {
        if (G.np == 0) return;
        const int lo = G.first == 0 ? G.N - 1 : G.first - 1, hi = G.first + G.np == G.N ? 0 : G.first + G.np;
        copy_in(smem<T>() + a + G.halo * G.NN, src + (size_t)G.first * G.NN, G.np * G.NN, G.nth);
        if (G.dist) {
            copy_in(smem<T>() + a, src + (size_t)lo * G.NN, G.NN, G.nth);
            copy_in(smem<T>() + a + (G.np + 1) * G.NN, src + (size_t)hi * G.NN, G.NN, G.nth);
        }
    }
    __device__ void load_own(const Level<T> &G, int a, const T *src) const
    {
        copy_in(smem<T>() + a, src + (size_t)G.first * G.NN, G.np * G.NN, G.nth);
    }
    __device__ void store_own(const Level<T> &G, int a, T *dst) const
    {
        for (int o = tid; o < G.np * G.NN; o += G.nth) dst[(size_t)G.first * G.NN + o] = smem<T>()[a + G.halo * G.NN + o];
    }
    // sum of an array without halos, to every working thread
    __device__ V total(const Level<T> &G, int a)
    {
        V s = M::of(0.0), z = s;
        for (int o = tid; o < G.np * G.NN; o += G.nth) s = acc_add(s, M::sum2(smem<T>()[a + o], T(0)));
        push(s, z, G);
        sync(G);
        get(s, z, G.dist, G.nth / 32);
        return s;
    }

    // fine += s P(cn - co): each parent of this block's cells (co < 0: P cn)
    __device__ void prolong(const Level<T> &G, int fine, int cn, int co, T s) const
    {
        const int Nc = G.half, NcNc = Nc * Nc;
        // rounded once: a quarter of `far` is exact
        auto mix = [](T near, T far) { return fma(T(0.75), near, T(0.25) * far); };
        parents(G, [&](int I, int J, int K, int fp) {
            const Home h = home(G.l + 1, I);
            const T *base = at(smem<T>(), h.r);
            const int P = h.lp + h.halo;
            const int Ip[3] = {(!h.halo && P == 0 ? Nc - 1 : P - 1) * NcNc, P * NcNc,
                               (!h.halo && P + 1 == Nc ? 0 : P + 1) * NcNc};
            const int Jp[3] = {(J == 0 ? Nc - 1 : J - 1) * Nc, J * Nc, (J + 1 == Nc ? 0 : J + 1) * Nc};
            const int Kp[3] = {K == 0 ? Nc - 1 : K - 1, K, K + 1 == Nc ? 0 : K + 1};
            T d[3][3][3];
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int b = 0; b < 3; ++b)
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        const int o = Ip[a] + Jp[b] + Kp[c];
                        d[a][b][c] = co >= 0 ? base[cn + o] - base[co + o] : base[cn + o];
                    }
#pragma unroll
            for (int ei = 0; ei < 2; ++ei) {
                T u[3][3];
#pragma unroll
                for (int b = 0; b < 3; ++b)
#pragma unroll
                    for (int c = 0; c < 3; ++c) u[b][c] = mix(d[1][b][c], d[ei ? 2 : 0][b][c]);
#pragma unroll
                for (int ej = 0; ej < 2; ++ej) {
                    T v[3];
#pragma unroll
                    for (int c = 0; c < 3; ++c) v[c] = mix(u[1][c], u[ej ? 2 : 0][c]);
                    Row w;
                    w.ip = fp + ei;
                    w.c = (w.ip + G.halo) * G.NN;
                    const int o = (2 * J + ej) * G.N + 2 * K;
                    const T *x = smem<T>() + fine + w.c + o;
                    const T x0 = x[0] + s * mix(v[1], v[0]), x1 = x[1] + s * mix(v[1], v[2]);
                    put(G, fine, w, o, x0);
                    put(G, fine, w, o + 1, x1);
                }
            }
        });
    }

    // The coarsest solve on stencil arrays a (the iterate), b, x (scratch).
    // both(src, row, kr, kb, rr, rb) returns the red cell's new value from src
    // and both cells' residuals; black(src, row, kb) the black cell's new
    // value.  Stops as described at the top of the file.
    template <class R, class B>
    __device__ void coarsest(const Level<T> &G, int a, int b, int x, R both, B black)
    {
        const int home_arr = a, n = G.np * G.N * G.half;
        V v0 = M::of(0.0), prev = v0;
        for (int s = 0;; ++s) {
            V s1 = M::of(0.0), s2 = s1;
            for (int base = 0; base + (tid & ~31) < n; base += G.nth) {
                const bool on = base + tid < n;
                int kr, kb;
                const Row w = pair(G, on ? base + tid : 0, kr, kb);
                T rr, rb;
                const T v = both(a, w, kr, kb, rr, rb);
                if (on) {
                    put(G, b, w, w.r + kr, v);
                    put(G, b, w, w.r + kb, smem<T>()[a + w.c + w.r + kb]);
                    s1 = acc_add(s1, M::sum2(rr, rb));
                    s2 = acc_add(s2, acc_add(M::square(rr), M::square(rb)));
                }
            }
            push(s1, s2, G);
            sync(G);
            get(s1, s2, G.dist, G.nth / 32);
            // n times the variance of the residual (the mean-free rms squared)
            V var = M::sub(s2, M::mul(M::mul(s1, s1), A.rn[G.l]));
            if (M::le(var, M::of(0.0))) var = M::of(0.0);
            if (s == 0)
                v0 = M::mul(var, A.rtol2);
            else if (M::le(var, v0) || (A.checked && M::le(prev, var)))
                break;   // reached, or no progress: the round-off floor
            if (s == A.cmax) break;
            prev = var;
            for (int base = 0; base + (tid & ~31) < n; base += G.nth) {
                const bool on = base + tid < n;
                int kr, kb;
                const Row w = pair(G, on ? base + tid : 0, kr, kb);
                const T v = black(b, w, kb);
                if (on) {
                    put(G, x, w, w.r + kb, v);
                    put(G, x, w, w.r + kr, smem<T>()[b + w.c + w.r + kr]);
                }
            }
            sync(G);
            const int t = a;
            a = x;
            x = t;
        }
        if (a != home_arr && G.np > 0)   // the halos travel with the planes
            for (int o = tid; o < (G.np + 2 * G.halo) * G.NN; o += G.nth) smem<T>()[home_arr + o] = smem<T>()[a + o];
        sync(G);
    }
};

// ---- FAS ---------------------------------------------------------------------
// arrays of a level: t, w, told (with halos), g (without), and on the coarsest
// level a third buffer (with halos)
template <typename T, int NT>
__global__ void __launch_bounds__(NT, 1) k_fas_tail(const __grid_constant__ TailArgs<T> A)
{
    using V = typename Math<T>::V;
    using M = Math<T>;
    Tail<T, NT> C(A);
    // right side of cell k of a row, without c (g has no halos)
    auto g_at = [&](const Level<T> &G, const Row &w, int k) { return smem<T>()[C.arr(G, 3) + w.ip * G.NN + w.r + k]; };
    auto update = [&](const Level<T> &G, int src, const Row &w, int k, T c) {
        return cell_update(C.nb(G, src, w, k), g_at(G, w, k) + c, A.ih2[G.l], A.h2_6[G.l], A.rule);
    };
    // snapshot red-black sweeps: t -> w (red), w -> t (black)
    auto sweeps = [&](const Level<T> &G, int count, T c) {
        const int t = C.arr(G, 0), w = C.arr(G, 1);
        for (int it = 0; it < 2 * count; ++it) {
            const bool black = it & 1;
            const int src = black ? w : t, dst = black ? t : w;
            C.twos(G, G.np * G.N * G.half, [&](int ia, int ib, bool ona, bool onb, bool two) {
                int ra, ba, rb, bb;
                const Row wa = C.pair(G, ia, ra, ba), wb = C.pair(G, ib, rb, bb);
                const int ka = black ? ba : ra, kb = black ? bb : rb, oa = black ? ra : ba, ob = black ? rb : bb;
                const T va = update(G, src, wa, ka, c), vb = two ? update(G, src, wb, kb, c) : va;
                if (ona) {
                    C.put(G, dst, wa, wa.r + ka, va);
                    C.put(G, dst, wa, wa.r + oa, smem<T>()[src + wa.c + wa.r + oa]);
                }
                if (onb) {
                    C.put(G, dst, wb, wb.r + kb, vb);
                    C.put(G, dst, wb, wb.r + ob, smem<T>()[src + wb.c + wb.r + ob]);
                }
            });
            C.sync(G);
        }
    };
    // f(row, k, det(I + H theta)) over this block's cells
    auto dets = [&](const Level<T> &G, auto f) {
        const int t = C.arr(G, 0);
        C.twos(G, G.np * G.NN, [&](int ia, int ib, bool ona, bool onb, bool two) {
            int ka, kb;
            const Row wa = C.cell(G, ia, ka), wb = C.cell(G, ib, kb);
            const T da = det_IH(C.nb(G, t, wa, ka), A.ih2[G.l]);
            const T db = two ? det_IH(C.nb(G, t, wb, kb), A.ih2[G.l]) : da;
            if (ona) f(wa, ka, da);
            if (onb) f(wb, kb, db);
        });
    };
    // the right side det(I + H R theta) + s (R r - mean R r) of a level from
    // its theta, R r in g and the sum of R r; s and 1 / s as in k_coarse_rhs
    auto form = [&](const Level<T> &G, V sum) {
        const int w = C.arr(G, 1), g = C.arr(G, 3);
        const V mean = M::mul(sum, A.rn[G.l]);
        const T m = M::round(mean), fl = A.floor_;
        T mn = T(INFINITY);
        dets(G, [&](const Row &x, int k, T d) {
            T &gc = smem<T>()[g + x.ip * G.NN + x.r + k];
            const T rr = gc - m;
            gc = rr;
            smem<T>()[w + x.c + x.r + k] = d;
            if (rr < T(0)) {
                const T cand = fl * (d > T(0) ? d : T(0)) / (-rr);
                mn = cand < mn ? cand : mn;
            }
        });
        C.push_min(mn, G);
        C.sync(G);
        mn = C.get_min(G);
        T s = fl <= T(0) ? T(1) : (mn < T(1) ? mn : T(1));
        if (s < T(1e-3)) s = T(0);
        if (C.rank == 0 && C.tid == 0) {
            const double ps = s > T(0) ? 1.0 / (double)s : 0.0;
            for (int r = 0; r < C.nctas; ++r) C.at(&C.shared(), r)->pscale[G.l] = ps;
            A.scal[slot_rmean(A.l0 + G.l)] = M::get(mean);
            A.scal[slot_scale(A.l0 + G.l)] = (double)s;
            A.scal[slot_pscale(A.l0 + G.l)] = ps;
        }
        // (every thread revisits the cells that it visited above)
        C.twos(G, G.np * G.NN, [&](int ia, int ib, bool ona, bool onb, bool) {
            if (ona) smem<T>()[g + ia] = smem<T>()[w + G.halo * G.NN + ia] + s * smem<T>()[g + ia];
            if (onb) smem<T>()[g + ib] = smem<T>()[w + G.halo * G.NN + ib] + s * smem<T>()[g + ib];
        });
        C.sync(G);
    };

    const int nl = A.nl;
    if (C.mine(0)) {
        const Level<T> G = C.level(0);
        C.load_halo(G, C.arr(G, 0), A.t);
        C.load_own(G, C.arr(G, 3), A.g);
        C.load_wait();
    }
    const T c0 = (T)(*A.cptr);
    cg::this_cluster().sync();   // loaded; every block's shared memory exists from here on
    if (A.raw && C.mine(0)) {
        const Level<T> G = C.level(0);
        form(G, C.total(G, C.arr(G, 3)));
    }
    // down: pre-smoothing, residual + restriction, the coarse right side
    for (int l = 0; l + 1 < nl; ++l) {
        if (!C.mine(l)) break;
        const Level<T> G = C.level(l);
        const T c = l == 0 ? c0 : T(0);
        sweeps(G, A.nu1, c);
        const int t = C.arr(G, 0), w = C.arr(G, 1), Nc = G.half, NcNc = Nc * Nc;
        const int tc = A.off[l + 1], oc = tc + 2 * A.planes[l + 1] * NcNc, gc = tc + 3 * A.planes[l + 1] * NcNc;
        // the residual of every cell (more threads than parents) into w, then the means of eight
        dets(G, [&](const Row &x, int k, T d) { smem<T>()[w + x.c + x.r + k] = (g_at(G, x, k) + c) - d; });
        C.block_sync(G);
        V sum = M::of(0.0), z = sum;
        C.parents(G, [&](int I, int J, int K, int fp) {
            T at = T(0), ar = T(0);
#pragma unroll
            for (int x = 0; x < 8; ++x) {
                const int o = (fp + (x >> 2) + G.halo) * G.NN + (2 * J + ((x >> 1) & 1)) * G.N + 2 * K + (x & 1);
                at += smem<T>()[t + o];
                ar += smem<T>()[w + o];
            }
            const T vt = at * T(0.125), vr = ar * T(0.125);
            const typename Tail<T, NT>::Home h = C.home(l + 1, I);
            const int o = J * Nc + K;
            C.put_home(h, NcNc, tc, o, vt);
            C.put_home(h, NcNc, oc, o, vt);
            C.at(smem<T>(), h.r)[gc + h.lp * NcNc + o] = vr;
            sum = acc_add(sum, M::sum2(vr, T(0)));
        });
        C.push(sum, z, G);
        C.sync(G);
        if (!C.mine(l + 1)) break;
        C.get(sum, z, G.dist, G.nth / 32);
        form(C.level(l + 1), sum);
    }
    if (C.mine(nl - 1)) {
        const Level<T> G = C.level(nl - 1);
        const T c = nl == 1 ? c0 : T(0);
        C.coarsest(
            G, C.arr(G, 0), C.arr(G, 1), C.arr(G, 3) + C.own(G),
            [&](int src, const Row &w, int kr, int kb, T &rr, T &rb) {
                rb = (g_at(G, w, kb) + c) - det_IH(C.nb(G, src, w, kb), A.ih2[G.l]);
                if constexpr (sizeof(T) == 8) {
                    return cell_update(C.nb(G, src, w, kr), g_at(G, w, kr) + c, A.ih2[G.l], A.h2_6[G.l], A.rule, &rr);
                } else {
                    rr = (g_at(G, w, kr) + c) - det_IH(C.nb(G, src, w, kr), A.ih2[G.l]);
                    // (loaded again: shared products would round differently than in cell_update alone)
                    asm volatile("" ::: "memory");
                    return update(G, src, w, kr, c);
                }
            },
            [&](int src, const Row &w, int kb) { return update(G, src, w, kb, c); });
    }
    // up: the corrections and post-smoothing
    for (int l = nl - 2; l >= 0; --l) {
        if (!C.mine(l)) continue;
        const Level<T> G = C.level(l);
        if (G.dist != C.split(l + 1) || G.nth != C.threads(l + 1)) C.sync(G);   // the level below is done
        const double ps = C.shared().pscale[l + 1];
        if (ps != 0.0)
            C.prolong(G, C.arr(G, 0), A.off[l + 1], A.off[l + 1] + 2 * A.planes[l + 1] * G.half * G.half, (T)ps);
        C.sync(G);
        sweeps(G, A.nu2, l == 0 ? c0 : T(0));
    }
    if (C.mine(0)) {
        const Level<T> G = C.level(0);
        C.store_own(G, C.arr(G, 0), A.t);
    }
}

// ---- linear: J e = f with stored cofactors ---------------------------------
// arrays of a level: e, w (with halos), f and the six cofactor fields
// (without), and on the coarsest level a third buffer (with halos)
template <int NT>
__global__ void __launch_bounds__(NT, 1) k_lin_tail(const __grid_constant__ TailArgs<float> A)
{
    using L = Level<float>;
    Tail<float, NT> C(A);
    auto f_at = [&](const L &G, const Row &w, int k) { return smem<float>()[C.arr(G, 2) + w.ip * G.NN + w.r + k]; };
    // cofactors of cell k of a row; their rows are colour split: (i + j + k) even first
    auto cof_at = [&](const L &G, const Row &w, int k) {
        const int n = C.own(G), j = (int)(((unsigned)w.r * G.rN) >> 20);
        const float *c = smem<float>() + C.arr(G, 2) + n + w.ip * G.NN + w.r + (((w.ip + j + k) & 1) ? G.half : 0) + (k >> 1);
        Cof<float> a;
        a.xx = c[0];
        a.yy = c[n];
        a.zz = c[2 * n];
        a.xy = c[3 * n];
        a.yz = c[4 * n];
        a.xz = c[5 * n];
        return a;
    };
    // a cell's residual f - J e, and its new value
    auto residual = [&](const L &G, int src, const Row &w, int k) {
        return f_at(G, w, k) - jac_apply(cof_at(G, w, k), C.nb(G, src, w, k), A.ih2[G.l]);
    };
    auto update = [&](const L &G, int src, const Row &w, int k, float &r) {
        const Cof<float> a = cof_at(G, w, k);
        const Nb19<float> n = C.nb(G, src, w, k);
        r = f_at(G, w, k) - jac_apply(a, n, A.ih2[G.l]);
        return n.c + r / (-2.0f * (a.xx + a.yy + a.zz) * A.ih2[G.l]);
    };
    auto sweeps = [&](const L &G, int count) {
        const int e = C.arr(G, 0), w = C.arr(G, 1);
        for (int it = 0; it < 2 * count; ++it) {
            const bool black = it & 1;
            const int src = black ? w : e, dst = black ? e : w;
            C.twos(G, G.np * G.N * G.half, [&](int ia, int ib, bool ona, bool onb, bool two) {
                int ra, ba, rb, bb;
                const Row wa = C.pair(G, ia, ra, ba), wb = C.pair(G, ib, rb, bb);
                const int ka = black ? ba : ra, kb = black ? bb : rb, oa = black ? ra : ba, ob = black ? rb : bb;
                float r;
                const float va = update(G, src, wa, ka, r), vb = two ? update(G, src, wb, kb, r) : va;
                if (ona) {
                    C.put(G, dst, wa, wa.r + ka, va);
                    C.put(G, dst, wa, wa.r + oa, smem<float>()[src + wa.c + wa.r + oa]);
                }
                if (onb) {
                    C.put(G, dst, wb, wb.r + kb, vb);
                    C.put(G, dst, wb, wb.r + ob, smem<float>()[src + wb.c + wb.r + ob]);
                }
            });
            C.sync(G);
        }
    };
    // f -= mean f, from the sum of f
    auto centre = [&](const L &G, df sum) {
        const float m = df_mul(sum, A.rn[G.l]).hi;
        for (int o = C.tid; o < G.np * G.NN; o += G.nth) smem<float>()[C.arr(G, 2) + o] -= m;
        C.sync(G);
    };

    const int nl = A.nl;
    for (int l = 0; l < nl; ++l) {
        if (!C.mine(l)) break;
        const L G = C.level(l);
        const size_t n = (size_t)G.N * G.NN;
        if (l == 0) C.load_own(G, C.arr(G, 2), A.g);
        for (int x = 0; x < 6; ++x) C.load_own(G, C.arr(G, 2) + (1 + x) * C.own(G), A.cof[l] + x * n);
        if (l > 0 || A.zero)
            for (int o = C.tid; o < A.planes[l] * G.NN; o += G.nth) smem<float>()[C.arr(G, 0) + o] = 0.0f;
        else
            C.load_halo(G, C.arr(G, 0), A.t);
    }
    C.load_wait();
    cg::this_cluster().sync();   // loaded; every block's shared memory exists from here on
    if (A.raw && C.mine(0)) {
        const L G = C.level(0);
        centre(G, C.total(G, C.arr(G, 2)));
    }
    for (int l = 0; l + 1 < nl; ++l) {
        if (!C.mine(l)) break;
        const L G = C.level(l);
        sweeps(G, A.nu1);
        const int e = C.arr(G, 0), w = C.arr(G, 1), Nc = G.half, NcNc = Nc * Nc;
        const int fc = A.off[l + 1] + 2 * A.planes[l + 1] * NcNc;
        // the residual of every cell into w, then the means of eight
        C.twos(G, G.np * G.NN, [&](int ia, int ib, bool ona, bool onb, bool two) {
            int ka, kb;
            const Row wa = C.cell(G, ia, ka), wb = C.cell(G, ib, kb);
            const float ra = residual(G, e, wa, ka), rb = two ? residual(G, e, wb, kb) : ra;
            if (ona) smem<float>()[w + wa.c + wa.r + ka] = ra;
            if (onb) smem<float>()[w + wb.c + wb.r + kb] = rb;
        });
        C.block_sync(G);
        df sum = df_make(0.0f, 0.0f), z = sum;
        C.parents(G, [&](int I, int J, int K, int fp) {
            float acc = 0.0f;
#pragma unroll
            for (int x = 0; x < 8; ++x)
                acc += smem<float>()[w + (fp + (x >> 2) + G.halo) * G.NN + (2 * J + ((x >> 1) & 1)) * G.N + 2 * K + (x & 1)];
            const float v = acc * 0.125f;
            const typename Tail<float, NT>::Home h = C.home(l + 1, I);
            C.at(smem<float>(), h.r)[fc + h.lp * NcNc + J * Nc + K] = v;
            sum = df_add(sum, df_make(v, 0.0f));
        });
        C.push(sum, z, G);
        C.sync(G);
        if (!C.mine(l + 1)) break;
        C.get(sum, z, G.dist, G.nth / 32);
        centre(C.level(l + 1), sum);
    }
    if (C.mine(nl - 1)) {
        const L G = C.level(nl - 1);
        C.coarsest(
            G, C.arr(G, 0), C.arr(G, 1), C.arr(G, 2) + 7 * C.own(G),
            [&](int src, const Row &w, int kr, int kb, float &rr, float &rb) {
                rb = residual(G, src, w, kb);
                return update(G, src, w, kr, rr);
            },
            [&](int src, const Row &w, int kb) {
                float r;
                return update(G, src, w, kb, r);
            });
    }
    for (int l = nl - 2; l >= 0; --l) {
        if (!C.mine(l)) continue;
        const L G = C.level(l);
        if (G.dist != C.split(l + 1) || G.nth != C.threads(l + 1)) C.sync(G);   // the level below is done
        C.prolong(G, C.arr(G, 0), A.off[l + 1], -1, 1.0f);
        C.sync(G);
        sweeps(G, A.nu2);
    }
    if (C.mine(0)) {
        const L G = C.level(0);
        C.store_own(G, C.arr(G, 0), A.t);
    }
}

// ---- launch ------------------------------------------------------------------
// Levels of at least this side are split over the cluster.  FP32: below 12^3
// a pass on one SM takes no longer than a cluster barrier.  FP64: one SM retires
// two FP64 operations a cycle, so 8^3 is already worth splitting.
template <typename T>
constexpr int dist_side() { return sizeof(T) == 8 ? 8 : 12; }
template <typename T>
constexpr int tail_threads() { return sizeof(T) == 8 ? 256 : 512; }

// fills off, planes, dist; returns the shared memory in bytes
template <typename T>
size_t place(TailArgs<T> &A, bool lin)
{
    size_t c = 0;
    A.dist = 0;
    for (int l = 0; l < A.nl; ++l) {
        const int N = A.N[l];
        const bool dist = N >= dist_side<T>();
        const int B = slab_blocks(N, dist), np = 2 * ((N / 2 + B - 1) / B);
        if (dist) A.dist |= 1u << l;
        const int rows = np + (dist ? 2 : 0);   // halos only between blocks
        A.planes[l] = rows;
        A.rn[l] = Math<T>::of(1.0 / ((double)N * N * N));
        A.off[l] = (int)c;
        const size_t halo = (size_t)rows * N * N, own = (size_t)np * N * N;
        c += lin ? 2 * halo + 7 * own : 3 * halo + own;
        if (l == A.nl - 1) c += halo;
    }
    return c * sizeof(T);
}

// dynamic shared memory: the linear tail of 32^3 and below takes 207360 bytes,
// the most of any side; the static part stays below 6 KB
constexpr int kTailSmem = 208 * 1024;

template <typename T>
cudaError_t launch(void (*kern)(TailArgs<T>), const TailArgs<T> &A, size_t smem, int threads, cudaStream_t s)
{
    if (smem > (size_t)kTailSmem) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    const unsigned n = A.dist ? kTailCtas : 1;
    cfg.gridDim = dim3(n);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = n;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    note_launch();
    return cudaLaunchKernelEx(&cfg, kern, A);
}

}  // namespace

// A level starts a tail when it has at most this many cells: 32^3 for FP32
// (the linear tail's arrays of 32^3 and below fill each block's memory);
// 16^3 for FP64, whose larger levels need more SMs for their FP64 rate.
template <typename T>
bool tail_ok(int N)
{
    const size_t cells = sizeof(T) == 8 ? 16 * 16 * 16 : 32 * 32 * 32;
    return (size_t)N * N * N <= cells;
}
template bool tail_ok<float>(int);
template bool tail_ok<double>(int);

template <typename T>
cudaError_t fas_tail(recon_handle *H, int l, T *t, const T *g, const double *cptr, bool raw)
{
    const recon_config &cf = H->cfg;
    TailArgs<T> A{};
    A.nl = H->nlev - l;
    if (A.nl > kMaxTail) return cudaErrorInvalidValue;
    for (int q = 0; q < A.nl; ++q) {
        A.N[q] = H->Nl[l + q];
        const double h = H->hl[l + q];
        A.ih2[q] = (T)(1.0 / (h * h));
        A.h2_6[q] = (T)(h * h / 6.0);
    }
    A.t = t;
    A.g = g;
    A.cptr = cptr;
    A.scal = H->scal;
    A.l0 = l;
    A.nu1 = cf.nu1;
    A.nu2 = cf.nu2;
    A.rule = cf.rule;
    A.cmax = cf.coarse_max_sweeps;
    A.floor_ = (T)cf.scale_floor;
    A.rtol2 = Math<T>::of(cf.coarse_rtol * cf.coarse_rtol);
    A.checked = cf.coarse_rtol > 0.0;
    A.raw = raw;
    const size_t smem = place(A, false);
    return launch<T>(k_fas_tail<T, tail_threads<T>()>, A, smem, tail_threads<T>(), H->stream);
}
template cudaError_t fas_tail<float>(recon_handle *, int, float *, const float *, const double *, bool);
template cudaError_t fas_tail<double>(recon_handle *, int, double *, const double *, const double *, bool);

cudaError_t lin_tail(recon_handle *H, int l, float *e, const float *f, const float *const *cof, bool raw, bool zero)
{
    const recon_config &cf = H->cfg;
    TailArgs<float> A{};
    A.nl = H->nlev - l;
    if (A.nl > kMaxTail) return cudaErrorInvalidValue;
    for (int q = 0; q < A.nl; ++q) {
        A.N[q] = H->Nl[l + q];
        const double h = H->hl[l + q];
        A.ih2[q] = (float)(1.0 / (h * h));
        A.cof[q] = cof[l + q];
    }
    A.t = e;
    A.g = f;
    A.nu1 = cf.nu1;
    A.nu2 = cf.nu2;
    A.cmax = cf.coarse_max_sweeps;
    A.rtol2 = Math<float>::of(cf.coarse_rtol * cf.coarse_rtol);
    A.checked = cf.coarse_rtol > 0.0;
    A.raw = raw;
    A.zero = zero;
    const size_t smem = place(A, true);
    return launch<float>(k_lin_tail<tail_threads<float>()>, A, smem, tail_threads<float>(), H->stream);
}

cudaError_t prepare_tails()
{
    cudaError_t e = cudaFuncSetAttribute(k_fas_tail<float, tail_threads<float>()>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, kTailSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_fas_tail<double, tail_threads<double>()>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, kTailSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_lin_tail<tail_threads<float>()>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kTailSmem);
    return e;
}

}  // namespace recon
