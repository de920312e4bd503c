// recon_adjoint.cu -- adjoint of the solve (implicit-function theorem).
//
// The solve defines phi(b) through F(phi, c; b) = det(I + H phi) - c - b = 0
// with mean(phi) = 0.  With J = dF/dphi = sum_ab adj(I+H)_ab D_ab (stencils
// of eq. discrete_examples) the gradient of a loss with respect to b is the
// lam of
//     J^T lam + mu 1 = gbar,   sum(lam) = 0,
// with J^T lam = sum_ab D_ab (adj_ab * lam) (the D_ab are symmetric).  J 1 = 0
// makes range(J^T) the mean-free fields, so mu = mean(gbar); J^T has one null
// vector n = 1 + w (J^T w = -J^T 1), and lam = lam0 - (sum lam0 / sum n) n for
// any solution lam0 of J^T lam0 = gbar - mean(gbar).
//
// Both linear solves correct an FP64 residual by FP32 red-black Gauss-Seidel
// multigrid on J^T (jt_solve_mixed), with FP64 multigrid behind it where that
// stops short.  The coarse levels' cofactors are computed once per solve from
// the restricted potential and kept; the finest level's are formed again from
// phi in every application of J^T (k_jt_fine) unless adjoint_store_cofactors
// keeps them too (48 N^3 bytes in FP64, 24 in FP32).
#include <cmath>
#include <string>

#include "cellmath.cuh"
#include "internal.cuh"

namespace recon {

namespace {

constexpr int kRT = kRowX * kRowY;

template <typename T>
struct CofPtr {
    const T *xx, *yy, *zz, *xy, *yz, *xz;
};
template <typename T>
__host__ __device__ inline CofPtr<T> cof_of(const T *base, size_t n)
{
    return {base, base + n, base + 2 * n, base + 3 * n, base + 4 * n, base + 5 * n};
}

template <typename T>
__global__ void __launch_bounds__(kRT)
k_cof6(const T *__restrict__ th, int N, T ih2, T *__restrict__ cof)
{
    const size_t n = (size_t)N * N * N;
    FOR_ROWS(N, i, j)
    for (int k = threadIdx.x; k < N; k += kRowX) {
        const Cof<T> a = cofactors(load19<T>(th, N, i, j, k), ih2);
        const unsigned id = offs(N, i, j, k);
        cof[id] = a.xx;
        cof[n + id] = a.yy;
        cof[2 * n + id] = a.zz;
        cof[3 * n + id] = a.xy;
        cof[4 * n + id] = a.yz;
        cof[5 * n + id] = a.xz;
    }
}

// (J^T lam) at (i, j, k) and the diagonal of J^T there.
template <typename T>
__device__ __forceinline__ T jt_at(const CofPtr<T> C, const T *lam, int N, int i, int j, int k, T ih2, T *diag)
{
    const int ip = wp(i, N), im = wm(i, N), jp = wp(j, N), jm = wm(j, N), kp = wp(k, N), km = wm(k, N);
    auto L = [&](int a, int b, int c) { return lam[offs(N, a, b, c)]; };
    auto X = [&](const T *cc, int a, int b, int c) {
        const unsigned o = offs(N, a, b, c);
        return cc[o] * lam[o];
    };
    const unsigned o = offs(N, i, j, k);
    const T dxx = X(C.xx, ip, j, k) + X(C.xx, im, j, k) - T(2) * C.xx[o] * L(i, j, k);
    const T dyy = X(C.yy, i, jp, k) + X(C.yy, i, jm, k) - T(2) * C.yy[o] * L(i, j, k);
    const T dzz = X(C.zz, i, j, kp) + X(C.zz, i, j, km) - T(2) * C.zz[o] * L(i, j, k);
    const T dxy = (X(C.xy, ip, jp, k) + X(C.xy, im, jm, k)) - (X(C.xy, im, jp, k) + X(C.xy, ip, jm, k));
    const T dyz = (X(C.yz, i, jp, kp) + X(C.yz, i, jm, km)) - (X(C.yz, i, jm, kp) + X(C.yz, i, jp, km));
    const T dxz = (X(C.xz, ip, j, kp) + X(C.xz, im, j, km)) - (X(C.xz, im, j, kp) + X(C.xz, ip, j, km));
    if (diag) *diag = T(-2) * (C.xx[o] + C.yy[o] + C.zz[o]) * ih2;
    return (dxx + dyy + dzz) * ih2 + (dxy + dyz + dxz) * (T(0.5) * ih2);
}

// one colour pass of Gauss-Seidel on J^T lam = f (snapshot semantics)
template <typename T>
__global__ void __launch_bounds__(kRT)
k_jt_pass(const T *__restrict__ src, T *__restrict__ dst, const T *__restrict__ f, const T *__restrict__ cof, int N,
          T ih2, int colour)
{
    const CofPtr<T> C = cof_of(cof, (size_t)N * N * N);
    const int half = N >> 1;
    FOR_ROWS(N, i, j)
    {
        const int par = (colour + i + j) & 1;
        const unsigned base = offs(N, i, j, 0);
        for (int m = threadIdx.x; m < half; m += blockDim.x) {
            const int ka = 2 * m + par, kb = 2 * m + 1 - par;
            T d;
            const T jt = jt_at<T>(C, src, N, i, j, ka, ih2, &d);
            dst[base + ka] = src[base + ka] + (f[base + ka] - jt) / d;
            dst[base + kb] = src[base + kb];
        }
    }
}

// fH = R(f - J^T lam) (8-son mean) and block partial sums of it
template <typename T>
__global__ void __launch_bounds__(kRT)
k_jt_restrict_residual(const T *__restrict__ lam, const T *__restrict__ f, const T *__restrict__ cof, int Nf, T ih2,
                       T *__restrict__ fH, double *__restrict__ partials)
{
    __shared__ double sh[32];
    const CofPtr<T> C = cof_of(cof, (size_t)Nf * Nf * Nf);
    const int Nc = Nf >> 1;
    ThreadSum<T> s;
    FOR_ROWS(Nc, I, J)
    for (int K = threadIdx.x; K < Nc; K += kRowX) {
        T acc = T(0);
        for (int a = 0; a < 2; ++a)
            for (int b = 0; b < 2; ++b)
                for (int cc = 0; cc < 2; ++cc) {
                    const int i = 2 * I + a, j = 2 * J + b, k = 2 * K + cc;
                    acc += f[offs(Nf, i, j, k)] - jt_at<T>(C, lam, Nf, i, j, k, ih2, nullptr);
                }
        const T v = acc * T(0.125);
        fH[offs(Nc, I, J, K)] = v;
        s.add(v);
    }
    const double v = block_sum<kRT>(s.get(), sh);
    if (ltid() == 0) partials[4 * blockIdx.x + 0] = v;
}

// out = sign * J^T v (v == nullptr: v = 1); partial sums of out^2 (col 1),
// or of (f - out)^2 when f is given (col 1 then holds the residual norm, and
// rout, if given, gets scale (f - out) as floats)
__global__ void __launch_bounds__(kRT)
k_jt_apply(const double *__restrict__ v, const double *__restrict__ f, const double *__restrict__ cof,
           int N, double ih2, double sign, double *__restrict__ out, double *__restrict__ partials,
           float *__restrict__ rout, double scale)
{
    __shared__ double sh[32];
    const CofPtr<double> C = cof_of(cof, (size_t)N * N * N);
    double s2 = 0.0;
    FOR_ROWS(N, i, j)
    for (int k = threadIdx.x; k < N; k += kRowX) {
        double r;
        if (v) {
            r = sign * jt_at<double>(C, v, N, i, j, k, ih2, nullptr);
        } else {
            // J^T 1 = sum_ab D_ab adj_ab
            const int ip = wp(i, N), im = wm(i, N), jp = wp(j, N), jm = wm(j, N), kp = wp(k, N), km = wm(k, N);
            auto c = [&](const double *a, int x, int y, int z) { return a[offs(N, x, y, z)]; };
            const unsigned o = offs(N, i, j, k);
            const double d = (c(C.xx, ip, j, k) + c(C.xx, im, j, k) - 2.0 * C.xx[o]) +
                             (c(C.yy, i, jp, k) + c(C.yy, i, jm, k) - 2.0 * C.yy[o]) +
                             (c(C.zz, i, j, kp) + c(C.zz, i, j, km) - 2.0 * C.zz[o]);
            const double m = ((c(C.xy, ip, jp, k) + c(C.xy, im, jm, k)) - (c(C.xy, im, jp, k) + c(C.xy, ip, jm, k))) +
                             ((c(C.yz, i, jp, kp) + c(C.yz, i, jm, km)) - (c(C.yz, i, jm, kp) + c(C.yz, i, jp, km))) +
                             ((c(C.xz, ip, j, kp) + c(C.xz, im, j, km)) - (c(C.xz, im, j, kp) + c(C.xz, ip, j, km)));
            r = sign * (d * ih2 + m * (0.5 * ih2));
        }
        const unsigned id = offs(N, i, j, k);
        if (f) {
            const double e = f[id] - r;
            if (rout) rout[id] = (float)(e * scale);
            s2 += e * e;
        } else {
            out[id] = r;
            s2 += r * r;
        }
    }
    const double t = block_sum<kRT>(s2, sh);
    if (ltid() == 0) partials[4 * blockIdx.x + 1] = t;
}

// ---- the finest level without stored cofactors ----------------------------
// J^T applied with the cofactors of I + H phi formed in shared memory: a CTA
// streams chunks of fine_chunk(N) planes of the i columns of 8 x 32 (j, k)
// tiles (work items taken in turn by the CTAs of a grid of at most
// kMaxRedBlocks); per plane p it stages phi (tile + 2-cell halo) and lam
// (tile + 1), forms the six cofactors of plane p + 1 on the tile + 1 ring, and
// applies J^T at plane p.  Three barriers per plane; no N^3 cofactor arrays.
// FP64 is bound by the FP64 pipe: MODE 1 stores the products adj_ab lam,
// formed once per ring cell instead of at each of their uses (~85 FP64
// operations per cell with the ring and the chunk's first planes, ~110
// before), and the chunk is short enough for several CTAs per SM: 128^3 540 ->
// 464 us (its operations: ~360).  FP32 is bound by latency between barriers
// (128^3: 60 us a colour pass, 174 with 64-plane chunks).
//   MODE 0: one colour pass of Gauss-Seidel on J^T lam = f (snapshot: out is
//           the destination array, cells of the other colour copied)
//   MODE 1: r = f - J^T lam in out, scale r as floats in rout (each if given)
//           and per-CTA sums (partials column 1) of r^2 for FP64, of r for FP32
//   MODE 2: out = sign * J^T 1 and per-CTA sums of out^2 (column 1)
constexpr int kFJ = 8, kFK = 32, kFT = kFJ * kFK;
constexpr int kMinItems = 512;
constexpr int kFPK = kFK + 4, kFPP = (kFJ + 4) * kFPK;   // phi planes
constexpr int kFCK = kFK + 2, kFCP = (kFJ + 2) * kFCK;   // cofactor / lam planes
// planes per work item: long chunks form fewer cofactors twice (two planes per
// chunk), short ones fill the SMs evenly
__host__ __device__ inline int fine_chunk(int N)
{
    int ci = N < 64 ? N : 64;
    while (ci > 16 && (N / kFK) * (N / kFJ) * (N / ci) < kMinItems && ci % 2 == 0 && N % (ci / 2) == 0) ci /= 2;
    return ci;
}
template <typename T>
constexpr size_t fine_smem() { return sizeof(T) * (5 * kFPP + 3 * 6 * kFCP + 3 * kFCP); }

template <int MODE, typename T>
__global__ void __launch_bounds__(kFT)
k_jt_fine(const T *__restrict__ phi, const T *__restrict__ lam, const T *__restrict__ f, T *__restrict__ out, int N,
          T ih2, int colour, T sign, double *__restrict__ partials, float *__restrict__ rout, T scale)
{
    extern __shared__ __align__(16) unsigned char smd[];
    T *sphi = reinterpret_cast<T *>(smd);     // [5][kFPP]
    T *scof = sphi + 5 * kFPP;                // [3][6][kFCP]
    T *slam = scof + 3 * 6 * kFCP;            // [3][kFCP]
    __shared__ double sh[32];
    const int tid = threadIdx.x, tj = tid / kFK, tk = tid % kFK;
    const unsigned NN = (unsigned)N * (unsigned)N;
    const int ncols = (N / kFK) * (N / kFJ), CI = fine_chunk(N), nchunks = N / CI;
    auto wr = [&](int x) { return x < 0 ? x + N : (x >= N ? x - N : x); };
    ThreadSum<T> s2;
    for (int item = blockIdx.x; item < ncols * nchunks; item += gridDim.x) {
        const int col = item % ncols, i0 = (item / ncols) * CI, i1 = i0 + CI;
        const int k0 = (col % (N / kFK)) * kFK, j0 = (col / (N / kFK)) * kFJ;
        auto load_phi = [&](int p) {
            T *d = sphi + ((p + 10) % 5) * kFPP;
            const unsigned pb = (unsigned)wr(p) * NN;
            for (int e = tid; e < kFPP; e += kFT) {
                const int r = e / kFPK, c = e - r * kFPK;
                d[e] = phi[pb + (unsigned)wr(j0 - 2 + r) * (unsigned)N + (unsigned)wr(k0 - 2 + c)];
            }
        };
        auto load_lam = [&](int p) {
            if (MODE == 2) return;
            T *d = slam + ((p + 9) % 3) * kFCP;
            const unsigned pb = (unsigned)wr(p) * NN;
            for (int e = tid; e < kFCP; e += kFT) {
                const int r = e / kFCK, c = e - r * kFCK;
                d[e] = lam[pb + (unsigned)wr(j0 - 1 + r) * (unsigned)N + (unsigned)wr(k0 - 1 + c)];
            }
        };
        auto cof_plane = [&](int p) {   // cofactors of plane p on the tile + 1 ring (phi planes p-1..p+1 staged)
            const T *pm = sphi + ((p + 9) % 5) * kFPP, *pc = sphi + ((p + 10) % 5) * kFPP,
                         *pp = sphi + ((p + 11) % 5) * kFPP;
            T *d = scof + ((p + 9) % 3) * 6 * kFCP;
            for (int e = tid; e < kFCP; e += kFT) {
                const int r = e / kFCK, c = e - r * kFCK;
                const int o = (r + 1) * kFPK + (c + 1);
                Nb19<T> v;
                v.c = pc[o];
                v.xp = pp[o];
                v.xm = pm[o];
                v.yp = pc[o + kFPK];
                v.ym = pc[o - kFPK];
                v.zp = pc[o + 1];
                v.zm = pc[o - 1];
                v.xpyp = pp[o + kFPK];
                v.xmym = pm[o - kFPK];
                v.xmyp = pm[o + kFPK];
                v.xpym = pp[o - kFPK];
                v.ypzp = pc[o + kFPK + 1];
                v.ymzm = pc[o - kFPK - 1];
                v.ymzp = pc[o - kFPK + 1];
                v.ypzm = pc[o + kFPK - 1];
                v.xpzp = pp[o + 1];
                v.xmzm = pm[o - 1];
                v.xmzp = pm[o + 1];
                v.xpzm = pp[o - 1];
                const Cof<T> a = cofactors(v, ih2);
                const T w = MODE == 1 ? slam[((p + 9) % 3) * kFCP + e] : T(1);
                d[e] = MODE == 1 ? a.xx * w : a.xx;
                d[kFCP + e] = MODE == 1 ? a.yy * w : a.yy;
                d[2 * kFCP + e] = MODE == 1 ? a.zz * w : a.zz;
                d[3 * kFCP + e] = MODE == 1 ? a.xy * w : a.xy;
                d[4 * kFCP + e] = MODE == 1 ? a.yz * w : a.yz;
                d[5 * kFCP + e] = MODE == 1 ? a.xz * w : a.xz;
            }
        };
        // prologue: phi planes i0-2..i0+1, lam planes i0-1, i0, cofactors of planes i0-1, i0
        for (int p = i0 - 2; p <= i0 + 1; ++p) load_phi(p);
        load_lam(i0 - 1);
        load_lam(i0);
        __syncthreads();
        cof_plane(i0 - 1);
        cof_plane(i0);
        for (int p = i0; p < i1; ++p) {
            __syncthreads();   // every read of the slots refilled below is done
            load_phi(p + 2);
            load_lam(p + 1);
            __syncthreads();
            cof_plane(p + 1);
            __syncthreads();
            // J^T lam at tile cell (tj, tk) of plane p
            const T *cm = scof + ((p + 8) % 3) * 6 * kFCP, *cc = scof + ((p + 9) % 3) * 6 * kFCP,
                         *cp = scof + ((p + 10) % 3) * 6 * kFCP;
            const T *lm = slam + ((p + 8) % 3) * kFCP, *lc = slam + ((p + 9) % 3) * kFCP,
                         *lp = slam + ((p + 10) % 3) * kFCP;
            const int o = (tj + 1) * kFCK + (tk + 1);
            auto X = [&](const T *cpl, const T *lpl, int comp, int off) {
                return MODE == 0 ? cpl[comp * kFCP + o + off] * lpl[o + off] : cpl[comp * kFCP + o + off];
            };
            auto jt_here = [&]() {
                const T dxx = X(cp, lp, 0, 0) + X(cm, lm, 0, 0) - T(2) * X(cc, lc, 0, 0);
                const T dyy = X(cc, lc, 1, kFCK) + X(cc, lc, 1, -kFCK) - T(2) * X(cc, lc, 1, 0);
                const T dzz = X(cc, lc, 2, 1) + X(cc, lc, 2, -1) - T(2) * X(cc, lc, 2, 0);
                const T dxy =
                    (X(cp, lp, 3, kFCK) + X(cm, lm, 3, -kFCK)) - (X(cm, lm, 3, kFCK) + X(cp, lp, 3, -kFCK));
                const T dyz = (X(cc, lc, 4, kFCK + 1) + X(cc, lc, 4, -kFCK - 1)) -
                                   (X(cc, lc, 4, -kFCK + 1) + X(cc, lc, 4, kFCK - 1));
                const T dxz = (X(cp, lp, 5, 1) + X(cm, lm, 5, -1)) - (X(cm, lm, 5, 1) + X(cp, lp, 5, -1));
                return (dxx + dyy + dzz) * ih2 + (dxy + dyz + dxz) * (T(0.5) * ih2);
            };
            const int j = j0 + tj, k = k0 + tk;
            const unsigned id = (unsigned)p * NN + (unsigned)j * (unsigned)N + (unsigned)k;
            if (MODE == 0) {
                const T l0 = lc[o];
                if (((p + j + k) & 1) == colour) {
                    const T diag = T(-2) * (cc[o] + cc[kFCP + o] + cc[2 * kFCP + o]) * ih2;
                    out[id] = l0 + (f[id] - jt_here()) / diag;
                } else {
                    out[id] = l0;
                }
            } else if (MODE == 1) {
                const T jt = jt_here();
                const T r = f[id] - jt;
                if (out) out[id] = r;
                if (rout) rout[id] = (float)(r * scale);
                s2.add(sizeof(T) == 8 ? r * r : r);
            } else {
                const T v = sign * jt_here();
                out[id] = v;
                s2.add(v * v);
            }
        }
        __syncthreads();   // the next column refills every slot
    }
    if (MODE != 0) {
        const double t = block_sum<kFT>(s2.get(), sh);
        if (ltid() == 0) partials[4 * blockIdx.x + 1] = t;
    }
}

// Single-CTA Gauss-Seidel on the coarsest level (N^3 <= 4096).
__global__ void __launch_bounds__(kCoarseThreads)
k_jt_coarse(double *lam, double *work, const double *f, const double *cof, int N, double ih2,
            int max_sweeps, double rtol)
{
    __shared__ double sh[32];
    __shared__ double sval;
    const CofPtr<double> C = cof_of(cof, (size_t)N * N * N);
    const int n = N * N * N, half = N >> 1, npairs = N * N * half;
    auto rms = [&]() -> double {
        double s2 = 0.0;
        for (int id = threadIdx.x; id < n; id += blockDim.x) {
            const int k = id % N, j = (id / N) % N, i = id / (N * N);
            const double r = f[id] - jt_at<double>(C, lam, N, i, j, k, ih2, nullptr);
            s2 += r * r;
        }
        const double tot = block_sum<kCoarseThreads>(s2, sh);
        if (ltid() == 0) sval = sqrt(tot / n);
        __syncthreads();
        const double v = sval;
        __syncthreads();
        return v;
    };
    const double r0 = rms();
    double prev = r0;
    for (int sw = 0; sw < max_sweeps; ++sw) {
        for (int colour = 0; colour < 2; ++colour) {
            const double *src = colour == 0 ? lam : work;
            double *dst = colour == 0 ? work : lam;
            for (int pi = threadIdx.x; pi < npairs; pi += blockDim.x) {
                const int m = pi % half, r = pi / half;
                const int j = r % N, i = r / N;
                const int par = (colour + i + j) & 1;
                const int ka = 2 * m + par, kb = 2 * m + 1 - par;
                double d;
                const double jt = jt_at<double>(C, src, N, i, j, ka, ih2, &d);
                const double vnew = src[offs(N, i, j, ka)] + (f[offs(N, i, j, ka)] - jt) / d;
                const double vcopy = src[offs(N, i, j, kb)];
                dst[offs(N, i, j, ka)] = vnew;
                dst[offs(N, i, j, kb)] = vcopy;
            }
            __syncthreads();
        }
        const double cur = rms();
        if (cur <= rtol * r0) break;
        if (rtol > 0.0 && cur >= prev) break;
        prev = cur;
    }
}

template <typename T>
__global__ void __launch_bounds__(kThreads)
k_sub_mean(T *__restrict__ a, size_t n, const double *__restrict__ mean)
{
    const size_t id = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (id < n) a[id] -= (T)*mean;
}

// float(scale a)
__global__ void __launch_bounds__(kThreads)
k_scaled(const double *__restrict__ a, size_t n, double scale, float *__restrict__ out)
{
    for (size_t id = (size_t)blockIdx.x * blockDim.x + threadIdx.x; id < n; id += (size_t)gridDim.x * blockDim.x)
        out[id] = (float)(a[id] * scale);
}
// per-block sums of a^2 (partials column 1)
__global__ void __launch_bounds__(kThreads)
k_sum_squares(const double *__restrict__ a, size_t n, double *__restrict__ partials)
{
    __shared__ double sh[32];
    double s = 0.0;
    for (size_t id = (size_t)blockIdx.x * blockDim.x + threadIdx.x; id < n; id += (size_t)gridDim.x * blockDim.x)
        s += a[id] * a[id];
    const double v = block_sum<kThreads>(s, sh);
    if (ltid() == 0) partials[4 * blockIdx.x + 1] = v;
}
// lam += scale e
__global__ void __launch_bounds__(kThreads)
k_add_scaled(double *__restrict__ lam, const float *__restrict__ e, size_t n, double scale)
{
    for (size_t id = (size_t)blockIdx.x * blockDim.x + threadIdx.x; id < n; id += (size_t)gridDim.x * blockDim.x)
        lam[id] = fma((double)e[id], scale, lam[id]);
}
// a -> floats
__global__ void __launch_bounds__(kThreads)
k_narrow(const double *__restrict__ a, float *__restrict__ out, size_t n)
{
    for (size_t id = (size_t)blockIdx.x * blockDim.x + threadIdx.x; id < n; id += (size_t)gridDim.x * blockDim.x)
        out[id] = (float)a[id];
}

__global__ void __launch_bounds__(kThreads)
k_add_one(double *__restrict__ a, size_t n)
{
    const size_t id = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (id < n) a[id] += 1.0;
}

// lam -= (s_lam / s_n) * nvec
__global__ void __launch_bounds__(kThreads)
k_null_fix(double *__restrict__ lam, const double *__restrict__ nvec, size_t n,
           const double *__restrict__ s_lam, const double *__restrict__ s_n)
{
    const size_t id = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (id < n) lam[id] -= (*s_lam / *s_n) * nvec[id];
}

__global__ void __launch_bounds__(kThreads)
k_sum(const double *__restrict__ a, size_t n, double *__restrict__ partials)
{
    __shared__ double sh[32];
    double s = 0.0;
    for (size_t id = (size_t)blockIdx.x * blockDim.x + threadIdx.x; id < n;
         id += (size_t)gridDim.x * blockDim.x)
        s += a[id];
    const double v = block_sum<kThreads>(s, sh);
    if (ltid() == 0) partials[4 * blockIdx.x + 0] = v;
}

__global__ void __launch_bounds__(kReduceThreads)
k_reduce_col(const double *__restrict__ partials, int nb, int col, double scale, double *out)
{
    __shared__ double sh[32];
    double v = 0.0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) v += partials[4 * b + col];
    v = block_sum<kReduceThreads>(v, sh);
    if (ltid() == 0) *out = v * scale;
}

inline unsigned nred(size_t n)
{
    const size_t b = (n + kThreads - 1) / kThreads;
    return (unsigned)(b < (size_t)kMaxRedBlocks ? (b ? b : 1) : kMaxRedBlocks);
}

#define CK(expr)                                                                   \
    do {                                                                           \
        cudaError_t e_ = (expr);                                                   \
        if (e_ != cudaSuccess) return e_;                                          \
    } while (0)

// grid of the cofactor-forming kernel: its (column, chunk) items,
// at most kMaxRedBlocks CTAs
inline unsigned fine_grid(int N)
{
    const unsigned items = (unsigned)(N / kFK) * (unsigned)(N / kFJ) * (unsigned)(N / fine_chunk(N));
    return items < (unsigned)kMaxRedBlocks ? items : (unsigned)kMaxRedBlocks;
}

// level l applies J^T with cofactors formed from phi (no stored arrays)
inline bool formed(const recon_handle *H, int l) { return l == 0 && !H->adj.stored0; }
inline size_t ncell(int N) { return (size_t)N * N * N; }

// The arrays of the V-cycle in precision T, all levels
template <typename T>
struct JtHier {
    T *th[kMaxLevels], *cof[kMaxLevels], *lam[kMaxLevels], *f[kMaxLevels];   // th: level 0 only
    T *work;     // N^3: ping-pong of the sweeps; residual of the formed level
};

template <typename T>
cudaError_t jt_sweep(recon_handle *H, const JtHier<T> &Y, int l, int sweeps)
{
    const int N = H->Nl[l];
    const T ih2 = (T)(1.0 / (H->hl[l] * H->hl[l]));
    cudaStream_t s = H->stream;
    const dim3 fit = fit_block(N / 2);
    for (int it = 0; it < sweeps; ++it)
        for (int c = 0; c < 2; ++c) {
            const T *src = c ? Y.work : Y.lam[l];
            T *dst = c ? Y.lam[l] : Y.work;
            note_launch();
            if (formed(H, l))
                k_jt_fine<0, T><<<fine_grid(N), kFT, fine_smem<T>(), s>>>(Y.th[0], src, Y.f[l], dst, N, ih2, c, T(1),
                                                                          nullptr, nullptr, T(1));
            else
                k_jt_pass<T><<<fit_grid(N, fit), fit, 0, s>>>(src, dst, Y.f[l], Y.cof[l], N, ih2, c);
        }
    return cudaGetLastError();
}

// linear V-cycle on J^T lam = f at level l.  FP32: the levels of a tail relax
// J instead of J^T (recon_tail.cu; see jt_solve_mixed).
template <typename T>
cudaError_t jt_vcycle(recon_handle *H, const JtHier<T> &Y, int l)
{
    cudaStream_t s = H->stream;
    const recon_config &cf = H->cfg;
    const int N = H->Nl[l];
    const T ih2 = (T)(1.0 / (H->hl[l] * H->hl[l]));
    if constexpr (sizeof(T) == 8) {
        if (l == H->nlev - 1) {
            note_launch();
            k_jt_coarse<<<1, kCoarseThreads, 0, s>>>(Y.lam[l], Y.work, Y.f[l], Y.cof[l], N, ih2,
                                                     cf.coarse_max_sweeps, cf.coarse_rtol);
            return cudaGetLastError();
        }
    }
    CK(jt_sweep<T>(H, Y, l, cf.nu1));
    const int Nc = H->Nl[l + 1];
    const size_t nc = ncell(Nc);
    unsigned nb = row_grid(Nc, kMaxRedBlocks);
    int col = 0;
    double scale = 1.0 / (double)nc;
    if (formed(H, l)) {
        // r = f - J^T lam (cofactors formed from phi), then its 8-son mean
        note_launch();
        k_jt_fine<1, T><<<fine_grid(N), kFT, fine_smem<T>(), s>>>(Y.th[0], Y.lam[l], Y.f[l], Y.work, N, ih2, 0, T(1),
                                                                  H->partials, nullptr, T(1));
        CK(restrict_plain<T>(N, Y.work, Y.f[l + 1], s));
        if (sizeof(T) == 4) {
            nb = fine_grid(N);
            col = 1;   // the sum of r itself
            scale = 1.0 / (double)ncell(N);
        } else {
            nb = nred(nc);
            note_launch();
            k_sum<<<nb, kThreads, 0, s>>>((const double *)Y.f[l + 1], nc, H->partials);
        }
    } else {
        note_launch();
        k_jt_restrict_residual<T><<<nb, row_block(), 0, s>>>(Y.lam[l], Y.f[l], Y.cof[l], N, ih2, Y.f[l + 1],
                                                            H->partials);
    }
    if (sizeof(T) == 4 && tail_ok<float>(Nc)) {
        CK(lin_tail(H, l + 1, (float *)Y.lam[l + 1], (const float *)Y.f[l + 1], (const float *const *)Y.cof, true,
                    true));
    } else {
        note_launch(2);
        k_reduce_col<<<1, kReduceThreads, 0, s>>>(H->partials, nb, col, scale, H->scal + S_ADJ_MEAN);
        k_sub_mean<T><<<blocks_for(nc), kThreads, 0, s>>>(Y.f[l + 1], nc, H->scal + S_ADJ_MEAN);
        CK(cudaMemsetAsync(Y.lam[l + 1], 0, sizeof(T) * nc, s));
        CK(jt_vcycle<T>(H, Y, l + 1));
    }
    CK(prolong_add<T>(Nc, Y.lam[l + 1], (const T *)nullptr, nullptr, 1.0, Y.lam[l], s));
    return jt_sweep<T>(H, Y, l, cf.nu2);
}

// ||f - J^T lam||^2 on the finest grid, or (rout) also scale (f - J^T lam) as floats
cudaError_t jt_residual(recon_handle *H, const double *lam, const double *f, float *rout, double scale, double *norm2)
{
    cudaStream_t s = H->stream;
    const int N = H->N;
    const double ih2 = 1.0 / (H->h * H->h);
    const bool fm = formed(H, 0);
    const unsigned nb = fm ? fine_grid(N) : row_grid(N, kMaxRedBlocks);
    note_launch(2);
    if (fm)
        k_jt_fine<1, double><<<nb, kFT, fine_smem<double>(), s>>>(H->last_phi, lam, f, nullptr, N, ih2, 0, 1.0,
                                                                  H->partials, rout, scale);
    else
        k_jt_apply<<<nb, row_block(), 0, s>>>(lam, f, H->adj.cof[0], N, ih2, 1.0, nullptr, H->partials, rout, scale);
    k_reduce_col<<<1, kReduceThreads, 0, s>>>(H->partials, nb, 1, 1.0, H->scal + S_ADJ_NORM);
    CK(cudaMemcpyAsync(&H->hscal[S_ADJ_NORM], H->scal + S_ADJ_NORM, sizeof(double), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    *norm2 = H->hscal[S_ADJ_NORM];
    return cudaSuccess;
}

// a power of two near 1 / x (x > 0 and finite)
double inv_scale(double x)
{
    int e;
    std::frexp(x, &e);
    e = e > 1000 ? 1000 : (e < -1000 ? -1000 : e);
    return std::ldexp(1.0, -e);
}

// V-cycles per residual of the mixed solve: a V-cycle contracts ~0.12 and the
// FP64 residual costs about as much as one (128^3: 0.46 ms against 0.7), so
// three take most of what FP32 can give (~1e-5) before the next residual.
constexpr int kMixedVcycles = 3;
// The mixed solve goes on to this fraction of the tolerance where it still
// contracts: its last step then leaves an error no larger than the FP64
// V-cycles left, which contracted only ~0.12 below their last residual.
constexpr double kMixedTarget = 0.02;

// J^T lam = f by defect correction: the residual f - J^T lam and lam in FP64,
// the corrections by kMixedVcycles FP32 V-cycles on J^T.  As in the mixed
// solve, the answer's accuracy is the residual's (FP64, relative tol); FP32
// only sets how fast it is reached.  On the levels of 32^3 and below the
// V-cycle relaxes J, which the linear solve's tail kernel does in one launch:
// the cofactors of I + H phi are divergence-free in the continuum, so J^T and
// J agree there up to the discretisation error, and the V-cycles taken stay the
// same.  (On the finer levels J does not do: corrections by J alone stop
// contracting at 160^3 and 192^3.)  Gradient of a 128^3 solve: two such solves
// 156 -> 24 ms; their errors against 64 bits are at most the FP64 V-cycles'.
// Returns the V-cycles taken, -1 on error; *rel is the residual reached
// (above tol when the corrections stopped contracting).
int jt_solve_mixed(recon_handle *H, const JtHier<float> &Y, double *lam, const double *f, double tol, int max_cycles,
                   double *rel)
{
    cudaStream_t s = H->stream;
    const size_t n = ncell(H->N);
    const unsigned nb = nred(n);
    note_launch(2);
    k_sum_squares<<<nb, kThreads, 0, s>>>(f, n, H->partials);
    k_reduce_col<<<1, kReduceThreads, 0, s>>>(H->partials, nb, 1, 1.0, H->scal + S_ADJ_NORM);
    if (cudaMemcpyAsync(&H->hscal[S_ADJ_NORM], H->scal + S_ADJ_NORM, sizeof(double), cudaMemcpyDeviceToHost, s) !=
            cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return -1;
    const double fnorm2 = H->hscal[S_ADJ_NORM];
    if (cudaMemsetAsync(lam, 0, sizeof(double) * n, s) != cudaSuccess) return -1;
    *rel = 0.0;
    if (fnorm2 == 0.0) return 0;
    if (!std::isfinite(fnorm2)) return -1;
    // the right side of a correction is scaled to rms ~1
    double scale = inv_scale(std::sqrt(fnorm2 / (double)n)), last = 1.0;
    note_launch();
    k_scaled<<<stride_blocks(n), kThreads, 0, s>>>(f, n, scale, Y.f[0]);
    int cyc = 0;
    while (cyc < max_cycles) {
        if (cudaMemsetAsync(Y.lam[0], 0, sizeof(float) * n, s) != cudaSuccess) return -1;
        for (int v = 0; v < kMixedVcycles; ++v)
            if (jt_vcycle<float>(H, Y, 0) != cudaSuccess) return -1;
        cyc += kMixedVcycles;
        note_launch();
        k_add_scaled<<<stride_blocks(n), kThreads, 0, s>>>(lam, Y.lam[0], n, 1.0 / scale);
        scale = inv_scale(std::sqrt(fnorm2 / (double)n) * last);
        double r2 = 0.0;
        if (jt_residual(H, lam, f, Y.f[0], scale, &r2) != cudaSuccess) return -1;
        *rel = std::sqrt(r2 / fnorm2);
        if (!std::isfinite(*rel) || *rel < kMixedTarget * tol || *rel > 0.5 * last) break;
        last = *rel;
    }
    return cyc;
}

// The same in FP64 throughout, from the lam given (zero: from 0).
int jt_solve(recon_handle *H, double *lam, const double *f, double tol, int max_cycles, bool zero, double *rel_out)
{
    AdjWork &A = H->adj;
    cudaStream_t s = H->stream;
    const size_t n = ncell(H->N);
    const unsigned nb = nred(n);
    JtHier<double> Y{};
    for (int l = 0; l < H->nlev; ++l) {
        Y.cof[l] = A.cof[l];
        Y.lam[l] = l ? A.lam[l] : lam;
        Y.f[l] = l ? A.f[l] : const_cast<double *>(f);
    }
    Y.th[0] = const_cast<double *>(H->last_phi);
    Y.work = H->work64;
    note_launch(2);
    k_sum_squares<<<nb, kThreads, 0, s>>>(f, n, H->partials);
    k_reduce_col<<<1, kReduceThreads, 0, s>>>(H->partials, nb, 1, 1.0, H->scal + S_ADJ_NORM);
    if (cudaMemcpyAsync(&H->hscal[S_ADJ_NORM], H->scal + S_ADJ_NORM, sizeof(double), cudaMemcpyDeviceToHost, s) !=
            cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return -1;
    const double fnorm = std::sqrt(H->hscal[S_ADJ_NORM]);
    if (zero && cudaMemsetAsync(lam, 0, sizeof(double) * n, s) != cudaSuccess) return -1;
    if (fnorm == 0.0) {
        *rel_out = 0.0;
        return 0;
    }
    int cyc = 0;
    double rel = 1.0;
    for (cyc = 1; cyc <= max_cycles; ++cyc) {
        if (jt_vcycle<double>(H, Y, 0) != cudaSuccess) return -1;
        double r2 = 0.0;
        if (jt_residual(H, lam, f, nullptr, 1.0, &r2) != cudaSuccess) return -1;
        rel = std::sqrt(r2) / fnorm;
        if (!std::isfinite(rel)) return -1;
        if (rel < tol) break;
    }
    *rel_out = rel;
    return cyc > max_cycles ? max_cycles : cyc;
}

// the finest level's cofactors are formed on the fly when configured so and
// the grid tiles into the kernel's 8 x 32 columns
inline bool store0(const recon_handle *H)
{
    return H->cfg.adjoint_store_cofactors != 0 || H->N % kFK != 0 || H->N % kFJ != 0 ||
           (H->N > 64 && H->N % 64 != 0);
}

// grids that are a single tail level solve in FP64 throughout: there is no
// level left to relax J^T on
inline bool mixed_ok(const recon_handle *H) { return !tail_ok<float>(H->N); }

template <typename T>
cudaError_t fine_attr()
{
    CK(cudaFuncSetAttribute(k_jt_fine<0, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fine_smem<T>()));
    CK(cudaFuncSetAttribute(k_jt_fine<1, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fine_smem<T>()));
    return cudaFuncSetAttribute(k_jt_fine<2, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fine_smem<T>());
}

// the arrays of the FP32 corrections
void free32(AdjWork &A)
{
    for (int l = 0; l < kMaxLevels; ++l)
        for (float **p : {&A.lam32[l], &A.f32[l], &A.cof32[l]}) {
            if (*p) cudaFree(*p);
            *p = nullptr;
        }
    A.mixed = A.cof32_ready = false;
}
cudaError_t alloc32(recon_handle *H)
{
    AdjWork &A = H->adj;
    for (int l = 0; l < H->nlev; ++l) {
        const size_t n = ncell(H->Nl[l]);
        if (l > 0) {
            CK(cudaMalloc(&A.lam32[l], sizeof(float) * n));
            CK(cudaMalloc(&A.f32[l], sizeof(float) * n));
        }
        if (l > 0 || A.stored0) CK(cudaMalloc(&A.cof32[l], sizeof(float) * 6 * n));
    }
    return cudaSuccess;
}

// The FP32 corrections' arrays come last: where they do not fit, the solves run
// in FP64 throughout, and where its coarse levels do not fit beside them, they
// make room.  A grid needs no more memory than FP64 alone needs.
cudaError_t adj_alloc(recon_handle *H)
{
    AdjWork &A = H->adj;
    if (A.ready) return cudaSuccess;
    A.stored0 = store0(H);
    CK(fine_attr<double>());
    CK(fine_attr<float>());
    if (A.stored0) CK(cudaMalloc(&A.cof[0], sizeof(double) * 6 * ncell(H->N)));
    CK(cudaMalloc(&A.nvec, sizeof(double) * ncell(H->N)));
    CK(cudaMalloc(&A.f[0], sizeof(double) * ncell(H->N)));
    A.mixed = mixed_ok(H);
    if (A.mixed) {
        const cudaError_t e = alloc32(H);
        if (e == cudaErrorMemoryAllocation) {
            cudaGetLastError();
            free32(A);
        } else if (e != cudaSuccess) {
            return e;
        }
    }
    A.ready = true;
    return cudaSuccess;
}

// the FP64 V-cycle's coarse levels, made when it first runs
cudaError_t alloc64(recon_handle *H)
{
    AdjWork &A = H->adj;
    if (A.ready64) return cudaSuccess;
    for (int l = 1; l < H->nlev; ++l) {
        const size_t n = ncell(H->Nl[l]);
        if (!A.th[l]) CK(cudaMalloc(&A.th[l], sizeof(double) * n));
        if (!A.lam[l]) CK(cudaMalloc(&A.lam[l], sizeof(double) * n));
        if (!A.f[l]) CK(cudaMalloc(&A.f[l], sizeof(double) * n));
        if (!A.cof[l]) CK(cudaMalloc(&A.cof[l], sizeof(double) * 6 * n));
    }
    A.ready64 = true;
    return cudaSuccess;
}

// FP64 potential of the coarse levels and their cofactors
cudaError_t setup64(recon_handle *H)
{
    AdjWork &A = H->adj;
    if (A.cof64_ready) return cudaSuccess;
    cudaError_t e = alloc64(H);
    if (e == cudaErrorMemoryAllocation && A.mixed) {   // in place of the FP32 corrections' arrays
        cudaGetLastError();
        free32(A);
        e = alloc64(H);
    }
    CK(e);
    for (int l = 1; l < H->nlev; ++l) {
        CK(restrict_plain<double>(H->Nl[l - 1], l > 1 ? A.th[l - 1] : H->last_phi, A.th[l], H->stream));
        note_launch();
        k_cof6<double><<<row_grid(H->Nl[l]), row_block(), 0, H->stream>>>(A.th[l], H->Nl[l],
                                                                         1.0 / (H->hl[l] * H->hl[l]), A.cof[l]);
    }
    A.cof64_ready = true;
    return cudaGetLastError();
}

// FP32 arrays of the mixed solve; the finest level's live in the handle's two
// N^3-double scratch arrays
JtHier<float> hier_mixed(recon_handle *H)
{
    AdjWork &A = H->adj;
    const size_t n = ncell(H->N);
    JtHier<float> Y{};
    for (int l = 0; l < H->nlev; ++l) {
        Y.cof[l] = A.cof32[l];
        Y.lam[l] = A.lam32[l];
        Y.f[l] = A.f32[l];
    }
    Y.th[0] = reinterpret_cast<float *>(H->work64);
    Y.f[0] = Y.th[0] + n;
    Y.lam[0] = reinterpret_cast<float *>(H->work64b);
    Y.work = Y.lam[0] + n;
    return Y;
}

// FP32 cofactors of every level from phi and its restrictions (the coarse
// potentials pass through the arrays of lam)
cudaError_t setup_mixed(recon_handle *H, const JtHier<float> &Y)
{
    cudaStream_t s = H->stream;
    for (int l = 0; l < H->nlev; ++l) {
        const int N = H->Nl[l];
        const float *th = l ? Y.lam[l] : Y.th[0];
        if (l) CK(restrict_plain<float>(H->Nl[l - 1], l > 1 ? Y.lam[l - 1] : Y.th[0], Y.lam[l], s));
        if (formed(H, l)) continue;
        if (tail_ok<float>(N)) {
            CK(cof6_split(N, H->hl[l], th, Y.cof[l], s));
        } else {
            note_launch();
            k_cof6<float><<<row_grid(N), row_block(), 0, s>>>(th, N, (float)(1.0 / (H->hl[l] * H->hl[l])), Y.cof[l]);
        }
    }
    return cudaGetLastError();
}

// J^T lam = f from lam = 0: mixed, and in FP64 from where that ends if it
// stops short of tol (or the grid is too small for it).  The V-cycles taken, or
// one of the two errors.
constexpr int kFailed = -1, kNoMemory = -2;
int solve_jt(recon_handle *H, double *lam, const double *f, double tol, int max_cycles, double *rel)
{
    int c = 0;
    *rel = 1.0;
    if (H->adj.mixed) {
        const JtHier<float> Y = hier_mixed(H);
        const size_t n = ncell(H->N);
        note_launch();
        k_narrow<<<stride_blocks(n), kThreads, 0, H->stream>>>(H->last_phi, Y.th[0], n);
        if (!H->adj.cof32_ready) {
            if (setup_mixed(H, Y) != cudaSuccess) return kFailed;
            H->adj.cof32_ready = true;
        }
        c = jt_solve_mixed(H, Y, lam, f, tol, max_cycles, rel);
        if (c < 0 || *rel < tol || c >= max_cycles) return c;
    }
    const bool zero = c == 0 || !std::isfinite(*rel) || *rel > 1.0;   // (a diverged correction is dropped)
    const cudaError_t e = setup64(H);
    if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? kNoMemory : kFailed;
    const int d = jt_solve(H, lam, f, tol, max_cycles - c, zero, rel);
    return d < 0 ? d : c + d;
}

}  // namespace

void adj_free(recon_handle *H)
{
    AdjWork &A = H->adj;
    for (int l = 0; l < kMaxLevels; ++l) {
        if (l > 0) {
            if (A.th[l]) cudaFree(A.th[l]);
            if (A.lam[l]) cudaFree(A.lam[l]);
        }
        if (A.f[l]) cudaFree(A.f[l]);
        if (A.cof[l]) cudaFree(A.cof[l]);
    }
    free32(A);
    if (A.nvec) cudaFree(A.nvec);
    A = AdjWork{};
}

static recon_status failed(recon_handle *H, int code, const char *what)
{
    if (code != kNoMemory) {
        H->err = what;
        return RECON_E_CUDA;
    }
    adj_free(H);
    cudaGetLastError();
    H->err = "adjoint workspace allocation failed";
    return RECON_E_OOM;
}

recon_status adjoint(recon_handle *H, const double *gbar, double *lam)
{
    cudaStream_t s = H->stream;
    AdjWork &A = H->adj;
    cudaError_t e = adj_alloc(H);
    if (e != cudaSuccess) {
        adj_free(H);
        cudaGetLastError();
        H->err = "adjoint workspace allocation failed";
        return RECON_E_OOM;
    }
    const int N = H->N;
    const size_t n = (size_t)N * N * N;
    const double tol = 1e-12;
    const int maxc = 100;
    if (A.ready && A.stored0 != store0(H)) {
        // the cofactor option changed since the workspace was made
        adj_free(H);
        if ((e = adj_alloc(H)) != cudaSuccess) {
            adj_free(H);
            cudaGetLastError();
            H->err = "adjoint workspace allocation failed";
            return RECON_E_OOM;
        }
    }
    if (!A.null_ready) {
        // cofactors follow phi: of this solve from here on
        A.cof32_ready = A.cof64_ready = false;
        if (A.stored0) {
            note_launch();
            k_cof6<double><<<row_grid(N), row_block(), 0, s>>>(H->last_phi, N, 1.0 / (H->h * H->h), A.cof[0]);
        }
        // null vector of J^T: n = 1 + w, J^T w = -J^T 1
        note_launch();
        if (A.stored0)
            k_jt_apply<<<row_grid(N, kMaxRedBlocks), row_block(), 0, s>>>(nullptr, nullptr, A.cof[0], N,
                                                                        1.0 / (H->h * H->h), -1.0, A.f[0],
                                                                        H->partials, nullptr, 1.0);
        else
            k_jt_fine<2, double><<<fine_grid(N), kFT, fine_smem<double>(), s>>>(
                H->last_phi, nullptr, nullptr, A.f[0], N, 1.0 / (H->h * H->h), 0, -1.0, H->partials, nullptr, 1.0);
        double rel = 0.0;
        const int c1 = solve_jt(H, A.nvec, A.f[0], tol, maxc, &rel);
        if (c1 < 0) return failed(H, c1, "adjoint null-vector solve failed");
        note_launch();
        k_add_one<<<blocks_for(n), kThreads, 0, s>>>(A.nvec, n);
        A.null_ready = true;
        A.null_rel = rel;
    }
    // f = gbar - mean(gbar)
    note_launch(3);
    k_sum<<<nred(n), kThreads, 0, s>>>(gbar, n, H->partials);
    k_reduce_col<<<1, kReduceThreads, 0, s>>>(H->partials, nred(n), 0, 1.0 / (double)n, H->scal + S_ADJ_MEAN);
    if ((e = cudaMemcpyAsync(A.f[0], gbar, sizeof(double) * n, cudaMemcpyDeviceToDevice, s)) != cudaSuccess)
        return RECON_E_CUDA;
    k_sub_mean<double><<<blocks_for(n), kThreads, 0, s>>>(A.f[0], n, H->scal + S_ADJ_MEAN);
    double rel = 0.0;
    const int c2 = solve_jt(H, lam, A.f[0], tol, maxc, &rel);
    if (c2 < 0) return failed(H, c2, "adjoint solve failed");
    // lam -= (sum lam / sum n) n
    note_launch(5);
    k_sum<<<nred(n), kThreads, 0, s>>>(lam, n, H->partials);
    k_reduce_col<<<1, kReduceThreads, 0, s>>>(H->partials, nred(n), 0, 1.0, H->scal + S_ADJ_SLAM);
    k_sum<<<nred(n), kThreads, 0, s>>>(A.nvec, n, H->partials);
    k_reduce_col<<<1, kReduceThreads, 0, s>>>(H->partials, nred(n), 0, 1.0, H->scal + S_ADJ_SN);
    k_null_fix<<<blocks_for(n), kThreads, 0, s>>>(lam, A.nvec, n, H->scal + S_ADJ_SLAM, H->scal + S_ADJ_SN);
    if ((e = cudaGetLastError()) != cudaSuccess) return RECON_E_CUDA;
    if (rel >= 1e-8 || A.null_rel >= 1e-8) {
        H->err = "adjoint linear solve stalled at relative residual " + std::to_string(rel);
        return RECON_E_NOCONV;
    }
    H->adj_cycles = c2;
    H->adj_rel = rel;
    return RECON_OK;
}

}  // namespace recon
