// nn_krylov.cu -- the operator-splitting step of the nearest-neighbour Lambda*
// (Sect. 3.2.1): (I - (1-eps) L*) x = y, with L* the 27-entry rows of nn.cu.
//
// With D the diagonal of A = I - (1-eps) L*, the Jacobi-preconditioned system
// is (I - M) x = D^-1 y with M_q,v = (1-eps_v) L*_q,v / D_v off the diagonal;
// a Jacobi sweep is x' = D^-1 y + M x and its change r = x' - x is the
// preconditioned residual.  The solve stops when a sweep would change x by at
// most jtol max |x'| and returns that sweep's x' (the criterion of the plain
// Jacobi iteration, which in optically thick grids at small eps contracts by a
// factor close to 1 per sweep: thousands of sweeps at eps = 1e-4, tau = 1e2).
//
// It gets there by defect correction: r is evaluated in FP64, the correction
// (I - M) d = r is solved by BiCGSTAB in FP32 to about 1e-5 of r, and x += d;
// each round gains about five decades.  The FP64 pipe, narrow on this GPU, only
// evaluates r (26 FMAs per voxel per round).  Should a round fail to halve r,
// the corrections are solved by BiCGSTAB in FP64 from then on; should the
// rounds run out, Jacobi sweeps finish the solve.
//
// Each block owns a contiguous range of voxels.  Where it fits in shared
// memory, the FP32 solve keeps the block's halo of the 27-point stencil
// (its range widened by n2 n3 + 2 n3 voxels either side on the spherical grid,
// 2 n2 n3 on the cylindrical one or n2 n3 + n3 + 1 with the phi seam left out)
// of r, p and v there, and the block's FP32 rows of M too where those fit, and
// needs two grid barriers an iteration (bicgstab_tile).
//
// The whole solve is one cooperative launch.  A vector operation on 1e5 voxels
// is a few microseconds of work, so one launch per BiCGSTAB phase plus a host
// round trip for each stopping test cost more than the arithmetic.  All blocks
// are resident and meet at a grid barrier between phases; every block sums the
// per-block partials of a reduction in the same fixed order, so all blocks
// take the same decisions and the solve is deterministic.  Every barrier wait
// is bounded: a block that has waited a second (or sees that another block
// gave up) raises the fail word and returns, and the host reports a timeout.
//
// The bound is latency: barriers, reductions and halos through L2, 16 % of it
// arithmetic.  Measured on a GB300 per BiCGSTAB iteration, at 65 x 33 x 65 /
// 33 x 17 x 33 / 17 x 9 x 17 voxels (33 x 32 x 33 / 65^3 cylindrical):
//   three phases, arrival counter, partials read after it, the coefficients'
//   FP64 arithmetic in every thread           32.6 / 23.8 / 23.6 (28.1 / 76.8) us
//   + partials in the arrival packets, coefficients in one thread, fence.acq_rel,
//     neighbour rows without branches         26.2 / 20.6 / 21.4 us
//   + two phases                              23.7 / 18.8 / 18.6 us
//   + polls of the packets' numbers alone (the partials in the polled words cost
//     3500 cycles a poll), two-float sums
//                                             17.1 / 12.8 / 13.3 (17.5 / 48.2) us
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>
#include <cmath>

#include "rt_internal.h"

namespace rtk {
namespace {

constexpr int RT_ = 512;              // threads per block at most: a block has about one per voxel it owns
constexpr int OS_BLOCKS_PER_SM = 1;   // resident blocks per SM the launch asks for (at most)
constexpr int MAXB = 2048;            // blocks of the launch at most (arrival packets)
constexpr int PW = 8;                 // 8-byte words of an arrival packet: its number and up to four partials
constexpr int MAX_ROUNDS = 40;        // defect-correction rounds before Jacobi sweeps take over
constexpr double TOL32 = 1e-5;        // FP32 correction solve: residual relative to r
enum { W_FAIL, W_ITS, W_SWEEPS, W_STATUS, W_XSEL, W_N };             // control words
constexpr int NPK = 5;                 // packets a lane of the polling warp holds at a time (152 blocks: one go)
constexpr int CTL_WORDS = 8;          // 8-byte words kept for them in front of the packets
constexpr unsigned long long WAIT_NS = 1000000000ull;  // a barrier wait gives up after 1 s
constexpr unsigned WAIT_POLLS = 1u << 26;              // or after this many polls

template <typename T>
struct Inner {  // one BiCGSTAB's vectors and the preconditioned rows in its precision
    T *d, *r, *rh, *p, *v, *s, *t;
    T *M;        // 27 planes (plane 13 unused), written and read by the thread owning the row
    int64_t ms;  // plane stride: n for FP64, n rounded up to 4 for FP32 (16-byte aligned planes)
};

struct Kv {  // the solve's vectors and constants
    int n, sph, n1, n2, n3;
    const double *L27, *eps, *y;
    double *x, *x1, *res, *yd;  // iterate, Jacobi output x', FP64 residual r, D^-1 y
    Inner<double> i64;
    Inner<float> i32;
    unsigned *ctl;  // W_N control words and then
    unsigned long long *pk;  // the arrival packets: 2 x blocks x PW words (all zeroed before the launch)
    double jtol;
    int krylov, kmax, jmax, stall;
    int64_t n4;     // n rounded up to 4: stride of the FP32 vectors
    int rows;       // voxels per block, a multiple of 4: block b owns [b rows, (b + 1) rows)
    int halo;       // halo reach in voxel index either side of the block's range
    int hcap;       // halo buffer length in shared memory (floats, a multiple of 4)
    int tile;       // the FP32 solve keeps its halos in shared memory
    int msm;        // ... and the block's FP32 rows M too
    int far;        // the halo leaves out the neighbours across the phi seam (cylindrical)
};

#define OWN(i) for (int i = lo + (int)threadIdx.x; i < hi; i += (int)blockDim.x)

__device__ __forceinline__ double fmat(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float fmat(float a, float b, float c) { return fmaf(a, b, c); }

// Maxima of non-negative values (or NaN) on their bit patterns: for
// non-negative values the order of the bits is the numeric order, and +inf and
// NaN sort last, so a non-finite entry survives the reduction.  Integer pipe.
__device__ __forceinline__ double maxb(double a, double b)
{
    const unsigned long long x = (unsigned long long)__double_as_longlong(a),
                             y = (unsigned long long)__double_as_longlong(b);
    return __longlong_as_double((long long)(x > y ? x : y));
}
__device__ __forceinline__ float maxb(float a, float b)
{
    const unsigned x = __float_as_uint(a), y = __float_as_uint(b);
    return __uint_as_float(x > y ? x : y);
}

// |a| by clearing the sign bit
__device__ __forceinline__ double absb(double a)
{
    return __longlong_as_double(__double_as_longlong(a) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ float absb(float a) { return __uint_as_float(__float_as_uint(a) & 0x7fffffffu); }

// Calls f(q, u) for each neighbour u of voxel v that exists, in slot order
// q = 9 (di+1) + 3 (dj+1) + (dk+1), q != 13; the phi axis (k spherical, j
// cylindrical) is periodic.  The offsets along each axis are formed once per
// voxel, so a neighbour costs an add and a predicate.
template <class F>
__device__ __forceinline__ void for_neighbours(const Kv &a, int v, F &&f)
{
    const int n23 = a.n2 * a.n3;
    const int i0 = v / n23, rem = v - i0 * n23, j0 = rem / a.n3, k0 = rem - j0 * a.n3;
    int oij[9], ok3[3];
    bool vij[9], vk3[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        int j = j0 + d - 1, k = k0 + d - 1;
        if (a.sph) k = (k < 0) ? k + a.n3 : ((k >= a.n3) ? k - a.n3 : k);
        else j = (j < 0) ? j + a.n2 : ((j >= a.n2) ? j - a.n2 : j);
        ok3[d] = k - k0;
        vk3[d] = k >= 0 && k < a.n3;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const int i = i0 + c - 1;
            oij[3 * c + d] = (c - 1) * n23 + (j - j0) * a.n3;
            vij[3 * c + d] = i >= 0 && i < a.n1 && j >= 0 && j < a.n2;
        }
    }
#pragma unroll
    for (int q = 0; q < 27; ++q) {
        if (q == 13) continue;
        if (vij[q / 3] && vk3[q % 3]) f(q, v + oij[q / 3] + ok3[q % 3]);
    }
}

// acc +- sum over q != 13 of M_q,v u[neighbour q of v] (minus with NEG); u is
// read past L1, since other blocks of this launch wrote it
template <bool NEG, typename T>
__device__ __forceinline__ T rowdot(const Kv &a, const T *M, int64_t ms, int v, const T *u, T acc)
{
    for_neighbours(a, v, [&](int q, int w) {
        const T m = M[q * ms + v];
        acc = fmat(NEG ? -m : m, __ldcg(u + w), acc);
    });
    return acc;
}

__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// 16-byte asynchronous copy from global to shared memory, cached in L2 only
// (other blocks of this launch write the source); done at cp_async_wait
__device__ __forceinline__ void cp_async16(float *smem, const float *gmem)
{
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gmem) : "memory");
}

// floats [b4, e4) of g (multiples of 4) into h[0 .. e4 - b4), asynchronously
__device__ __forceinline__ void halo_copy(float *h, const float *g, int b4, int e4)
{
    for (int j = 4 * (int)threadIdx.x; j < e4 - b4; j += 4 * (int)blockDim.x) cp_async16(h + j, g + b4 + j);
}

__device__ __forceinline__ unsigned long long now_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Sums that travel between lanes and blocks.  Of FP32 values: an unevaluated sum
// of two floats (48 bits), added with the error-free transformation of Knuth's
// two-sum on the FP32 pipe, where an addition takes 4 cycles; an FP64 addition
// takes a warp above 100 here, and a reduction is a chain of 14 of them.  Of FP64
// values: FP64.  The partials carry the rounding of FP32 products and sums, 3e-9 to
// 1e-8 of the sum of their sizes; added as two floats or in FP64, 300 sets of 608
// partials over six decades gave the exact sum both times.
struct Two {
    float h, l;
};
__device__ __forceinline__ Two add2(Two a, Two b)
{
    const float s = a.h + b.h, bb = s - a.h;
    const float e = (a.h - (s - bb)) + (b.h - bb) + (a.l + b.l);
    const float h = s + e;
    return Two{h, e - (h - s)};
}
template <typename T> struct Acc;
template <> struct Acc<float> {
    using V = Two;
    __device__ static V of(float x) { return V{x, 0.0f}; }
    __device__ static V add(V a, V b) { return add2(a, b); }
    // non-negative values, their low parts 0
    __device__ static V max(V a, V b) { return V{maxb(a.h, b.h), 0.0f}; }
    __device__ static V down(V a, int o)
    {
        return V{__shfl_down_sync(0xffffffffu, a.h, o), __shfl_down_sync(0xffffffffu, a.l, o)};
    }
    __device__ static unsigned long long bits(V a)
    {
        return (unsigned long long)__float_as_uint(a.h) | (unsigned long long)__float_as_uint(a.l) << 32;
    }
    __device__ static V from(unsigned long long w)
    {
        return V{__uint_as_float((unsigned)w), __uint_as_float((unsigned)(w >> 32))};
    }
    __device__ static double value(V a) { return (double)a.h + (double)a.l; }
};
template <> struct Acc<double> {
    using V = double;
    __device__ static V of(double x) { return x; }
    __device__ static V add(V a, V b) { return a + b; }
    __device__ static V max(V a, V b) { return maxb(a, b); }
    __device__ static V down(V a, int o) { return __shfl_down_sync(0xffffffffu, a, o); }
    __device__ static unsigned long long bits(V a) { return (unsigned long long)__double_as_longlong(a); }
    __device__ static V from(unsigned long long w) { return __longlong_as_double((long long)w); }
    __device__ static double value(V a) { return a; }
};

__device__ __forceinline__ unsigned long long ld_acquire64(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release64(unsigned long long *p, unsigned long long v)
{
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// What a launch carries from barrier to barrier.
struct Bar {
    unsigned gen;  // barriers passed
    bool hold;     // leave this block's next arrival out (the test hook)
};

// Grid-wide barrier of the cooperative launch and reduction in one: w[0..K) is
// reduced over the block (a sum, or the maxb maximum where bit c of MAXM is
// set; in T within a warp, as Acc<T> across the warps), the block's arrival is a 64-byte packet with its partials behind a word
// that holds the barrier's number, and warp 0 of every block waits for all
// packets and adds them in one fixed order into tot, so all blocks take the same
// decisions.  Packets alternate between two slots: a block overwrites the one of
// barrier g at g + 2, which it reaches only after every block arrived at g + 1,
// that is, read g.  The release store and the acquire loads of the number order
// the partials and the blocks' other writes around the barrier.  False when the
// wait gave up: the fail word is then set and every block returns at its next
// barrier.
template <int K, unsigned MAXM, typename T>
__device__ __forceinline__ bool grid_reduce(const Kv &a, Bar &bar, T (&w)[K], double *tot)
{
    using A = Acc<T>;
    using V = typename A::V;
    __shared__ V red[K][RT_ / 32];
    __shared__ int ok_s;
    constexpr unsigned FULL = 0xffffffffu;
    static_assert(K + 1 <= PW, "packet");
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int c = 0; c < K; ++c) {
            const T u = __shfl_down_sync(FULL, w[c], o);
            w[c] = ((MAXM >> c) & 1u) ? maxb(w[c], u) : w[c] + u;
        }
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int c = 0; c < K; ++c) red[c][threadIdx.x >> 5] = A::of(w[c]);
    ++bar.gen;
    __syncthreads();
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        unsigned long long *const slot = a.pk + (size_t)(bar.gen & 1u) * gridDim.x * PW;
        V s[K];
#pragma unroll
        for (int c = 0; c < K; ++c) s[c] = lane < (int)(blockDim.x >> 5) ? red[c][lane] : A::of(T(0));
#pragma unroll
        for (int o = RT_ / 64; o > 0; o >>= 1)
#pragma unroll
            for (int c = 0; c < K; ++c) {
                const V u = A::down(s[c], o);
                s[c] = ((MAXM >> c) & 1u) ? A::max(s[c], u) : A::add(s[c], u);
            }
        if (lane == 0 && !bar.hold) {
            unsigned long long *const mine = slot + (size_t)PW * blockIdx.x;
#pragma unroll
            for (int c = 0; c < K; ++c) __stcg(mine + 1 + c, A::bits(s[c]));
            st_release64(mine, bar.gen);
        }
#pragma unroll
        for (int c = 0; c < K; ++c) s[c] = A::of(T(0));
        int good = 1;
        unsigned polls = 0;
        unsigned long long t0 = 0;
        for (int b0 = 0; b0 < (int)gridDim.x; b0 += 32 * NPK) {  // NPK packets per lane at a time
            const unsigned long long *pk[NPK];
#pragma unroll
            for (int h = 0; h < NPK; ++h)  // lanes past the last block wait for it and leave its partials out
                pk[h] = slot + (size_t)PW * min(b0 + 32 * h + lane, (int)gridDim.x - 1);
            for (;;) {
                unsigned long long x[NPK];
#pragma unroll
                for (int h = 0; h < NPK; ++h) x[h] = ld_acquire64(pk[h]);
                bool all = true;
#pragma unroll
                for (int h = 0; h < NPK; ++h) all = all && x[h] == bar.gen;
                if (__all_sync(FULL, all)) break;
                if ((++polls & 255u) == 0u) {  // every 256 polls: the clock, the fail word
                    const unsigned long long t = now_ns();
                    if (t0 == 0) t0 = t;
                    const bool out = ld_acquire(a.ctl + W_FAIL) != 0u || polls >= WAIT_POLLS || t - t0 > WAIT_NS;
                    if (__any_sync(FULL, out)) {
                        if (lane == 0) atomicExch(a.ctl + W_FAIL, 1u);
                        good = 0;
                        break;
                    }
                }
            }
            if (!good) break;
            unsigned long long x[NPK][K];
#pragma unroll
            for (int h = 0; h < NPK; ++h)
#pragma unroll
                for (int c = 0; c < K; ++c) x[h][c] = __ldcg(pk[h] + 1 + c);
#pragma unroll
            for (int h = 0; h < NPK; ++h)
#pragma unroll
                for (int c = 0; c < K; ++c) {
                    const V u = b0 + 32 * h + lane < (int)gridDim.x ? A::from(x[h][c]) : A::of(T(0));
                    s[c] = ((MAXM >> c) & 1u) ? A::max(s[c], u) : A::add(s[c], u);
                }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int c = 0; c < K; ++c) {
                const V u = A::down(s[c], o);
                s[c] = ((MAXM >> c) & 1u) ? A::max(s[c], u) : A::add(s[c], u);
            }
        if (lane == 0) {
#pragma unroll
            for (int c = 0; c < K; ++c) tot[c] = A::value(s[c]);
            ok_s = good;
        }
    }
    bar.hold = false;
    __syncthreads();
    return ok_s != 0;
}

// The barrier alone.
__device__ __forceinline__ bool grid_sync(const Kv &a, Bar &bar, double *tot)
{
    float w[1] = {0.0f};
    return grid_reduce<1, 0u>(a, bar, w, tot);
}

// Scalars of an iteration that thread 0 forms from the totals and every thread
// reads (behind a block barrier).
struct Scal {
    double d[2];
    float f[2];
    int stop;  // 0 go on
};
template <typename T> __device__ __forceinline__ T scal(const Scal &s, int i);
template <> __device__ __forceinline__ double scal<double>(const Scal &s, int i) { return s.d[i]; }
template <> __device__ __forceinline__ float scal<float>(const Scal &s, int i) { return s.f[i]; }
__device__ __forceinline__ void put(Scal &s, int i, double v)
{
    s.d[i] = v;
    s.f[i] = (float)v;
}

// The BiCGSTAB coefficients and the stopping rules, kept by thread 0.
struct Coefs {
    double rho, alpha, omega, beta, best;
    int best_it;
    bool bad;
    __device__ void start() { rho = 0.0, alpha = omega = 1.0, beta = 0.0, best = INFINITY, best_it = 0, bad = false; }
    __device__ void set_alpha(double rv)
    {
        alpha = rho / rv;
        if (!(rv != 0.0) || !isfinite(alpha)) {
            bad = true;
            alpha = 0.0;
        }
    }
    __device__ void set_omega(double ts, double tt)
    {
        omega = tt > 0.0 ? ts / tt : 0.0;
        if (!isfinite(omega)) {
            bad = true;
            omega = 0.0;
        }
    }
    // after set_omega: quotients of like sizes, so that a source function of any scale
    // passes (rho and the sums go with its square, their products with its fourth power)
    __device__ void set_rho(double rho_new)
    {
        beta = (rho_new / rho) * (alpha / omega);
        rho = rho_new;
        if (!isfinite(beta) || !(rho != 0.0)) bad = true;
    }
    // after iteration it with max |residual| mr: whether to stop (the FP64 residual judges the outcome)
    __device__ bool stop(double mr, double tol, int it, int window)
    {
        if (!isfinite(mr) || !(mr > tol) || bad) return true;
        if (mr < 0.5 * best) {
            best = mr;
            best_it = it;
        } else if (it - best_it >= window) {
            return true;  // stagnation
        }
        return false;
    }
};

// BiCGSTAB in T on (I - M) d = r (r the FP64 residual, own rows) from d = 0,
// until max |residual| <= tol, a breakdown, `window` iterations without
// halving the residual, or kmax iterations.  Vectors in global memory; each
// thread owns the same voxels of the block's range in every phase, so only the
// neighbour reads of the matrix-vector products and the partials cross blocks.
// Returns the iterations, or -1 when a barrier wait gave up.
template <typename T>
__device__ __forceinline__ int bicgstab(const Kv &a, const Inner<T> &b, double tol, int window, Bar &bar, double *tot,
                                        int lo, int hi)
{
    __shared__ Scal sc;
    Coefs q;
    q.start();
    T w0[1] = {T(0)};
    OWN(i) {
        const T ri = (T)a.res[i];
        b.d[i] = T(0);
        b.r[i] = ri;
        b.rh[i] = ri;
        b.p[i] = T(0);
        b.v[i] = T(0);
        w0[0] = fmat(ri, ri, w0[0]);
    }
    if (!grid_reduce<1, 0u>(a, bar, w0, tot)) return -1;
    if (threadIdx.x == 0) {
        q.rho = tot[0];
        put(sc, 0, 0.0);  // beta
        put(sc, 1, 1.0);  // omega
        sc.stop = 0;
    }
    __syncthreads();
    int it = 0;
    while (it < a.kmax) {
        ++it;
        // p = r + beta (p - omega v)
        {
            const T bt = scal<T>(sc, 0), om = scal<T>(sc, 1);
            OWN(i) b.p[i] = fmat(bt, fmat(-om, b.v[i], b.p[i]), b.r[i]);
        }
        if (!grid_sync(a, bar, tot)) return -1;
        // v = (I - M) p; alpha = rho / (rh, v)
        T w1[1] = {T(0)};
        OWN(i) {
            const T vi = rowdot<true>(a, b.M, b.ms, i, b.p, b.p[i]);
            b.v[i] = vi;
            w1[0] = fmat(b.rh[i], vi, w1[0]);
        }
        if (!grid_reduce<1, 0u>(a, bar, w1, tot)) return -1;
        if (threadIdx.x == 0) {
            q.set_alpha(tot[0]);
            put(sc, 0, q.alpha);
        }
        __syncthreads();
        const T al = scal<T>(sc, 0);
        // s = r - alpha v
        OWN(i) b.s[i] = fmat(-al, b.v[i], b.r[i]);
        if (!grid_sync(a, bar, tot)) return -1;
        // t = (I - M) s; omega = (t, s) / (t, t)
        T w2[2] = {T(0), T(0)};
        OWN(i) {
            const T si = b.s[i];
            const T ti = rowdot<true>(a, b.M, b.ms, i, b.s, si);
            b.t[i] = ti;
            w2[0] = fmat(ti, si, w2[0]);
            w2[1] = fmat(ti, ti, w2[1]);
        }
        if (!grid_reduce<2, 0u>(a, bar, w2, tot)) return -1;
        if (threadIdx.x == 0) {
            q.set_omega(tot[0], tot[1]);
            put(sc, 1, q.omega);
        }
        __syncthreads();
        // d += alpha p + omega s; r = s - omega t; rho = (rh, r); max |r|
        T w3[2] = {T(0), T(0)};
        {
            const T om = scal<T>(sc, 1);
            OWN(i) {
                const T si = b.s[i];
                b.d[i] = fmat(om, si, fmat(al, b.p[i], b.d[i]));
                const T ri = fmat(-om, b.t[i], si);
                b.r[i] = ri;
                w3[0] = fmat(b.rh[i], ri, w3[0]);
                w3[1] = maxb(w3[1], absb(ri));
            }
        }
        if (!grid_reduce<2, 2u>(a, bar, w3, tot)) return -1;
        if (threadIdx.x == 0) {
            q.set_rho(tot[0]);
            sc.stop = q.stop(tot[1], tol, it, window);
            put(sc, 0, q.beta);
        }
        __syncthreads();
        if (sc.stop) break;
    }
    return it;
}

// The value at neighbour j of p = r + beta (p - omega v) or s = r - alpha v,
// formed by its owner in shared memory; a block that finds j outside its halo
// forms it from the published vectors with the same operations.
__device__ __forceinline__ float form_p(float r, float p, float v, float bt, float om)
{
    return fmaf(bt, fmaf(-om, v, p), r);
}
__device__ __forceinline__ float form_s(float r, float v, float al) { return fmaf(-al, v, r); }
__device__ __forceinline__ float4 form_p4(float4 r, float4 p, float4 v, float bt, float om)
{
    return make_float4(form_p(r.x, p.x, v.x, bt, om), form_p(r.y, p.y, v.y, bt, om), form_p(r.z, p.z, v.z, bt, om),
                       form_p(r.w, p.w, v.w, bt, om));
}

// u_v - sum over q != 13 of M_q,v u[neighbour q of v], u read from the halo h
// (voxels hb .. he-1) or, past it, formed by far(j); M from the block's copy sm
// (plane stride rows, from voxel lo) or from global memory
template <class F>
__device__ __forceinline__ float rowdot_tile(const Kv &a, const float *sm, int lo, int v, const float *h, int hb, int he,
                                             F &&far, float acc)
{
    const unsigned span = (unsigned)(he - hb);
    for_neighbours(a, v, [&](int q, int u) {
        const float val = (unsigned)(u - hb) < span ? h[u - hb] : far(u);
        const float m = a.msm ? sm[q * a.rows + (v - lo)] : a.i32.M[q * a.i32.ms + v];
        acc = fmaf(-m, val, acc);
    });
    return acc;
}

// The same for a voxel whose neighbours are all in the halo (any voxel of the
// spherical grid, and those off the phi seam of the cylindrical one): without a
// branch or a predicate, so that the 52 shared-memory reads of a row are in flight
// together (in the branched form each waits for the one before: 3 us a row).
// A neighbour that does not exist has M = 0 and reads some voxel of the halo.
// Same order of sums.
template <bool MSM>
__device__ __forceinline__ float rowdot_halo(const Kv &a, const float *M, int64_t ms, int v, const float *h, float acc)
{
    const int n23 = a.n2 * a.n3;
    const int i0 = v / n23, rem = v - i0 * n23, j0 = rem / a.n3, k0 = rem - j0 * a.n3;
    int oi[3], oj[3], ok[3];
    oi[0] = i0 > 0 ? -n23 : 0;
    oi[2] = i0 + 1 < a.n1 ? n23 : 0;
    oj[0] = j0 > 0 ? -a.n3 : (a.sph ? 0 : (a.n2 - 1) * a.n3);
    oj[2] = j0 + 1 < a.n2 ? a.n3 : (a.sph ? 0 : (1 - a.n2) * a.n3);
    ok[0] = k0 > 0 ? -1 : (a.sph ? a.n3 - 1 : 0);
    ok[2] = k0 + 1 < a.n3 ? 1 : (a.sph ? 1 - a.n3 : 0);
    oi[1] = oj[1] = ok[1] = 0;
    float m[27], x[27];
#pragma unroll
    for (int q = 0; q < 27; ++q) {
        if (q == 13) continue;
        m[q] = MSM ? M[q * (int)ms] : M[q * ms];
        x[q] = h[oi[q / 9] + oj[(q / 3) % 3] + ok[q % 3]];
    }
#pragma unroll
    for (int q = 0; q < 27; ++q)
        if (q != 13) acc = fmaf(-m[q], x[q], acc);
    return acc;
}

// u_v - the row of v by whichever of the two forms applies
template <class F>
__device__ __forceinline__ float row_tile(const Kv &a, const float *sm, int lo, int v, const float *h, int hb, int he,
                                          F &&far, float acc)
{
    bool seam = false;
    if (a.far) {
        const int j = (v / a.n3) % a.n2;
        seam = j == 0 || j + 1 == a.n2;
    }
    if (seam) return rowdot_tile(a, sm, lo, v, h, hb, he, far, acc);
    return a.msm ? rowdot_halo<true>(a, sm + (v - lo), a.rows, v, h + (v - hb), acc)
                 : rowdot_halo<false>(a, a.i32.M + v, a.i32.ms, v, h + (v - hb), acc);
}

// FP32 BiCGSTAB as bicgstab<float>, with the halos of r (then s), p and v and
// the own-range d and rh in shared memory, in two phases an iteration, a grid
// barrier after each:
//   A: r = s - omega t and p = r + beta (p - omega v) over the halo (each block
//      forms its copies with the owners' operations; only t is read from L2);
//      v = (I - M) p published; (rh, v) and max |r|
//   B: s = r - alpha v over the halo (only v is read); t = (I - M) s published;
//      (t, s), (t, t), (rh, s) and (rh, t), from which rho = (rh, s) - omega (rh, t)
// so rho needs no third phase (the difference cancels where rho is small; iterations of
// six steps on 14 grids and opacities, tau 1 to 1e4 and eps 1e-2 to 1e-8, against those
// with (rh, r) summed by itself: 54 to 3000, between 0.96 and 1.02 times as many); the stopping test of an iteration comes with the
// next one's A.  A barrier, its reduction and the halo's way through L2 are most
// of a phase.  With OWN, (rh, r) and max |r| are reduced as soon as r is formed
// (a third barrier between the two lines of A, the iterates of bicgstab<float>).
// Adds d to x.  Returns the iterations, or -1 when a barrier wait gave up.
constexpr int TPF = 3;  // 16-byte pieces of the t halo a thread has in flight while thread 0 forms the scalars

template <bool OWN_RHO>
__device__ __forceinline__ int bicgstab_tile(const Kv &a, double tol, int window, Bar &bar, double *tot, int lo, int hi)
{
    extern __shared__ float4 dsm4[];
    __shared__ Scal sc;
    float *const dsm = reinterpret_cast<float *>(dsm4);
    Coefs k;
    k.start();
    // halo [hb, he) widened to 16-byte boundaries; hl floats copied per vector
    const int hb = max(0, lo - a.halo) & ~3;
    const int he = (int)min((long long)((min(a.n, hi + a.halo) + 3) & ~3), (long long)a.n4);
    const int hl = max(0, he - hb), hl4 = hl >> 2;
    float *const hr = dsm, *const hp = hr + a.hcap, *const hv = hp + a.hcap;
    float *const sd = hv + a.hcap, *const srh = sd + a.rows;
    float *const sm = srh + a.rows;  // 27 planes of rows floats when a.msm
    if (a.msm && hi > lo) {
        const int e4 = (int)min((long long)((hi + 3) & ~3), (long long)a.n4);
        for (int q = 0; q < 27; ++q)
            if (q != 13) halo_copy(sm + q * a.rows, a.i32.M + q * a.i32.ms, lo, e4);
    }
    float *const gr = a.i32.r, *const gv = a.i32.v, *const gt = a.i32.t;  // published: r at the start, v, t
    float w0[1] = {0.0f};
    OWN(i)
    {
        const float ri = (float)a.res[i];
        gr[i] = ri;
        srh[i - lo] = ri;
        sd[i - lo] = 0.0f;
        w0[0] = fmaf(ri, ri, w0[0]);
    }
    cp_async_wait();
    if (!grid_reduce<1, 0u>(a, bar, w0, tot)) return -1;
    halo_copy(hr, gr, hb, he);
    if (threadIdx.x == 0) {
        k.rho = tot[0];
        sc.stop = 0;
    }
    cp_async_wait();
    __syncthreads();
    for (int j = threadIdx.x; j < hl; j += blockDim.x) hp[j] = hr[j];
    __syncthreads();
    int it = 0;
    float al = 0.0f, bt = 0.0f, om = 0.0f;
    for (;;) {
        float w1[2] = {0.0f, 0.0f};
        if (it > 0) {  // A's update from the last iteration's t, with its omega and the new rho
            const float4 *t4 = reinterpret_cast<const float4 *>(gt + hb);
            float4 tv[TPF];
#pragma unroll
            for (int u = 0; u < TPF; ++u) {
                const int j = (int)threadIdx.x + u * (int)blockDim.x;
                tv[u] = j < hl4 ? __ldcg(t4 + j) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            }
            if (threadIdx.x == 0) {
                k.set_omega(tot[0], tot[1]);
                if (!OWN_RHO) {
                    k.set_rho(tot[2] - k.omega * tot[3]);
                    put(sc, 0, k.beta);
                }
                put(sc, 1, k.omega);
            }
            __syncthreads();
            if (!OWN_RHO) bt = sc.f[0];
            om = sc.f[1];
            OWN(i) sd[i - lo] = fmaf(om, hr[i - hb], fmaf(al, hp[i - hb], sd[i - lo]));
            __syncthreads();  // the own range's s and p are read before they change
            auto update = [&](int j, float4 t) {
                float4 &r4 = reinterpret_cast<float4 *>(hr)[j], &p4 = reinterpret_cast<float4 *>(hp)[j];
                float4 r = r4, p, v;
                if (!OWN_RHO) p = p4, v = reinterpret_cast<const float4 *>(hv)[j];
                r = make_float4(form_s(r.x, t.x, om), form_s(r.y, t.y, om), form_s(r.z, t.z, om), form_s(r.w, t.w, om));
                r4 = r;
                if (!OWN_RHO) p4 = form_p4(r, p, v, bt, om);
            };
#pragma unroll
            for (int u = 0; u < TPF; ++u) {
                const int j = (int)threadIdx.x + u * (int)blockDim.x;
                if (j < hl4) update(j, tv[u]);
            }
            for (int j = (int)threadIdx.x + TPF * (int)blockDim.x; j < hl4; j += (int)blockDim.x)
                update(j, __ldcg(t4 + j));
            __syncthreads();
            if (OWN_RHO) {
                float w3[2] = {0.0f, 0.0f};
                OWN(i)
                {
                    const float ri = hr[i - hb];
                    w3[0] = fmaf(srh[i - lo], ri, w3[0]);
                    w3[1] = maxb(w3[1], absb(ri));
                }
                if (!grid_reduce<2, 2u>(a, bar, w3, tot)) return -1;
                if (threadIdx.x == 0) {
                    k.set_rho(tot[0]);
                    sc.stop = k.stop(tot[1], tol, it, window) || it >= a.kmax;
                    put(sc, 0, k.beta);
                }
                __syncthreads();
                if (sc.stop) break;  // d holds the iterations done
                bt = sc.f[0];
                for (int j = threadIdx.x; j < hl4; j += (int)blockDim.x) {
                    float4 &p4 = reinterpret_cast<float4 *>(hp)[j];
                    p4 = form_p4(reinterpret_cast<const float4 *>(hr)[j], p4, reinterpret_cast<const float4 *>(hv)[j], bt,
                                 om);
                }
                __syncthreads();
            }
        }
        // v = (I - M) p; alpha = rho / (rh, v).  Past the halo (the phi seam of the
        // cylindrical grid) p is published too and read there.
        if (a.far) {
            float *const gp = a.i32.p;
            OWN(i) gp[i] = hp[i - hb];
            float w[1] = {0.0f};
            if (!grid_reduce<1, 0u>(a, bar, w, tot)) return -1;
        }
        OWN(i)
        {
            const float pi = hp[i - hb];
            const float vi =
                row_tile(a, sm, lo, i, hp, hb, he, [&](int u) { return __ldcg(a.i32.p + u); }, pi);
            gv[i] = vi;
            w1[0] = fmaf(srh[i - lo], vi, w1[0]);
            w1[1] = maxb(w1[1], absb(hr[i - hb]));
        }
        if (!grid_reduce<2, 2u>(a, bar, w1, tot)) return -1;
        // B: halo of v; alpha; s over the halo; t = (I - M) s
        halo_copy(hv, gv, hb, he);
        if (threadIdx.x == 0) {
            sc.stop = !OWN_RHO && it > 0 && (k.stop(tot[1], tol, it, window) || it >= a.kmax);
            k.set_alpha(tot[0]);
            put(sc, 0, k.alpha);
        }
        cp_async_wait();
        __syncthreads();
        if (sc.stop) break;  // d holds the iterations done
        ++it;
        al = sc.f[0];
        for (int j = threadIdx.x; j < hl4; j += blockDim.x) {
            float4 &r4 = reinterpret_cast<float4 *>(hr)[j];
            const float4 v4 = reinterpret_cast<const float4 *>(hv)[j];
            r4 = make_float4(form_s(r4.x, v4.x, al), form_s(r4.y, v4.y, al), form_s(r4.z, v4.z, al),
                             form_s(r4.w, v4.w, al));
        }
        __syncthreads();
        if (a.far) {
            float *const gs = a.i32.s;
            OWN(i) gs[i] = hr[i - hb];
            float w[1] = {0.0f};
            if (!grid_reduce<1, 0u>(a, bar, w, tot)) return -1;
        }
        float w2[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        OWN(i)
        {
            const float si = hr[i - hb];
            const float ti =
                row_tile(a, sm, lo, i, hr, hb, he, [&](int u) { return __ldcg(a.i32.s + u); }, si);
            gt[i] = ti;
            const float rh = srh[i - lo];
            w2[0] = fmaf(ti, si, w2[0]);
            w2[1] = fmaf(ti, ti, w2[1]);
            w2[2] = fmaf(rh, si, w2[2]);
            w2[3] = fmaf(rh, ti, w2[3]);
        }
        if (!grid_reduce<4, 0u>(a, bar, w2, tot)) return -1;
    }
    OWN(i) a.x[i] += (double)sd[i - lo];
    return it;
}

// OWN_RHO: the form of the FP32 solve, a kernel each.
template <bool OWN_RHO>
__global__ void __launch_bounds__(RT_, 1) k_os_solve(Kv a)
{
    __shared__ double tot[4];
    Bar bar{0u, a.stall != 0 && blockIdx.x == 0};
    const int lo = min(a.n, (int)blockIdx.x * a.rows), hi = min(a.n, lo + a.rows);
    // preconditioned rows (FP64 and FP32), D^-1 y and x = 0 (own rows)
    OWN(i) {
        const double e = 1.0 - __ldg(a.eps + i);
        const double id = 1.0 / (1.0 - e * __ldg(a.L27 + 13 * (int64_t)a.n + i));
        const double f = e * id;
#pragma unroll
        for (int q = 0; q < 27; ++q)
            if (q != 13) {
                const double m = f * __ldg(a.L27 + (int64_t)q * a.n + i);
                a.i64.M[q * a.i64.ms + i] = m;
                a.i32.M[q * a.i32.ms + i] = (float)m;
            }
        a.yd[i] = __ldg(a.y + i) * id;
        a.x[i] = 0.0;
    }
    if (!grid_sync(a, bar, tot)) return;
    int its = 0, sweeps = 0, status = 1;
    bool done = false;
    if (a.krylov) {
        double prev = INFINITY;
        bool fp64 = false;
        for (int round = 0; round <= MAX_ROUNDS; ++round) {
            // x' = D^-1 y + M x, r = x' - x; max |r|, max |x'|
            double w[2] = {0.0, 0.0};
            OWN(i) {
                const double xi = a.x[i];
                const double xn = rowdot<false>(a, a.i64.M, a.i64.ms, i, a.x, a.yd[i]);
                const double ri = xn - xi;
                a.x1[i] = xn;
                a.res[i] = ri;
                w[0] = maxb(w[0], absb(ri));
                w[1] = maxb(w[1], absb(xn));
            }
            if (!grid_reduce<2, 3u>(a, bar, w, tot)) return;
            ++sweeps;
            const double mr = tot[0], mx = tot[1];
            if (!isfinite(mr) || !isfinite(mx)) {  // as the sweeps would: non-finite
                status = 2;
                done = true;
                break;
            }
            if (!(mr > a.jtol * mx)) {  // x' (in x1) meets the criterion
                status = 0;
                done = true;
                break;
            }
            if (round == MAX_ROUNDS) break;
            if (round > 0 && !(mr < 0.5 * prev)) fp64 = true;  // the FP32 corrections stopped paying
            prev = mr;
            const int k = fp64 ? bicgstab(a, a.i64, 0.5 * a.jtol * mx, 64, bar, tot, lo, hi)
                    : a.tile ? bicgstab_tile<OWN_RHO>(a, TOL32 * mr, 16, bar, tot, lo, hi)
                             : bicgstab(a, a.i32, TOL32 * mr, 16, bar, tot, lo, hi);
            if (k < 0) return;
            its += k;
            // x += d (the shared-memory solve has added its d)
            if (fp64)
                OWN(i) a.x[i] += a.i64.d[i];
            else if (!a.tile)
                OWN(i) a.x[i] += (double)a.i32.d[i];
            if (!grid_sync(a, bar, tot)) return;
        }
    }
    // Jacobi sweeps from x (zero without Krylov) until one changes x by <= jtol
    // max |x'|, tested after every sweep
    double *xi = a.x, *xo = a.x1;
    if (done) {
        xi = a.x1;  // the result
    } else {
        for (int m = 0;;) {
            double w4[2] = {0.0, 0.0};
            OWN(i) {
                const double xn = rowdot<false>(a, a.i64.M, a.i64.ms, i, xi, a.yd[i]);
                w4[0] = maxb(w4[0], absb(xn - xi[i]));
                w4[1] = maxb(w4[1], absb(xn));
                xo[i] = xn;
            }
            if (!grid_reduce<2, 3u>(a, bar, w4, tot)) return;
            const double t4[2] = {tot[0], tot[1]};
            double *const tmp = xi;
            xi = xo;
            xo = tmp;
            ++m;
            ++sweeps;
            if (!isfinite(t4[0]) || !isfinite(t4[1])) {
                status = 2;
                break;
            }
            if (!(t4[0] > a.jtol * t4[1])) {
                status = 0;
                break;
            }
            if (m >= a.jmax) break;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.ctl[W_ITS] = (unsigned)its;
        a.ctl[W_SWEEPS] = (unsigned)sweeps;
        a.ctl[W_STATUS] = (unsigned)status;
        a.ctl[W_XSEL] = xi == a.x1 ? 1u : 0u;
    }
}

// blocks of the cooperative launch on the current device: SMs x resident
// blocks per SM (at most OS_BLOCKS_PER_SM), cached per device
cudaError_t os_blocks(const void *kernel, bool own_rho, int *nb)
{
    static std::atomic<int> caches[2][64];
    std::atomic<int> *const cache = caches[own_rho];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool cached = dev >= 0 && dev < 64;
    if (cached && (*nb = cache[dev].load(std::memory_order_acquire)) > 0) return cudaSuccess;
    int sms = 0, coop = 0, per = 0;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev)) != cudaSuccess) return e;
    if (!coop) return cudaErrorNotSupported;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, RT_, 0)) != cudaSuccess) return e;
    if (per < 1) return cudaErrorLaunchOutOfResources;
    *nb = std::min(MAXB, sms * std::min(per, OS_BLOCKS_PER_SM));
    if (cached) cache[dev].store(*nb, std::memory_order_release);
    return cudaSuccess;
}

// Dynamic shared memory of the FP32 halo solve: three halo buffers of hcap and
// two own-range vectors of rows floats, plus the block's 27 planes of rows
// (*msm = 1) when that fits too, beside the kernel's static shared memory on
// the current device, with the kernel's attribute raised to it; 0 (the
// global-memory solve) when even the halos do not fit.
cudaError_t os_tile_smem(const void *kernel, int hcap, int rows, int threads, size_t *smem, int *msm)
{
    *smem = 0;
    *msm = 0;
    int dev = 0, optin = 0, per = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return e;
    cudaFuncAttributes fa{};
    if ((e = cudaFuncGetAttributes(&fa, kernel)) != cudaSuccess) return e;
    const size_t base = sizeof(float) * (3 * (size_t)hcap + 2 * (size_t)rows);
    const size_t full = base + sizeof(float) * 27 * (size_t)rows;
    if (base + fa.sharedSizeBytes > (size_t)optin) return cudaSuccess;
    const bool rows_too = full + fa.sharedSizeBytes <= (size_t)optin;
    const size_t want = rows_too ? full : base;
    if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)want)) != cudaSuccess)
        return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, want)) != cudaSuccess) return e;
    if (per >= 1) {
        *smem = want;
        *msm = rows_too;
    }
    return cudaSuccess;
}

// work layout in doubles: x, x1, res, yd (4 n); FP64 BiCGSTAB vectors (7 n);
// FP64 rows (27 n); FP32 vectors and rows (34 n4 floats = 17 n4, n4 = n rounded
// up to 4, so that every FP32 vector and plane starts on 16 bytes); control
// words; arrival packets
constexpr int64_t F64_VECS = 11, F64_ROWS = 27, F32_DOUBLES = 17;

int64_t round4(int64_t v) { return (v + 3) & ~(int64_t)3; }

}  // namespace

int64_t nn_os_work_elems(int nvox)
{
    return (F64_VECS + F64_ROWS) * (int64_t)nvox + F32_DOUBLES * round4(nvox) + CTL_WORDS + 2 * (int64_t)PW * MAXB + 1;
}

cudaError_t nn_os_solve(const NnOs &o, cudaStream_t st, double **x_out, int *krylov_its, int *sweeps, int *status)
{
    *status = 1;
    *krylov_its = 0;
    *sweeps = 0;
    const int n = o.nvox;
    if ((int64_t)o.n1 * o.n2 * o.n3 != (int64_t)n || n < 1) return cudaErrorInvalidValue;
    int nb = 0;
    const void *const kernel = o.own_rho ? (const void *)k_os_solve<true> : (const void *)k_os_solve<false>;
    cudaError_t e = os_blocks(kernel, o.own_rho != 0, &nb);
    if (e != cudaSuccess) return e;
    Kv a{};
    a.n = n;
    a.sph = o.sph;
    a.n1 = o.n1;
    a.n2 = o.n2;
    a.n3 = o.n3;
    a.L27 = o.L27;
    a.eps = o.eps;
    a.y = o.y;
    double *w = o.work;
    const int64_t N = n, N4 = round4(n);
    a.x = w;
    a.x1 = w + N;
    a.res = w + 2 * N;
    a.yd = w + 3 * N;
    double **slots64[] = {&a.i64.d, &a.i64.r, &a.i64.rh, &a.i64.p, &a.i64.v, &a.i64.s, &a.i64.t};
    for (int q = 0; q < 7; ++q) *slots64[q] = w + (4 + q) * N;
    a.i64.M = w + F64_VECS * N;
    a.i64.ms = N;
    float *f = reinterpret_cast<float *>(w + (F64_VECS + F64_ROWS) * N);
    float **slots32[] = {&a.i32.d, &a.i32.r, &a.i32.rh, &a.i32.p, &a.i32.v, &a.i32.s, &a.i32.t};
    for (int q = 0; q < 7; ++q) *slots32[q] = f + q * N4;
    a.i32.M = f + 7 * N4;
    a.i32.ms = N4;
    a.n4 = N4;
    // control words and packets on a 16-byte boundary (the work space starts on one)
    const int64_t c0 = ((F64_VECS + F64_ROWS) * N + F32_DOUBLES * N4 + 1) & ~(int64_t)1;
    a.ctl = reinterpret_cast<unsigned *>(w + c0);
    a.pk = reinterpret_cast<unsigned long long *>(w + c0 + CTL_WORDS);
    a.jtol = o.jtol;
    a.krylov = o.krylov;
    a.kmax = std::max(1, o.kmax);
    a.jmax = std::max(1, o.jmax);
    a.stall = o.stall;
    a.rows = (int)round4((N + nb - 1) / nb);
    // stencil reach in voxel index: n2 n3 + n3 + 1, and on the spherical grid also
    // the k neighbours across the phi seam (n3 - 1 away); across the cylindrical
    // seam j neighbours are (n2 - 1) n3 away: the halo takes them in (2 n2 n3)
    // where that fits with the rows, else they are read past it behind a barrier
    // of their own (65^3 voxels)
    size_t smem = 0;
    const int threads = std::min(RT_, std::max(128, (a.rows + 31) & ~31));
    auto halo = [&](int64_t reach) {
        a.halo = (int)std::min<int64_t>(reach, N);
        a.hcap = (int)round4(std::min<int64_t>(N4, (int64_t)a.rows + 2 * (int64_t)a.halo + 8));
        return os_tile_smem(kernel, a.hcap, a.rows, threads, &smem, &a.msm);
    };
    const int64_t n23 = (int64_t)o.n2 * o.n3;
    if ((e = halo(o.sph ? n23 + 2 * o.n3 : 2 * n23)) != cudaSuccess) return e;
    if (!o.sph && !a.msm) {
        if ((e = halo(n23 + o.n3 + 1)) != cudaSuccess) return e;
        a.far = 1;
    }
    a.tile = smem > 0;
    if ((e = cudaMemsetAsync(a.ctl, 0, 8 * (size_t)(CTL_WORDS + 2 * PW * nb), st)) != cudaSuccess) return e;
    void *args[] = {&a};
    if ((e = cudaLaunchCooperativeKernel(kernel, dim3(nb), dim3(threads), args, smem, st)) != cudaSuccess)
        return e;
    unsigned h[W_N];
    if ((e = cudaMemcpyAsync(h, a.ctl, sizeof(h), cudaMemcpyDeviceToHost, st)) != cudaSuccess) return e;
    if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
    if (h[W_FAIL] != 0u) {
        *status = 3;
        return cudaSuccess;
    }
    *krylov_its = (int)h[W_ITS];
    *sweeps = (int)h[W_SWEEPS];
    *status = (int)h[W_STATUS];
    *x_out = h[W_XSEL] ? a.x1 : a.x;
    return cudaSuccess;
}

}  // namespace rtk
