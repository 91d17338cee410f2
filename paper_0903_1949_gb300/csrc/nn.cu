// nn.cu -- nearest-neighbour approximate Lambda operator (3^3 neighbour voxels
// built exactly, Sect. 2 and 3.2.1) and its operator-splitting step.
//
// L27[q nvox + v] = dJ_v / dS_u for the voxel u at offset (q/9 - 1, (q/3)%3 - 1,
// q%3 - 1) of v in (i, j, k), the phi index periodic (axis 3 spherical, axis 2
// cylindrical); 27 planes of n_vox, so that the sweeps read them coalesced.  Along a characteristic I_s = E_s I_{s-1} + alpha_s S_prev +
// beta_s S_{v_s} + gamma_s S_{v_{s+1}}, so the derivatives d_u = dI_s/dS_u obey
// d_u <- E_s d_u + (the weight of S_u in segment s's increment).  One thread
// per characteristic carries d_u for the NNW most recently touched voxels (the
// least recently touched makes room when the window is full) and emits, per segment,
// c_s d_u with u's neighbour slot of v_s (c_s = w_Omega l_s / L_{Omega v_s});
// one warp per piece of a voxel's ownership list sums them in list order.  The
// OS step (I - (1-eps) L*) x = y is solved in nn_krylov.cu.  All FP64, and the FP64
// pipe is the bound: per segment 16 products with E, 16 with c, 3 additions, and
// the weights, which a kernel of their own evaluates sorted by branch.  Measured
// for 6.5e6 segments (33 x 17 x 33 voxels, 64 solid angles): weights and walk
// 2.0 ms (2.8 ms with the weights in the walk and a predicated addition per window
// entry), gather 0.5 ms (1.0 ms with a thread per piece).
#include <cuda_runtime.h>
#include <stdint.h>

#include "coef.cuh"
#include "rt_internal.h"

namespace rtk {
namespace {

constexpr int NNW = RTK_NNW;

struct Ijk {
    int i, j, k;
};

__device__ __forceinline__ Ijk decode(int v, int n2, int n3)
{
    Ijk r;
    r.k = v % n3;
    r.j = (v / n3) % n2;
    r.i = v / (n2 * n3);
    return r;
}

// neighbour slot of b in a's 3x3x3 neighbourhood, or -1
__device__ __forceinline__ int slot_of(const Ijk &a, const Ijk &b, int sph, int n2, int n3)
{
    int d0 = b.i - a.i, d1 = b.j - a.j, d2 = b.k - a.k;
    if (sph) {
        if (d2 == n3 - 1) d2 = -1;
        else if (d2 == 1 - n3) d2 = 1;
    } else {
        if (d1 == n2 - 1) d1 = -1;
        else if (d1 == 1 - n2) d1 = 1;
    }
    if (d0 < -1 || d0 > 1 || d1 < -1 || d1 > 1 || d2 < -1 || d2 > 1) return -1;
    return (d0 + 1) * 9 + (d1 + 1) * 3 + (d2 + 1);
}

// Interpolation weights (E, alpha, beta, gamma) of the block's segments for chi.
// The FP64 pipe bounds the walk, and a warp of consecutive segments mixes small
// and large optical depths, parabolas and lines, and so pays for every branch of
// Coef64Series on each of them.  Here a block sorts COEF_TILE segments into the four
// kinds first; every warp then runs one branch.
constexpr int COEF_TILE = 1024;

__global__ void __launch_bounds__(256) k_nn_coef(NnWalk a, int64_t nseg)
{
    __shared__ double sx[COEF_TILE], sp[COEF_TILE];
    __shared__ uint16_t idx[4][COEF_TILE];
    __shared__ int cnt[4];
    for (int64_t t0 = blockIdx.x * (int64_t)COEF_TILE; t0 < nseg; t0 += (int64_t)gridDim.x * COEF_TILE) {
        if (threadIdx.x < 4) cnt[threadIdx.x] = 0;
        __syncthreads();
        for (int i = threadIdx.x; i < COEF_TILE && t0 + i < nseg; i += 256) {
            const int64_t s = a.seg_lo + t0 + i;
            const uint32_t w = a.vox[s];
            const bool para = a.pbits ? ((a.pbits[s >> 5] >> (s & 31)) & 1u) != 0u : (w & RTK_PARA) != 0u;
            const double x = a.chi[w & RTK_VOXMASK] * a.len64[s];
            sx[i] = x;
            sp[i] = para ? a.chi[a.vox[s + 1] & RTK_VOXMASK] * a.len64[s + 1] : 0.0;
            const int k = (x < 0.5 ? 0 : 2) + (para ? 1 : 0);
            idx[k][atomicAdd(cnt + k, 1)] = (uint16_t)i;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 4; ++k)
            for (int j = threadIdx.x; j < cnt[k]; j += 256) {
                const int i = idx[k][j];
                double E, al, be, ga;
                Coef64Series::eval(sx[i], sp[i], (k & 1) != 0, E, al, be, ga);
                double2 *o = reinterpret_cast<double2 *>(a.cw + t0 + i);
                o[0] = make_double2(E, al);
                o[1] = make_double2(be, ga);
            }
        __syncthreads();
    }
}

// A voxel in the window as one integer: (i, j, k) in 10 + 11 + 11 bits where the
// grid allows it, else its index.
template <bool PACK>
__device__ __forceinline__ int cell_of(int v, const Ijk &c)
{
    return PACK ? (int)((unsigned)c.i << 22 | (unsigned)c.j << 11 | (unsigned)c.k) : v;
}
template <bool PACK>
__device__ __forceinline__ Ijk cell_ijk(int p, int n2, int n3)
{
    return PACK ? Ijk{(int)((unsigned)p >> 22), (p >> 11) & 2047, p & 2047} : decode(p, n2, n3);
}

// The NNW most recently touched voxels of a characteristic, newest first, and
// their derivatives; an empty entry is NOCELL.
constexpr int NOCELL = -1;
struct Window {
    int cell[NNW];
    double d[NNW];
};

// Moves cell u to the front (d as it was, 0 when it is new, the oldest entry
// making room): the entries before it shift by one.  Fixed positions make the
// three additions of a step FP64 operations on named registers.
__device__ __forceinline__ void win_front(Window &W, int u, bool on)
{
    bool past = !on;  // entries behind u's old place stay
    int pc = u;
    double pd = 0.0;
#pragma unroll
    for (int e = 0; e < NNW; ++e)
        if (W.cell[e] == u) pd = W.d[e];
#pragma unroll
    for (int e = 0; e < NNW; ++e) {
        const int oc = W.cell[e];
        const double od = W.d[e];
        W.cell[e] = past ? oc : pc;
        W.d[e] = past ? od : pd;
        past = past || oc == u;
        pc = oc;
        pd = od;
    }
}

template <bool PACK>
__global__ void __launch_bounds__(128) k_nn_walk(NnWalk a)
{
    const int64_t r = a.r_lo + blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (r >= a.r_hi) return;
    const int64_t s0 = a.ray_off[r], s1 = a.ray_off[r + 1];
    const int ang = a.ray_angle[r];
    const double wq = a.wt[ang];
    const double *invLq = a.invL + (int64_t)ang * a.nvox;
    Window W;
#pragma unroll
    for (int e = 0; e < NNW; ++e) {
        W.cell[e] = NOCELL;
        W.d[e] = 0.0;
    }
    uint32_t w = a.vox[s0];
    Ijk cv = decode((int)(w & RTK_VOXMASK), a.n2, a.n3);
    bool ahead = false;  // this segment's voxel is in front already (touched by the one before)
    for (int64_t s = s0; s < s1; ++s) {
        const int v = (int)(w & RTK_VOXMASK);
        const bool para = a.pbits ? ((a.pbits[s >> 5] >> (s & 31)) & 1u) != 0u : (w & RTK_PARA) != 0u;
        const bool run0 = (w & (RTK_RAYSTART | RTK_RESTART)) != 0u;
        const uint32_t wn = s + 1 < s1 ? a.vox[s + 1] : 0u;
        const double2 *cw = reinterpret_cast<const double2 *>(a.cw + (s - a.seg_lo));
        const double2 Ea = __ldcs(cw), bg = __ldcs(cw + 1);
        const double E = Ea.x, al = Ea.y, be = bg.x, ga = bg.y;
        const double c = wq * a.len64[s] * invLq[v];
#pragma unroll
        for (int e = 0; e < NNW; ++e) W.d[e] = __dmul_rn(W.d[e], E);
        // S_prev (in front, or second when v was touched ahead), S_v and S_next
        win_front(W, cell_of<PACK>(v, cv), !ahead);
        if (!run0) W.d[1] = __dadd_rn(W.d[1], al);
        W.d[0] = __dadd_rn(W.d[0], run0 ? __dadd_rn(al, be) : be);  // S_0 := S_1 at the start of a run
        const int vn = (int)(wn & RTK_VOXMASK);
        const Ijk cn = decode(vn, a.n2, a.n3);
        win_front(W, cell_of<PACK>(vn, cn), para);
        if (para) W.d[0] = __dadd_rn(W.d[0], ga);
        ahead = para;
        const int64_t o = (s - a.seg_lo) * NNW;
        // the segment's 16 slots as one 16-byte store, its 16 values as eight
        unsigned sw[4] = {0u, 0u, 0u, 0u};
        double2 *vo = reinterpret_cast<double2 *>(a.val + o);
#pragma unroll
        for (int e = 0; e < NNW; e += 2) {
            int q[2];
#pragma unroll
            for (int h = 0; h < 2; ++h)
                q[h] = W.cell[e + h] != NOCELL
                           ? slot_of(cv, cell_ijk<PACK>(W.cell[e + h], a.n2, a.n3), a.sph, a.n2, a.n3)
                           : -1;
            sw[e >> 2] |= ((unsigned)(uint8_t)(int8_t)q[0]) << (8 * (e & 3));
            sw[(e + 1) >> 2] |= ((unsigned)(uint8_t)(int8_t)q[1]) << (8 * ((e + 1) & 3));
            vo[e >> 1] = make_double2(q[0] >= 0 ? c * W.d[e] : 0.0, q[1] >= 0 ? c * W.d[e + 1] : 0.0);
        }
        *reinterpret_cast<uint4 *>(a.slot + o) = make_uint4(sw[0], sw[1], sw[2], sw[3]);
        w = wn;
        cv = cn;
    }
}

// L27 rows of one block by gather work units (at most a fixed number of
// consecutive entries of one voxel's ownership list each, so that the outer
// voxels crossed by thousands of characteristics do not hold up the launch): one
// warp per unit, lane q holding slot q's sum.  An entry's 16 values arrive as one
// line, are laid out by slot in shared memory and added in list order, the next
// entries' lines in flight.  (A thread per unit with 27 sums in shared memory
// waited for one read-add-write after another: 0.89 ms for 6e6 segments.)
// A voxel with one unit is finished here; the units of a longer list leave their
// 27 sums in part for k_nn_gather_rows.
constexpr int NN_AHEAD = 4;  // entries a warp has in flight

__global__ void __launch_bounds__(256) k_nn_gather_units(int nvox, int64_t nunits, const int32_t *urow,
                                                         const int32_t *ubeg, const int32_t *off, const int32_t *perm,
                                                         const int8_t *slot, const double *val, double *part,
                                                         double *L27, int first)
{
    __shared__ double lay[8][NN_AHEAD][32];
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t u = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (u >= nunits) return;
    const int v = urow[u];
    const bool next_same = u + 1 < nunits && urow[u + 1] == v;
    const bool single = (u == 0 || urow[u - 1] != v) && !next_same;
    const int e0 = ubeg[u], e1 = next_same ? ubeg[u + 1] : off[v + 1];
    double acc = 0.0;
    for (int b = e0; b < e1; b += 32) {
        const int here = min(32, e1 - b);
        const int64_t p = lane < here ? (int64_t)perm[b + lane] * NNW : 0;
        for (int j = 0; j < here; j += NN_AHEAD) {
            // lanes 0..15: the values, and their slots
            double x[NN_AHEAD];
            int q[NN_AHEAD];
#pragma unroll
            for (int h = 0; h < NN_AHEAD; ++h) {
                const int64_t o = __shfl_sync(FULL, p, min(j + h, here - 1));
                const bool on = j + h < here && lane < NNW;
                x[h] = on ? val[o + lane] : 0.0;
                q[h] = on ? (int)slot[o + lane] : -1;
            }
            unsigned have[NN_AHEAD];
#pragma unroll
            for (int h = 0; h < NN_AHEAD; ++h) {
                have[h] = __reduce_or_sync(FULL, q[h] >= 0 ? 1u << q[h] : 0u);
                if (q[h] >= 0) lay[wid][h][q[h]] = x[h];
            }
            __syncwarp();
#pragma unroll
            for (int h = 0; h < NN_AHEAD; ++h)
                if ((have[h] >> lane) & 1u) acc += lay[wid][h][lane];
            __syncwarp();
        }
    }
    if (lane > 26) return;
    if (single) {
        double *e = L27 + (int64_t)lane * nvox + v;  // slot planes
        *e = first ? acc : *e + acc;
    } else {
        part[27 * u + lane] = acc;
    }
}

// Voxels with several units: their sums added in unit order, a thread per voxel
// and slot (32 threads a voxel, 27 of them at work), eight sums in flight.  (A
// thread per voxel took 158 us a block of 33 x 17 x 33 voxels and 64 solid angles.)
__global__ void __launch_bounds__(256) k_nn_gather_rows(int nvox, int nmulti, const int32_t *multi,
                                                        const int64_t *ufirst, const double *part, double *L27, int first)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int i = (int)(t >> 5), q = (int)(t & 31);
    if (i >= nmulti || q > 26) return;
    const int v = multi[i];
    const int64_t u0 = ufirst[v], u1 = ufirst[v + 1];
    double a = 0.0;
    for (int64_t u = u0; u < u1; u += 8) {
        double x[8];
#pragma unroll
        for (int h = 0; h < 8; ++h) x[h] = u + h < u1 ? part[27 * (u + h) + q] : 0.0;
#pragma unroll
        for (int h = 0; h < 8; ++h)
            if (u + h < u1) a += x[h];
    }
    double *e = L27 + (int64_t)q * nvox + v;
    *e = first ? a : *e + a;
}

__global__ void k_nn_diag(int nvox, const double *L27, double *L)
{
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v < nvox) L[v] = L27[13 * (int64_t)nvox + v];
}

__device__ __forceinline__ void max_to(double x, unsigned long long *dst)
{
    for (int o = 16; o > 0; o >>= 1) x = fmax(x, __shfl_down_sync(0xffffffffu, x, o));
    if ((threadIdx.x & 31) == 0) atomicMax(dst, (unsigned long long)__double_as_longlong(x));
}

// rows[27 v + q] = planes[q nvox + v]
__global__ void k_nn_rows(int nvox, const double *planes, double *rows)
{
    const int64_t n = 27 * (int64_t)nvox;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t v = e / 27, q = e - 27 * v;
        rows[e] = planes[q * nvox + v];
    }
}

// y = (1-eps) J + eps B - S   (ALI step, and the residual of the refinement)
__global__ void k_nn_rhs(int n, const double *S, const double *J, const double *eps, const double *B, double *y)
{
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v < n) y[v] = (1.0 - eps[v]) * J[v] + eps[v] * B[v] - S[v];
}

// y = (1-eps) Jd + r - d   (correction sweep of the refinement)
__global__ void k_nn_rhs_corr(int n, const double *d, const double *Jd, const double *r, const double *eps, double *y)
{
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v < n) y[v] = (1.0 - eps[v]) * Jd[v] + r[v] - d[v];
}

// target += x (when target is not NULL); maxrel of |x| / |ref + target_new| (ref may be NULL)
__global__ void k_nn_apply(int n, double *target, const double *x, const double *ref, double *slot,
                           unsigned long long *maxrel)
{
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    double rel = 0.0;
    if (v < n) {
        const double xv = x[v];
        double t = xv;
        if (target) {
            t = target[v] + xv;
            target[v] = t;
            if (slot) slot[v] = t;
        }
        const double den = (ref ? ref[v] : 0.0) + t;
        rel = fabs(xv) / fabs(den);
    }
    max_to(rel, maxrel);
}

unsigned nb(int64_t n, int bs) { return (unsigned)((n + bs - 1) / bs); }

}  // namespace

cudaError_t nn_walk(const NnWalk &a, int64_t nseg, cudaStream_t st)
{
    if (a.r_hi <= a.r_lo) return cudaSuccess;
    const int64_t tiles = (nseg + COEF_TILE - 1) / COEF_TILE;
    k_nn_coef<<<(unsigned)(tiles < 152 * 16 ? tiles : 152 * 16), 256, 0, st>>>(a, nseg);
    const bool pack = (int64_t)a.nvox <= (int64_t)1023 * a.n2 * a.n3 && a.n2 <= 2048 && a.n3 <= 2048;
    if (pack) k_nn_walk<true><<<nb(a.r_hi - a.r_lo, 128), 128, 0, st>>>(a);
    else k_nn_walk<false><<<nb(a.r_hi - a.r_lo, 128), 128, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t nn_gather(int nvox, const int32_t *off, const int32_t *perm, const int8_t *slot, const double *val,
                      const NnUnits &un, double *part, double *L27, int first, cudaStream_t st)
{
    if (un.nunits > 0)
        k_nn_gather_units<<<(unsigned)((un.nunits + 7) / 8), 256, 0, st>>>(nvox, un.nunits, un.urow, un.ubeg, off, perm,
                                                                              slot, val, part, L27, first);
    if (un.nmulti > 0)
        k_nn_gather_rows<<<(unsigned)((un.nmulti * 32 + 255) / 256), 256, 0, st>>>(nvox, (int)un.nmulti, un.multi, un.ufirst,
                                                                             part, L27, first);
    return cudaGetLastError();
}

cudaError_t nn_diag(int nvox, const double *L27, double *L, cudaStream_t st)
{
    k_nn_diag<<<nb(nvox, 256), 256, 0, st>>>(nvox, L27, L);
    return cudaGetLastError();
}

cudaError_t nn_rows(int nvox, const double *planes, double *rows, cudaStream_t st)
{
    k_nn_rows<<<152 * 8, 256, 0, st>>>(nvox, planes, rows);
    return cudaGetLastError();
}

cudaError_t nn_rhs(int n, const double *S, const double *J, const double *eps, const double *B, double *y,
                   cudaStream_t st)
{
    k_nn_rhs<<<nb(n, 256), 256, 0, st>>>(n, S, J, eps, B, y);
    return cudaGetLastError();
}

cudaError_t nn_rhs_corr(int n, const double *d, const double *Jd, const double *r, const double *eps, double *y,
                        cudaStream_t st)
{
    k_nn_rhs_corr<<<nb(n, 256), 256, 0, st>>>(n, d, Jd, r, eps, y);
    return cudaGetLastError();
}

cudaError_t nn_apply(int n, double *target, const double *x, const double *ref, double *slot,
                     unsigned long long *maxrel, cudaStream_t st)
{
    k_nn_apply<<<nb(n, 256), 256, 0, st>>>(n, target, x, ref, slot, maxrel);
    return cudaGetLastError();
}

}  // namespace rtk
