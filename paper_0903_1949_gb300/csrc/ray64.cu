// ray64.cu -- FP64 J-only formal solution of the ALI iteration and its
// transpose (the adjoint iteration) with streamed weights, one characteristic
// per lane.
//
// The FP64 pipe is the bound (1.06 TFLOP/s on a GB300, an instruction of a
// warp about every 19 cycles of an SM), so the layout is chosen for the fewest
// FP64 instructions per segment: a lane runs the recurrence I_k = E_k I_{k-1} +
// alpha_k S_{k-1} + beta_k S_k + gamma_k S_{k+1} down its own characteristic (5
// instructions: the source term 3, the recurrence 1, the gather weight 1).  A
// warp that spreads a characteristic over its lanes needs a scan of affine maps
// as well (12 per segment with two segments per lane).  The characteristics of
// an angle block are sorted by length, 32 of a warp have nearly the same one,
// and the streams are stored by step across them (slot = group base + 32 k +
// lane), so that every load of a step but the S lookups is one coalesced
// request; what is in flight meanwhile stands beside each kernel.  Measured on
// 65 x 33 x 65 voxels with 16 x 16 solid angles (2.1e8 segments, 37 angle blocks): the
// ALI iteration takes 3.4 ms, 7.2 ms with the warp scan; a block's march 98 us with the
// FP64 pipe 60 % active.  One sweep of the adjoint iteration on 33 x 17 x 33 x 64 (6.5e6
// segments) takes 0.18 ms with its gather, 1.9 ms with the march that evaluates the
// weights each time.
#include <cuda_runtime.h>
#include <stdint.h>

#include "coef.cuh"
#include "rt_internal.h"

namespace rtk {
namespace {

constexpr double FOUR_PI_R = 12.566370614359172953850573533118;
constexpr int STEPS_PER_WARP = 8;  // steps of a group that one warp of the set-up kernels takes at a time

// Sort keys of the characteristics, longest first: cap - length.
__global__ void k_ray_keys(int64_t n_rays, const int64_t *__restrict__ ray_off, int cap, uint32_t *__restrict__ key)
{
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n_rays; r += (int64_t)gridDim.x * blockDim.x)
        key[r] = (uint32_t)(cap - (int)(ray_off[r + 1] - ray_off[r]));
}

// order holds a block's characteristics relative to r_lo: make them global, and note their lengths.
__global__ void k_ray_order(int64_t r_lo, int64_t n, const int64_t *__restrict__ ray_off, int32_t *__restrict__ order,
                            int32_t *__restrict__ olen)
{
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = r_lo + order[r_lo + p];
        order[r_lo + p] = (int32_t)r;
        olen[r_lo + p] = (int32_t)(ray_off[r + 1] - ray_off[r]);
    }
}

// Slots of each group of 32 characteristics of one block: 32 times its longest length.
__global__ void k_group_slots(int64_t r_lo, int64_t ngroups, const int32_t *__restrict__ olen, int32_t *__restrict__ gw)
{
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g < ngroups) gw[g] = 32 * olen[r_lo + 32 * g];
}

// Set-up walks: lane = characteristic p of the group, steps in pieces of
// STEPS_PER_WARP over blockIdx.y; body(slot, segment, ray, k, n).
template <typename F>
__device__ __forceinline__ void each_slot(const Ray64 &m, F body)
{
    const int lane = threadIdx.x & 31;
    const int64_t g = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (g >= m.ngroups) return;
    const int64_t p = m.r_lo + 32 * g + lane;
    const bool have = p < m.r_hi;
    const int n = have ? m.olen[p] : 0;
    const int width = __shfl_sync(0xffffffffu, n, 0);
    const int r = have ? m.order[p] : 0;
    const int64_t s0 = have ? m.ray_off[r] : 0;
    const int64_t base = m.gbase[g] + lane;
    for (int k0 = blockIdx.y * STEPS_PER_WARP; k0 < width; k0 += gridDim.y * STEPS_PER_WARP)
        for (int k = k0; k < k0 + STEPS_PER_WARP && k < n; ++k) body(base + 32 * (int64_t)k, s0 + k, r);
}

// (word, output position) and w_Omega l / L of every slot (geometry only).
__global__ void __launch_bounds__(128) k_slot_fill(Ray64 m, const uint32_t *__restrict__ vox,
                                                   const double *__restrict__ len64, const int32_t *__restrict__ pos,
                                                   const int32_t *__restrict__ ray_angle, const double *__restrict__ wt,
                                                   const double *__restrict__ invL, int nvox, uint2 *__restrict__ wp,
                                                   double *__restrict__ cg)
{
    each_slot(m, [&](int64_t q, int64_t s, int r) {
        const uint32_t w = vox[s] & ~RTK_PARA;  // the parabola choices belong to chi, the slots to the grid
        const int a = ray_angle[r];
        wp[q] = make_uint2(w, pos ? (uint32_t)pos[s] : (uint32_t)(s - m.seg_lo));
        cg[q] = wt[a] * len64[s] * invL[(int64_t)a * nvox + (w & RTK_VOXMASK)];
    });
}

// FP64 weights (E, alpha, beta + [run start] alpha, gamma) of every slot for the
// current chi.  A CTA sorts the slots of four groups and eight steps by the branch
// of the weights they take (small or large optical depth, parabola or line), so
// that a warp runs one of them; the FP64 pipe is the bound.
constexpr int COEF_SLOTS = 128 * STEPS_PER_WARP;

__global__ void __launch_bounds__(128) k_slot_coef(Ray64 m, const uint32_t *__restrict__ vox,
                                                   const double *__restrict__ len64, const double *__restrict__ chi,
                                                   Wd4 *__restrict__ cw)
{
    __shared__ double sx[COEF_SLOTS], sp[COEF_SLOTS];
    __shared__ uint16_t idx[4][COEF_SLOTS];  // slot of the CTA, bit 15: first of a run
    __shared__ int64_t base[4];
    __shared__ int cnt[4], wmax;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t g = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const bool on = g < m.ngroups;
    const int64_t p = m.r_lo + 32 * g + lane;
    const bool have = on && p < m.r_hi;
    const int n = have ? m.olen[p] : 0;
    const int64_t s0 = have ? m.ray_off[m.order[p]] : 0;
    if (threadIdx.x == 0) wmax = 0;
    __syncthreads();
    if (lane == 0) {
        base[wid] = on ? m.gbase[g] : 0;
        atomicMax(&wmax, n);
    }
    __syncthreads();
    const int width = wmax;
    for (int k0 = blockIdx.y * STEPS_PER_WARP; k0 < width; k0 += gridDim.y * STEPS_PER_WARP) {
        if (threadIdx.x < 4) cnt[threadIdx.x] = 0;
        __syncthreads();
        for (int k = k0; k < k0 + STEPS_PER_WARP && k < n; ++k) {
            const int64_t s = s0 + k;
            const uint32_t w = vox[s];
            const bool para = (w & RTK_PARA) != 0u;  // set only when segment s + 1 continues the run
            const double x = chi[w & RTK_VOXMASK] * len64[s];
            const int i = (k - k0) * 128 + (int)threadIdx.x;
            sx[i] = x;
            sp[i] = para ? chi[vox[s + 1] & RTK_VOXMASK] * len64[s + 1] : 0.0;
            const int c = (below_one(x) ? 0 : 2) + (para ? 1 : 0);
            idx[c][atomicAdd(cnt + c, 1)] =
                (uint16_t)(i | ((w & (RTK_RAYSTART | RTK_RESTART)) ? 0x8000 : 0));
        }
        __syncthreads();
#pragma unroll
        for (int c = 0; c < 4; ++c)
            for (int j = threadIdx.x; j < cnt[c]; j += 128) {
                const int q = idx[c][j], i = q & 0x7fff, t = i & 127;
                double E, al, be, ga;
                Coef64::eval(sx[i], sp[i], (c & 1) != 0, E, al, be, ga);
                if (q & 0x8000) {  // S_0 := S_1 at the start of a run
                    be += al;
                    al = 0.0;
                }
                cw[base[t >> 5] + 32 * (int64_t)(k0 + (i >> 7)) + (t & 31)] = Wd4{E, al, be, ga};
            }
        __syncthreads();
    }
}

__device__ __forceinline__ Wd4 ldw64(const Wd4 *p)
{
    const double2 a = __ldcs(reinterpret_cast<const double2 *>(p));
    const double2 b = __ldcs(reinterpret_cast<const double2 *>(p) + 1);
    return Wd4{a.x, a.y, b.x, b.y};
}

// Forward march of one angle block: out[pos] = c_k I_k.  A characteristic is a
// serial chain and an angle block gives an SM nine warps or fewer, so what is in
// flight per lane decides: RD steps a turn, the weights of the next RD steps and S
// of those after them on their way, the words one turn further.  Against one step
// at a time with two in flight: four iterations on 65 x 33 x 65 voxels x 16 x 16
// solid angles 14.0 -> 13.7 ms, a solve on 17 x 9 x 17 x 8 x 8 1.97 -> 1.87 ms, three
// iterations on 43 x 14 x 5 x 4 x 4, where 2e3 characteristics are long, 0.26 -> 0.22.
constexpr int RD = 4;
__global__ void __launch_bounds__(64) k_march_ray64(Ray64 m, const double *__restrict__ S, const double *__restrict__ B,
                                                    double I_outer, int homog, double *__restrict__ out)
{
    const int lane = threadIdx.x & 31;
    const int64_t g = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (g >= m.ngroups) return;
    const int64_t p = m.r_lo + 32 * g + lane;
    const int n = p < m.r_hi ? m.olen[p] : 0;
    const int64_t base = m.gbase[g] + lane;
    const uint2 *wp = m.wp + base;
    const Wd4 *cw = m.cw + base;
    const double *cg = m.cg + base;
    const Wd4 zero{0.0, 0.0, 0.0, 0.0};
    if (n <= 0) return;
    auto word = [&](int k) { return k < n ? __ldcs(wp + 32 * (int64_t)k) : make_uint2(0u, 0u); };
    uint2 w0[RD], w1[RD], w2[RD];
    Wd4 c0[RD];
    double g0[RD], S0[RD], S1[RD];
#pragma unroll
    for (int j = 0; j < RD; ++j) {
        w0[j] = word(j);
        w1[j] = word(RD + j);
        w2[j] = word(2 * RD + j);
        c0[j] = j < n ? ldw64(cw + 32 * j) : zero;
        g0[j] = j < n ? __ldcs(cg + 32 * j) : 0.0;
    }
#pragma unroll
    for (int j = 0; j < RD; ++j) {
        S0[j] = j < n ? S[w0[j].x & RTK_VOXMASK] : 0.0;
        S1[j] = RD + j < n ? S[w1[j].x & RTK_VOXMASK] : 0.0;
    }
    double Sm = 0.0;
    double I = homog ? 0.0 : ((w0[0].x & RTK_CORE) ? B[w0[0].x & RTK_VOXMASK] : I_outer);
    for (int k = 0; k < n; k += RD) {
        uint2 w3[RD];
        Wd4 c1[RD];
        double g1[RD], S2[RD];
#pragma unroll
        for (int j = 0; j < RD; ++j) {
            const int q = k + RD + j;
            w3[j] = word(k + 3 * RD + j);
            c1[j] = q < n ? ldw64(cw + 32 * (int64_t)q) : zero;
            g1[j] = q < n ? __ldcs(cg + 32 * (int64_t)q) : 0.0;
            S2[j] = q + RD < n ? S[w2[j].x & RTK_VOXMASK] : 0.0;
        }
#pragma unroll
        for (int j = 0; j < RD; ++j)
            if (k + j < n) {
                I = fma(c0[j].x, I, fma(c0[j].y, Sm, fma(c0[j].z, S0[j], c0[j].w * (j + 1 < RD ? S0[j + 1] : S1[0]))));
                __stcg(out + w0[j].y, g0[j] * I);
                Sm = S0[j];
            }
#pragma unroll
        for (int j = 0; j < RD; ++j) {
            w0[j] = w1[j];
            w1[j] = w2[j];
            w2[j] = w3[j];
            c0[j] = c1[j];
            g0[j] = g1[j];
            S0[j] = S1[j];
            S1[j] = S2[j];
        }
    }
}

// The same march for the full formal solution: per segment of the block, in
// segment order, c_k I_k and c_k lambda_k with the local Lambda* element lambda_k =
// dI_k/dS_k = beta_k + gamma_{k-1} E_k (alpha_k is in beta_k at a run start, where
// the gamma before it is 0).
__global__ void __launch_bounds__(128) k_march_ray64_full(Ray64 m, const double *__restrict__ S,
                                                          const double *__restrict__ B, double I_outer, int homog,
                                                          double2 *__restrict__ out)
{
    const int lane = threadIdx.x & 31;
    const int64_t g = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (g >= m.ngroups) return;
    const int64_t p = m.r_lo + 32 * g + lane;
    const int n = p < m.r_hi ? m.olen[p] : 0;
    if (n <= 0) return;
    const int64_t base = m.gbase[g] + lane;
    const uint2 *wp = m.wp + base;
    const Wd4 *cw = m.cw + base;
    const double *cg = m.cg + base;
    double2 *o2 = out + (m.ray_off[m.order[p]] - m.seg_lo);
    const Wd4 zero{0.0, 0.0, 0.0, 0.0};
    uint32_t w0 = __ldcs(wp).x, w1 = n > 1 ? __ldcs(wp + 32).x : 0u, w2 = n > 2 ? __ldcs(wp + 64).x : 0u;
    Wd4 c0 = ldw64(cw), c1 = n > 1 ? ldw64(cw + 32) : zero;
    double g0 = __ldcs(cg), g1 = n > 1 ? __ldcs(cg + 32) : 0.0;
    double Sk = S[w0 & RTK_VOXMASK], Sn = n > 1 ? S[w1 & RTK_VOXMASK] : 0.0, Sm = 0.0, gm = 0.0;
    double I = homog ? 0.0 : ((w0 & RTK_CORE) ? B[w0 & RTK_VOXMASK] : I_outer);
    for (int k = 0; k < n; ++k) {
        const int64_t o = 32 * (int64_t)k;
        const uint32_t w3 = k + 3 < n ? __ldcs(wp + o + 96).x : 0u;
        const Wd4 c2 = k + 2 < n ? ldw64(cw + o + 64) : zero;
        const double g2 = k + 2 < n ? __ldcs(cg + o + 64) : 0.0;
        const double S2 = k + 2 < n ? S[w2 & RTK_VOXMASK] : 0.0;
        I = fma(c0.x, I, fma(c0.y, Sm, fma(c0.z, Sk, c0.w * Sn)));
        __stcg(o2 + k, make_double2(g0 * I, g0 * fma(gm, c0.x, c0.z)));
        gm = c0.w;
        Sm = Sk;
        Sk = Sn;
        Sn = S2;
        w1 = w2;
        w2 = w3;
        c0 = c1;
        c1 = c2;
        g0 = g1;
        g1 = g2;
    }
}

// Transpose of the march of one angle block: with the adjoint source a_k = c_k
// u_{v_k} of I_k (FLUX: u plus 4 pi n_Omega . gc), the adjoint intensity runs
// from the end, It_k = a_k + E_{k+1} It_{k+1}, and segment k's voxel receives
//   out[pos] = beta_k It_k + alpha_{k+1} It_{k+1} + gamma_{k-1} It_{k-1}
// (alpha is 0 at a run start and gamma at a run end, where S is not shared).
template <bool FLUX>
__global__ void __launch_bounds__(128) k_adjoint_ray64(Ray64 m, const double *__restrict__ u,
                                                       const double *__restrict__ gc, const double *__restrict__ dirs,
                                                       const int32_t *__restrict__ ray_angle, double *__restrict__ out)
{
    const int lane = threadIdx.x & 31;
    const int64_t g = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (g >= m.ngroups) return;
    const int64_t p = m.r_lo + 32 * g + lane;
    const int n = p < m.r_hi ? m.olen[p] : 0;
    if (n <= 0) return;
    const int64_t base = m.gbase[g] + lane + 32 * (int64_t)(n - 1);  // the last segment's slot
    const uint2 *wp = m.wp + base;
    const Wd4 *cw = m.cw + base;
    const double *cg = m.cg + base;
    const Wd4 zero{0.0, 0.0, 0.0, 0.0};
    double nx = 0.0, ny = 0.0, nz = 0.0;
    if (FLUX) {
        const int a = ray_angle[m.order[p]];
        nx = dirs[3 * a];
        ny = dirs[3 * a + 1];
        nz = dirs[3 * a + 2];
    }
    auto src = [&](uint32_t w) {
        const int64_t v = w & RTK_VOXMASK;
        double x = u[v];
        if (FLUX) x += FOUR_PI_R * (nx * gc[3 * v] + ny * gc[3 * v + 1] + nz * gc[3 * v + 2]);
        return x;
    };
    uint2 w0 = __ldcs(wp), w1 = n > 1 ? __ldcs(wp - 32) : make_uint2(0u, 0u);
    uint2 w2 = n > 2 ? __ldcs(wp - 64) : make_uint2(0u, 0u);
    Wd4 c0 = ldw64(cw), c1 = n > 1 ? ldw64(cw - 32) : zero;
    double g0 = __ldcs(cg), g1 = n > 1 ? __ldcs(cg - 32) : 0.0;
    double u0 = src(w0.x), u1 = n > 1 ? src(w1.x) : 0.0;
    double It = 0.0, En = 0.0, an = 0.0, part = 0.0;
    uint32_t op = 0;
    for (int k = 0; k < n; ++k) {  // k-th segment from the end
        const int64_t o = -32 * (int64_t)k;
        const uint2 w3 = k + 3 < n ? __ldcs(wp + o - 96) : make_uint2(0u, 0u);
        const Wd4 c2 = k + 2 < n ? ldw64(cw + o - 64) : zero;
        const double g2 = k + 2 < n ? __ldcs(cg + o - 64) : 0.0;
        const double u2 = k + 2 < n ? src(w2.x) : 0.0;
        const double Ik = fma(En, It, g0 * u0);
        if (k) __stcg(out + op, fma(c0.w, Ik, part));  // the segment behind this one is complete now
        part = fma(c0.z, Ik, an * It);
        op = w0.y;
        It = Ik;
        En = c0.x;
        an = c0.y;
        u0 = u1;
        u1 = u2;
        w0 = w1;
        w1 = w2;
        w2 = w3;
        c0 = c1;
        c1 = c2;
        g0 = g1;
        g1 = g2;
    }
    __stcg(out + op, part);
}

unsigned rblocks(int64_t n, int per)
{
    return (unsigned)((n + per - 1) / per);
}

unsigned rcap(int64_t n)
{
    int64_t b = (n + 255) / 256;
    if (b > 152 * 32) b = 152 * 32;
    return (unsigned)(b > 0 ? b : 1);
}

// set-up kernels: groups over x, pieces of the groups' steps over y
dim3 slot_grid(const Ray64 &m) { return dim3(rblocks(32 * m.ngroups, 128), 8); }

}  // namespace

cudaError_t ray64_keys(int64_t n_rays, const int64_t *ray_off, int cap, uint32_t *key, cudaStream_t st)
{
    k_ray_keys<<<rcap(n_rays), 256, 0, st>>>(n_rays, ray_off, cap, key);
    return cudaGetLastError();
}

cudaError_t ray64_order(int64_t r_lo, int64_t n, const int64_t *ray_off, int32_t *order, int32_t *olen, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    k_ray_order<<<rcap(n), 256, 0, st>>>(r_lo, n, ray_off, order, olen);
    return cudaGetLastError();
}

cudaError_t ray64_group_slots(int64_t r_lo, int64_t ngroups, const int32_t *olen, int32_t *gw, cudaStream_t st)
{
    if (ngroups <= 0) return cudaSuccess;
    k_group_slots<<<rblocks(ngroups, 256), 256, 0, st>>>(r_lo, ngroups, olen, gw);
    return cudaGetLastError();
}

cudaError_t ray64_fill(const Ray64 &m, const uint32_t *vox, const double *len64, const int32_t *pos,
                       const int32_t *ray_angle, const double *wt, const double *invL, int nvox, cudaStream_t st)
{
    if (m.ngroups <= 0) return cudaSuccess;
    k_slot_fill<<<slot_grid(m), 128, 0, st>>>(m, vox, len64, pos, ray_angle, wt, invL, nvox, m.wp, m.cg);
    return cudaGetLastError();
}

cudaError_t ray64_coef(const Ray64 &m, const uint32_t *vox, const double *len64, const double *chi, cudaStream_t st)
{
    if (m.ngroups <= 0) return cudaSuccess;
    k_slot_coef<<<slot_grid(m), 128, 0, st>>>(m, vox, len64, chi, m.cw);
    return cudaGetLastError();
}

cudaError_t ray64_march(const Ray64 &m, const double *S, const double *B, double I_outer, int homog, double *out,
                        cudaStream_t st)
{
    if (m.ngroups <= 0) return cudaSuccess;
    k_march_ray64<<<rblocks(32 * m.ngroups, 64), 64, 0, st>>>(m, S, B, I_outer, homog, out);
    return cudaGetLastError();
}

cudaError_t ray64_full(const Ray64 &m, const double *S, const double *B, double I_outer, int homog, double2 *out,
                       cudaStream_t st)
{
    if (m.ngroups <= 0) return cudaSuccess;
    k_march_ray64_full<<<rblocks(32 * m.ngroups, 128), 128, 0, st>>>(m, S, B, I_outer, homog, out);
    return cudaGetLastError();
}

cudaError_t ray64_adjoint(const Ray64 &m, const double *u, const double *gc, const double *dirs,
                          const int32_t *ray_angle, double *out, cudaStream_t st)
{
    if (m.ngroups <= 0) return cudaSuccess;
    const unsigned grid = rblocks(32 * m.ngroups, 128);
    if (gc) k_adjoint_ray64<true><<<grid, 128, 0, st>>>(m, u, gc, dirs, ray_angle, out);
    else k_adjoint_ray64<false><<<grid, 128, 0, st>>>(m, u, gc, dirs, ray_angle, out);
    return cudaGetLastError();
}

}  // namespace rtk
