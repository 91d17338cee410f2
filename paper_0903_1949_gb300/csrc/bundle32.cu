// bundle32.cu -- J-only mixed-precision formal solution in bundles of
// neighbouring characteristics (the hot loop of the mixed ALI iteration).
//
// What bounds it: the weight stream, 16 bytes a segment from HBM.  The march of
// fs_sw.cu takes the characteristics in launch order, looks S up once per
// segment and stores c I once per segment at its place in the voxels' lists;
// these are two requests to L2 of 32 bytes each for 4 bytes used, and they, not
// the stream, bound it.
//
// Here the characteristics of one direction are sorted by the place of their
// middle voxel along a space-filling (Morton) curve, and a CTA takes a bundle of
// up to BUN_CAP segments of neighbours.  They cross each other's voxels: a
// bundle of 5.9e3 segments of 65 x 33 x 65 voxels holds 1.5e3 different ones
// (2.9e3 on 65^3 cylindrical voxels).  So S is fetched once per voxel of the
// bundle into shared memory, the lines are marched out of shared memory, c I goes
// to its place in the bundle's own lists in shared memory, and a voxel's values
// are added there (compensated); one sum per voxel and bundle goes to L2, to
// its place in the voxel order of a part of the solid angles, and the gather of
// a part adds a quarter as many values.  A voxel with more than BUN_RUN values
// in a bundle is split into units, and units of equal length lie side by side, a
// warp's values 32 places apart: without the order by length the additions took
// twice the instructions.
//
// Below 1000 solid angles a unit's sum is two floats (BUN_PAIR in rt_api.cu), and only
// grids on which the tables pay take this march by default (bun_pays there).
//
// Measured, one GB300, per formal solution against the march in launch order: 8.4e8
// segments (65 x 33 x 65 voxels x 32 x 32 solid angles) 6.76 -> 4.33 ms, 2.1e8 (16 x 16,
// two floats) 1.76 -> 1.24, 2e8 (65^3 cylindrical x 16 x 16) 1.60 -> 1.91, or 1.52 with
// one float.  A part of 5.7e6 segments takes 41 to 43 us and moves 25.4 bytes a segment to
// and from HBM (20 of them its stream), 3.4 of 6.8 TB/s; with S, the sums and the scan
// left out the same stream took 3.8 of the 4.3 ms, so what is left is the HBM latency
// that 32 warps an SM (64 registers, 40 kB of shared memory a bundle) cover.  Not
// better: two segments a lane and five CTAs an SM (4.8 ms), persistent CTAs that fetch
// the next bundle's S during the additions (4.9), bundles of 8192 (5.5 without the order
// by length).  The tables cost about 0.09 s once per grid at 8.4e8 segments.
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "coef.cuh"
#include "rt_internal.h"

namespace rtk {
namespace {

constexpr int K = BUN_K;       // consecutive segments per lane
constexpr int T = 32 * K;      // segments of a warp's tile
constexpr int NW = BUN_WARPS;  // warps of a bundle, one share of whole characteristics each
constexpr int UT = 1024;       // threads of the table kernel
constexpr int SORT_CAP = 8192;  // keys of the table kernel's sorts
constexpr int UE = SORT_CAP / UT;
// places of a bundle: units by falling length, 32 to a group, a group's values 32 apart;
// the groups' padding is below 32 times the longest unit.  One more for what is not kept.
constexpr int PLACES = BUN_CAP + 32 * BUN_RUN;
// word of a segment: 4 x unit | start | core << 1 | 4 x place << 16 (byte offsets)
constexpr uint32_t WSTART = 1u, WCORE = 2u, WUNIT = 0x7ffcu;
constexpr uint32_t WNONE = (uint32_t)(4 * PLACES) << 16;
constexpr unsigned FULL = 0xffffffffu;
static_assert(BUN_CAP <= SORT_CAP && 4 * BUN_CAP <= 0x8000 && 4 * PLACES < 0x10000, "fields of a segment's word");

// slot of segment i of a share whose slots begin at `base`: lane i / K mod 32 takes K
// consecutive segments of a tile, and each of its K loads is one run over the lanes
__device__ __forceinline__ int64_t slot_of(int64_t base, int i)
{
    const int t = i / T, q = i - t * T;
    return base + t * T + (q % K) * 32 + q / K;
}
// first slot of share k of a part, which begins at the part's segment s: shares are padded
// to whole tiles
__device__ __forceinline__ int64_t share_base(const Bun32 &m, int64_t k, int s)
{
    return m.slot_lo + (int64_t)(s / T) * T + k * T;
}

__device__ __forceinline__ uint32_t spread3(uint32_t x)  // bits of x (10 at most) at every third place
{
    uint32_t z = 0;
    for (int b = 0; b < 10; ++b) z |= ((x >> b) & 1u) << (3 * b);
    return z;
}

// Sort keys: direction, then the middle voxel along the Morton curve of its indices.
__global__ void k_bun_keys(const int64_t *ray_off, int64_t r_lo, int64_t n, const uint32_t *vox, const int32_t *ray_angle,
                           int a0, int n2, int n3, int drop, int mbits, int shift, uint32_t *key)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = r_lo + i, a = ray_off[r], e = ray_off[r + 1];
        uint64_t z = 0;
        if (e > a) {
            const uint32_t v = vox[a + (e - a) / 2] & RTK_VOXMASK;
            const uint32_t vk = v % (uint32_t)n3, vj = v / (uint32_t)n3 % (uint32_t)n2, vi = v / (uint32_t)n3 / (uint32_t)n2;
            z = spread3(vi >> drop) | spread3(vj >> drop) << 1 | spread3(vk >> drop) << 2;
        }
        key[i] = (uint32_t)((((uint64_t)(ray_angle[r] - a0) << mbits) | z) >> shift);
    }
}

__global__ void k_bun_maxlen(int64_t n, const int64_t *ray_off, int32_t *mx)
{
    int m = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        m = max(m, (int)(ray_off[i + 1] - ray_off[i]));
    m = __reduce_max_sync(FULL, m);
    if ((threadIdx.x & 31) == 0) atomicMax(mx, m);
}

// Bounds of the shares: share k holds the characteristics whose first segment,
// in sorted order, lies in [k sub, (k + 1) sub) of the part.
__global__ void k_bun_bounds(Bun32 m, int64_t nseg, int32_t *sray, int32_t *sseg)
{
    const int64_t nsub = (int64_t)m.nbun * NW;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k <= nsub; k += (int64_t)gridDim.x * blockDim.x) {
        const int64_t key = m.seg_lo + (k * m.sub < nseg ? k * m.sub : nseg);
        int64_t lo = m.r_lo, hi = m.r_hi;
        while (lo < hi) {
            const int64_t mid = lo + ((hi - lo) >> 1);
            if (m.boff[mid] < key) lo = mid + 1;
            else hi = mid;
        }
        sray[k] = (int32_t)(lo - m.r_lo);
        sseg[k] = (int32_t)(m.boff[lo] - m.seg_lo);
    }
}

// Inclusive scan of one int per thread over the CTA (sum or maximum).
template <bool MAX>
__device__ __forceinline__ int cta_scan(int x, int *sh)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, x, o);
        if (lane >= o) x = MAX ? max(x, y) : x + y;
    }
    if (lane == 31) sh[w] = x;
    __syncthreads();
    if (w == 0) {
        int s = sh[lane];
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULL, s, o);
            if (lane >= o) s = MAX ? max(s, y) : s + y;
        }
        sh[lane] = s;
    }
    __syncthreads();
    if (w > 0) x = MAX ? max(x, sh[w - 1]) : x + sh[w - 1];
    __syncthreads();
    return x;
}

// Place of key i: the bank (low 5 bits) exchanged by a linear map of bits 5 to 7, such
// that 32 threads with 8 keys each, at any power of two apart, read 32 banks.
__device__ __forceinline__ int padded(int i)
{
    return i ^ ((i >> 3) & 4) ^ ((i >> 6 & 1) * 9) ^ ((i >> 7 & 1) * 18);
}

// Steps j = 4 s, 2 s, s (as far as they exist: j < k) of the bitonic merge of size k
// on 8 keys at distance s; `first` of 2, 1, 0 skips the steps above it.
template <typename KEY>
__device__ __forceinline__ void merge8(KEY *key, int t, int s, int k, int first)
{
    const int i0 = (t / s) * (8 * s) + t % s;
    KEY x[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) x[e] = key[padded(i0 + e * s)];
#pragma unroll
    for (int l = 2; l >= 0; --l) {
        if (l > first) continue;
#pragma unroll
        for (int e = 0; e < 8; ++e)
            if (!(e & (1 << l))) {
                const int f = e | (1 << l);
                const bool up = ((i0 + e * s) & k) == 0;
                if ((x[e] > x[f]) == up) {
                    const KEY y = x[e];
                    x[e] = x[f];
                    x[f] = y;
                }
            }
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) key[padded(i0 + e * s)] = x[e];
}

// N keys (a power of two, 8 at least) in increasing order.  Three steps of the bitonic
// network per pass over shared memory, on 8 keys a thread.
template <typename KEY>
__device__ __forceinline__ void cta_sort(KEY *key, int N)
{
    const int t = threadIdx.x;
    for (int k = 2; k <= N; k <<= 1) {
        int j = k >> 1;
        while (j > 0) {
            // the steps j, j / 2, j / 4 at distance s = j / 4, or the last one or two at s = 1
            const int s = j >= 4 ? j >> 2 : 1, first = j >= 4 ? 2 : (j == 2 ? 1 : 0);
            if (t < N / 8) merge8(key, t, s, k, first);
            __syncthreads();
            j = j >= 4 ? j >> 3 : 0;
        }
    }
}

template <typename KEY>
constexpr size_t units_smem()
{
    return sizeof(KEY) * SORT_CAP + sizeof(uint32_t) * SORT_CAP + 2 * sizeof(uint16_t) * (SORT_CAP + 8);
}

// One stable pass of a radix sort over the CTA: n <= SORT_CAP items get(i) go to dst in
// the order of their digit (get(i) >> shift) & (2^bits - 1), place i at dst[put(i)].  A warp
// takes a run of SORT_CAP / 32 items; items of one digit in a warp are ranked by
// __match_any_sync.
constexpr int DIGIT = 6;
struct RadixSmem {
    uint16_t cnt[UT / 32][1 << DIGIT];
    int sh[32];
};
template <typename G, typename P>
__device__ __forceinline__ void cta_radix_pass(RadixSmem &r, G get, P put, uint32_t *dst, int n, int shift, int bits)
{
    constexpr int R = SORT_CAP / UT;  // items of a thread
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, mask = (1 << bits) - 1;
    for (int d = lane; d < 1 << DIGIT; d += 32) r.cnt[w][d] = 0;
    __syncwarp();
    uint32_t x[R];
    int at[R];
#pragma unroll
    for (int q = 0; q < R; ++q) {
        const int i = w * (SORT_CAP / 32) + 32 * q + lane;
        const bool on = i < n;
        x[q] = on ? get(i) : 0u;
        const int d = on ? (int)(x[q] >> shift) & mask : 1 << DIGIT;
        const unsigned same = __match_any_sync(FULL, d), below = same & ((1u << lane) - 1u);
        const int before = on ? r.cnt[w][d] : 0;
        at[q] = before + __popc(below);
        __syncwarp();
        if (on && below == 0u) r.cnt[w][d] = (uint16_t)(before + __popc(same));
        __syncwarp();
    }
    __syncthreads();
    // first place of every (digit, warp): digits in order, a digit's warps in order
    constexpr int E = (1 << DIGIT) * (UT / 32) / UT;  // counters of a thread
    int c[E], sum = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int k = E * threadIdx.x + e;
        c[e] = r.cnt[k % (UT / 32)][k / (UT / 32)];
        sum += c[e];
    }
    int first = cta_scan<false>(sum, r.sh) - sum;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int k = E * threadIdx.x + e;
        r.cnt[k % (UT / 32)][k / (UT / 32)] = (uint16_t)first;
        first += c[e];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < R; ++q)
        if (w * (SORT_CAP / 32) + 32 * q + lane < n) dst[put(r.cnt[w][(int)(x[q] >> shift) & mask] + at[q])] = x[q];
    __syncthreads();
}

// Tables of one bundle per CTA (once per grid): its segments sorted by voxel,
// stable in the order of the march; runs of a voxel cut into units of at most
// BUN_RUN; the units sorted by falling length, so that the threads of a warp add
// equally long ones; voxel (its number among the bundle's) and place of every
// segment into its word.  The units' voxels, first places and lengths go to tv and
// tb, the different voxels in order to td, each from the bundle's first segment on.
// KEY: 32 bits hold (voxel, number in the bundle) on grids of up to 2^19 voxels; they
// are sorted by the voxel's vbits bits in radix passes (the bitonic sort, which 64-bit
// keys keep, took half of the tables' time).
template <typename KEY>
__global__ void __launch_bounds__(UT, sizeof(KEY) == 4 ? 2 : 1)
    k_bun_units(Bun32 m, int vbits, const uint32_t *__restrict__ vox, uint32_t *__restrict__ tv,
                uint32_t *__restrict__ tb, uint32_t *__restrict__ td, int32_t *__restrict__ nunit,
                int32_t *__restrict__ ndist, int *err)
{
    constexpr bool WIDE = sizeof(KEY) == 8;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int sh[32], gbase[SORT_CAP / 32];
    __shared__ RadixSmem rs;
    KEY *key = reinterpret_cast<KEY *>(smem);  // the sorted segments
    uint32_t *key2 = reinterpret_cast<uint32_t *>(key + SORT_CAP);  // sort of the units, then unit and place
    uint16_t *ustart = reinterpret_cast<uint16_t *>(key2 + SORT_CAP), *now = ustart + SORT_CAP + 8;
    const int64_t b = blockIdx.x;
    const int32_t *sr = m.sray + b * NW, *ss = m.sseg + b * NW;
    const int seg0 = ss[0], n = ss[NW] - seg0;
    if (n > BUN_CAP) {  // cannot be: sub leaves room for the longest characteristic
        if (threadIdx.x == 0) {
            *err = 1;
            nunit[b] = ndist[b] = 0;
        }
        return;
    }
    int N = 8;
    while (N < n) N <<= 1;
    if (WIDE) {
        for (int i = threadIdx.x; i < N; i += UT) key[padded(i)] = ~(KEY)0;
        __syncthreads();
    }
    const int lane = threadIdx.x & 31;
    for (int q = sr[0] + (threadIdx.x >> 5); q < sr[NW]; q += UT / 32) {
        const int64_t r = m.order[m.r_lo + q], s0 = m.ray_off[r];
        const int len = (int)(m.ray_off[r + 1] - s0), at = (int)(m.boff[m.r_lo + q] - m.seg_lo) - seg0;
        for (int i = lane; i < len; i += 32)
            key[WIDE ? padded(at + i) : at + i] = (KEY)(vox[s0 + i] & RTK_VOXMASK) << 13 | (uint32_t)(at + i);
    }
    __syncthreads();
    if constexpr (WIDE) {
        cta_sort(key, N);
    } else {
        const int passes = (vbits + DIGIT - 1) / DIGIT;
        for (int q = 0; q < passes; ++q) {
            const uint32_t *from = key;
            const bool last = q == passes - 1;
            cta_radix_pass(rs, [from](int i) { return from[i]; }, [last](int i) { return last ? padded(i) : i; }, key2, n,
                           13 + DIGIT * q, min(DIGIT, vbits - DIGIT * q));
            uint32_t *const t = key;
            key = key2;
            key2 = t;
        }
    }
    uint16_t *unit = reinterpret_cast<uint16_t *>(key2), *place = unit + SORT_CAP;
    // first places of the voxels' runs, then heads of units
    const int p0 = threadIdx.x * UE;
    auto newvox = [&](int p) { return p == 0 || key[padded(p)] >> 13 != key[padded(p - 1)] >> 13; };
    int last = -1;
    for (int e = 0; e < UE; ++e)
        if (p0 + e < n && newvox(p0 + e)) last = p0 + e;
    const int incl = cta_scan<true>(last, sh);
    int run = __shfl_up_sync(FULL, incl, 1);
    __shared__ int prev[32];
    if (lane == 31) prev[threadIdx.x >> 5] = incl;
    __syncthreads();
    if (lane == 0) run = threadIdx.x > 0 ? prev[(threadIdx.x >> 5) - 1] : -1;
    uint32_t heads = 0, fresh = 0;
    for (int e = 0; e < UE; ++e) {
        const int p = p0 + e;
        if (p >= n) break;
        if (newvox(p)) {
            run = p;
            fresh |= 1u << e;
        }
        if ((p - run) % BUN_RUN == 0) heads |= 1u << e;
    }
    const int cnt = __popc(heads), upto = cta_scan<false>(cnt, sh);
    const int cntd = __popc(fresh), uptod = cta_scan<false>(cntd, sh);
    if (threadIdx.x == UT - 1) ndist[b] = uptod;
    __shared__ int total;
    if (threadIdx.x == UT - 1) total = upto;
    int u = upto - cnt - 1, dv = uptod - cntd - 1;
    for (int e = 0, h = u; e < UE; ++e)
        if (heads >> e & 1u) ustart[++h] = (uint16_t)(p0 + e);
    __syncthreads();
    const int U = total;
    if (threadIdx.x == 0) {
        ustart[U] = (uint16_t)n;
        nunit[b] = U;
    }
    __syncthreads();
    // units by falling length: one pass over 0 .. BUN_RUN - 1
    static_assert(BUN_RUN <= 1 << DIGIT, "a length is one digit");
    cta_radix_pass(rs, [ustart](int i) { return (uint32_t)(BUN_RUN - (ustart[i + 1] - ustart[i])) << 16 | (uint32_t)i; },
                   [](int i) { return i; }, key2, U, 16, DIGIT);
    const int ng = (U + 31) / 32;  // at most SORT_CAP / 32 = 256 groups
    const int glen = (int)threadIdx.x < ng ? 32 * (BUN_RUN - (int)(key2[32 * threadIdx.x] >> 16)) : 0;
    const int gend = cta_scan<false>(glen, sh);
    if ((int)threadIdx.x < ng) gbase[threadIdx.x] = gend - glen;
    __syncthreads();
    for (int i = threadIdx.x; i < U; i += UT) {
        const int o = (int)(key2[i] & 0xffffu), s = ustart[o];
        now[o] = (uint16_t)i;
        tv[seg0 + i] = (uint32_t)(key[padded(s)] >> 13);
        tb[seg0 + i] = (uint32_t)(gbase[i >> 5] + (i & 31)) | (uint32_t)(ustart[o + 1] - s) << 16;
    }
    __syncthreads();  // key2 is free from here on
    for (int e = 0; e < UE; ++e) {
        const int p = p0 + e;
        if (p >= n) break;
        if (heads >> e & 1u) ++u;
        if (fresh >> e & 1u) td[seg0 + ++dv] = (uint32_t)(key[padded(p)] >> 13);
        const int i = (int)(key[padded(p)] & 8191u), w = now[u];
        unit[i] = (uint16_t)dv;
        place[i] = (uint16_t)(gbase[w >> 5] + (w & 31) + 32 * (p - ustart[u]));
    }
    __syncthreads();
    for (int q = sr[0] + (threadIdx.x >> 5); q < sr[NW]; q += UT / 32) {
        const int64_t r = m.order[m.r_lo + q], s0 = m.ray_off[r];
        const int len = (int)(m.ray_off[r + 1] - s0), at = (int)(m.boff[m.r_lo + q] - m.seg_lo);
        int k = 0;
        while (k + 1 < NW && sr[k + 1] <= q) ++k;
        const int64_t base = share_base(m, b * NW + k, ss[k]);
        for (int i = lane; i < len; i += 32) {
            const uint32_t w = vox[s0 + i];
            const int l = at + i - seg0;
            m.wd[slot_of(base, at + i - ss[k])] = (uint32_t)unit[l] << 2 | ((w & RTK_RAYSTART) ? WSTART : 0u) |
                                                  ((w & RTK_CORE) ? WCORE : 0u) | (uint32_t)place[l] << 18;
        }
    }
}

__global__ void k_bun_compact(Bun32 m, const uint32_t *tv, const uint32_t *tb, const uint32_t *td, uint32_t *uvox)
{
    const int64_t b = blockIdx.x;
    const int u0 = m.ub[b].x, nu = m.ub[b + 1].x - u0, d0 = m.ub[b].y, nd = m.ub[b + 1].y - d0, s = m.sseg[b * NW];
    for (int u = threadIdx.x; u < nu; u += blockDim.x) {
        uvox[u0 + u] = tv[s + u];
        m.ubeg[u0 + u] = tb[s + u];
    }
    for (int d = threadIdx.x; d < nd; d += blockDim.x) m.dvox[d0 + d] = td[s + d];
}

__global__ void k_bun_ub(int n, const int64_t *uoff, const int64_t *doff, int2 *ub, int32_t *mx)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i <= n; i += gridDim.x * blockDim.x) {
        ub[i] = make_int2((int)uoff[i], (int)doff[i]);
        if (i < n) atomicMax(mx, (int)(doff[i + 1] - doff[i]));
    }
}

// Weights of every segment for the current chi, with the gather weight folded in,
// as k_coef_stream_fold forms them (same values), to the segments' slots: a warp per
// characteristic (a warp per share waited for one characteristic after another).
__global__ void __launch_bounds__(256) k_bun_coef(Bun32 m, const uint32_t *__restrict__ vox,
                                                  const double *__restrict__ len64, const double *__restrict__ chi,
                                                  const int32_t *__restrict__ ray_angle, const double *__restrict__ wt,
                                                  const double *__restrict__ invL, int nvox)
{
    const int64_t q = m.r_lo + ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
    if (q >= m.r_hi) return;
    const int lane = threadIdx.x & 31;
    const int64_t r = m.order[q], s0 = m.ray_off[r];
    const int len = (int)(m.ray_off[r + 1] - s0), at0 = (int)(m.boff[q] - m.seg_lo);
    if (len <= 0) return;
    const int64_t k = at0 / m.sub;  // its share, by k_bun_bounds
    const int at = at0 - m.sseg[k];
    const int64_t base = share_base(m, k, m.sseg[k]);
    const int a = ray_angle[r];
    const double wa = wt[a];
    const double *iL = invL + (int64_t)a * nvox;
    for (int i = lane; i < len; i += 32) {
        const int64_t s = s0 + i;
        const uint32_t w = vox[s];
        const bool para = (w & RTK_PARA) != 0u;
        const float x = (float)(chi[w & RTK_VOXMASK] * len64[s]);
        const float p = para ? (float)(chi[vox[s + 1] & RTK_VOXMASK] * len64[s + 1]) : 0.0f;
        float E, al, be, ga;
        Coef32::eval(x, p, para, E, al, be, ga);
        if (w & (RTK_RAYSTART | RTK_RESTART)) {
            be += al;
            al = 0.0f;
        }
        const float c = (float)(wa * len64[s] * iL[w & RTK_VOXMASK]);
        float A = c * E;
        if (!(w & RTK_RAYSTART)) A = __fdividef(A, (float)(wa * len64[s - 1] * iL[vox[s - 1] & RTK_VOXMASK]));
        __stcs(m.cw + slot_of(base, at + i), make_float4(A, c * al, c * be, c * ga));
    }
}

constexpr int AHEAD = 2;  // tiles fetched to L2 ahead of the march (1, 2, 4, 8: 18.7, 18.2, 18.8, 19.6 ms)
__device__ __forceinline__ void l2_prefetch(const void *p, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// [p + a, p + b) as whole 16-byte pieces (the arrays end with 16 bytes to spare)
__device__ __forceinline__ void l2_prefetch_range(const void *p, int64_t a, int64_t b)
{
    const uintptr_t lo = ((uintptr_t)p + a) & ~(uintptr_t)15, hi = ((uintptr_t)p + b + 15) & ~(uintptr_t)15;
    if (hi > lo) l2_prefetch((const void *)lo, (uint32_t)(hi - lo));
}

__device__ __forceinline__ void st_keep(float *p, float x, float y, uint64_t pol)
{
    asm volatile("st.global.L2::cache_hint.f32 [%0], %1, %2;" ::"l"(p), "f"(x + y), "l"(pol) : "memory");
}
__device__ __forceinline__ void st_keep(float2 *p, float x, float y, uint64_t pol)
{
    asm volatile("st.global.L2::cache_hint.v2.f32 [%0], {%1, %2}, %3;" ::"l"(p), "f"(x), "f"(y), "l"(pol) : "memory");
}

// One tile of a share: K slots of this lane; past the share's end neutral weights and the
// place that is not kept.
__device__ __forceinline__ void load_tile(const float4 *cf, const uint32_t *wp, int t, int len, int lane, uint32_t (&w)[K],
                                          float4 (&c)[K])
{
    if (t + T <= len) {
#pragma unroll
        for (int j = 0; j < K; ++j) {
            w[j] = __ldcs(wp + t + 32 * j);
            c[j] = __ldcs(cf + t + 32 * j);
        }
        return;
    }
#pragma unroll
    for (int j = 0; j < K; ++j) {
        const bool ok = t + K * lane + j < len;
        w[j] = ok ? __ldcs(wp + t + 32 * j) : WNONE;
        c[j] = ok ? __ldcs(cf + t + 32 * j) : make_float4(1.f, 0.f, 0.f, 0.f);
    }
}

// One bundle per CTA: S of its units to shared memory; each warp marches its
// share, a tile of K segments per lane at a time, the lane maps I -> A I + b
// composed by a shuffle scan, the next tile's stream in flight meanwhile and the
// third one on its way to L2; the values of a unit added in the order of the
// march, compensated.  Four CTAs an SM cover each other's phases.  OUT: float or
// float2, a unit's sum with its compensation added or as a second float.
template <typename OUT>
__global__ void __launch_bounds__(32 * NW, 4) k_march_bun(Bun32 m, const double *__restrict__ S,
                                                          const double *__restrict__ B, float I_outer, int homog,
                                                          OUT *__restrict__ out)
{
    extern __shared__ __align__(16) unsigned char smem[];
    float *val = reinterpret_cast<float *>(smem), *Ss = val + PLACES + 1;
    unsigned char *sbase = reinterpret_cast<unsigned char *>(Ss);
    const int64_t b = blockIdx.x;
    const int lane = threadIdx.x & 31;
    const int64_t k = b * NW + (threadIdx.x >> 5);
    const int s0 = m.sseg[k], len = m.sseg[k + 1] - s0;
    const int64_t base = share_base(m, k, s0) + lane;
    const float4 *cf = m.cw + base;
    const uint32_t *wp = m.wd + base;
    uint64_t pol;  // the units' values stay in L2 for the gather, the streams pass
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    uint32_t w0[K], w1[K];
    float4 c0[K], c1[K];
    load_tile(cf, wp, 0, len, lane, w0, c0);
    if (lane == 0 && len > T) {
        const int n = (min(len, AHEAD * T) - 1) / T * T;
        l2_prefetch(cf + T, n * sizeof(float4));
        l2_prefetch(wp + T, n * sizeof(uint32_t));
    }
    const int2 ua = m.ub[b], ue = m.ub[b + 1];
    const int u0 = ua.x, nu = ue.x - u0, d0 = ua.y, nd = ue.y - d0;
    if (threadIdx.x == 0) {
        l2_prefetch_range(m.dvox, 4 * (int64_t)d0, 4 * (int64_t)ue.y);
        l2_prefetch_range(m.ubeg, 4 * (int64_t)u0, 4 * (int64_t)ue.x);
        l2_prefetch_range(m.upos, 4 * (int64_t)u0, 4 * (int64_t)ue.x);
    }
    for (int u = threadIdx.x; u < nd; u += 4 * 32 * NW) {  // four lookups in flight
        uint32_t v[4];
        double x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = u + q * 32 * NW < nd ? __ldcs(m.dvox + d0 + u + q * 32 * NW) : 0u;
#pragma unroll
        for (int q = 0; q < 4; ++q) x[q] = __ldg(S + v[q]);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (u + q * 32 * NW < nd) Ss[u + q * 32 * NW] = (float)x[q];
    }
    __syncthreads();
    const float I_far = homog ? 0.f : I_outer;
    float Icarry = 0.f, Sprev = 0.f;
    auto s_of = [&](uint32_t w) { return *reinterpret_cast<const float *>(sbase + (w & WUNIT)); };
    auto step = [&](const uint32_t (&w)[K], const float4 (&c)[K], uint32_t next) {
        float Sv[K];
#pragma unroll
        for (int j = 0; j < K; ++j) Sv[j] = s_of(w[j]);
        float Sp = __shfl_up_sync(FULL, Sv[K - 1], 1);
        if (lane == 0) Sp = Sprev;
        Sprev = __shfl_sync(FULL, Sv[K - 1], 31);
        float Sn = __shfl_down_sync(FULL, Sv[0], 1);
        const uint32_t wf = __shfl_sync(FULL, next, 0);
        if (lane == 31) Sn = s_of(wf);  // the next tile's first segment
        float b_[K], A[K];
#pragma unroll
        for (int j = 0; j < K; ++j) {
            b_[j] = fmaf(c[j].y, j ? Sv[j - 1] : Sp, fmaf(c[j].z, Sv[j], c[j].w * (j + 1 < K ? Sv[j + 1] : Sn)));
            A[j] = c[j].x;
            if (w[j] & WSTART) {
                float Iin = I_far;
                if ((w[j] & WCORE) && !homog) Iin = (float)B[m.dvox[d0 + ((w[j] & WUNIT) >> 2)]];
                b_[j] = fmaf(A[j], Iin, b_[j]);
                A[j] = 0.f;
            }
        }
        float LA = A[0], LB = b_[0];
#pragma unroll
        for (int j = 1; j < K; ++j) {
            LB = fmaf(A[j], LB, b_[j]);
            LA = A[j] * LA;
        }
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const float Ao = __shfl_up_sync(FULL, LA, d);
            const float Bo = __shfl_up_sync(FULL, LB, d);
            if (lane >= d) {
                LB = fmaf(LA, Bo, LB);
                LA = LA * Ao;
            }
        }
        float PA = __shfl_up_sync(FULL, LA, 1);
        float PB = __shfl_up_sync(FULL, LB, 1);
        if (lane == 0) {
            PA = 1.f;
            PB = 0.f;
        }
        float I = fmaf(PA, Icarry, PB);
#pragma unroll
        for (int j = 0; j < K; ++j) {
            I = fmaf(A[j], I, b_[j]);
            *reinterpret_cast<float *>(smem + (w[j] >> 16)) = I;
        }
        Icarry = __shfl_sync(FULL, I, 31);
    };
    for (int t = 0; t < len; t += 2 * T) {
        if (lane == 0) {  // two tiles further on, to L2
            const int n = min(2 * T, (len - t - AHEAD * T + T - 1) / T * T);
            if (n > 0) {
                l2_prefetch(cf + t + AHEAD * T, n * sizeof(float4));
                l2_prefetch(wp + t + AHEAD * T, n * sizeof(uint32_t));
            }
        }
        load_tile(cf, wp, t + T, len, lane, w1, c1);
        step(w0, c0, w1[0]);
        if (t + T >= len) break;
        load_tile(cf, wp, t + 2 * T, len, lane, w0, c0);
        step(w1, c1, w0[0]);
    }
    __syncthreads();
    for (int u = threadIdx.x; u < nu; u += 2 * 32 * NW) {  // two units a thread
        const int v = u + 32 * NW;
        const uint32_t pl = __ldcs(m.ubeg + u0 + u), ql = v < nu ? __ldcs(m.ubeg + u0 + v) : 0u;
        const int po = __ldcs(m.upos + u0 + u), qo = v < nu ? __ldcs(m.upos + u0 + v) : 0;
        const float *p = val + (pl & 0xffffu), *q = val + (ql & 0xffffu);
        const int np = (int)(pl >> 16), nq = (int)(ql >> 16);  // np >= nq: the units' lengths fall
        float s = 0.f, sc = 0.f, r = 0.f, rc = 0.f;
        int i = 0;
        for (; i < nq; ++i) {
            const float y = p[32 * i] - sc, x = s + y;
            sc = (x - s) - y;
            s = x;
            const float z = q[32 * i] - rc, a = r + z;
            rc = (a - r) - z;
            r = a;
        }
        for (; i < np; ++i) {
            const float y = p[32 * i] - sc, x = s + y;
            sc = (x - s) - y;
            s = x;
        }
        st_keep(out + po, s, -sc, pol);
        if (v < nu) st_keep(out + qo, r, -rc, pol);
    }
}

unsigned cap_grid(int64_t n)
{
    int64_t b = (n + 255) / 256;
    if (b > 152 * 32) b = 152 * 32;
    return (unsigned)(b > 0 ? b : 1);
}

// The shared-memory limit of a kernel belongs to one device: set once per device.
template <typename F>
cudaError_t allow_smem(F *f, size_t bytes, std::atomic<uint64_t> &done)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t bit = dev < 64 ? (uint64_t)1 << dev : 0;
    if (bit && (done.load(std::memory_order_acquire) & bit)) return cudaSuccess;
    e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_acq_rel);
    return e;
}

}  // namespace

cudaError_t bun_keys(const int64_t *ray_off, int64_t r_lo, int64_t n, const uint32_t *vox, const int32_t *ray_angle,
                     int a0, int n_ang, int n1, int n2, int n3, uint32_t *key, int *bits, cudaStream_t st)
{
    int vb = 0, ab = 0;
    while (vb < 31 && (1 << vb) < (n1 > n2 ? (n1 > n3 ? n1 : n3) : (n2 > n3 ? n2 : n3))) ++vb;
    const int drop = vb > 10 ? vb - 10 : 0;  // at most 10 bits an index
    while (ab < 31 && (1 << ab) < n_ang) ++ab;
    const int mbits = 3 * (vb - drop), shift = mbits + ab > 28 ? mbits + ab - 28 : 0;
    *bits = mbits + ab - shift;
    if (n > 0)
        k_bun_keys<<<cap_grid(n), 256, 0, st>>>(ray_off, r_lo, n, vox, ray_angle, a0, n2, n3, drop, mbits, shift, key);
    return cudaGetLastError();
}

cudaError_t bun_maxlen(int64_t n_rays, const int64_t *ray_off, int32_t *mx, cudaStream_t st)
{
    k_bun_maxlen<<<cap_grid(n_rays), 256, 0, st>>>(n_rays, ray_off, mx);
    return cudaGetLastError();
}

cudaError_t bun_bounds(const Bun32 &m, int64_t nseg, int32_t *sray, int32_t *sseg, cudaStream_t st)
{
    k_bun_bounds<<<cap_grid((int64_t)m.nbun * NW + 1), 256, 0, st>>>(m, nseg, sray, sseg);
    return cudaGetLastError();
}

cudaError_t bun_units(const Bun32 &m, int nvox, const uint32_t *vox, uint32_t *tv, uint32_t *tb, uint32_t *td, int32_t *nunit,
                      int32_t *ndist, int *err, cudaStream_t st)
{
    static std::atomic<uint64_t> done32{0}, done64{0};
    int vbits = 1;
    while (vbits < 31 && (int64_t)1 << vbits < nvox) ++vbits;
    if (nvox <= 1 << 19) {
        const cudaError_t e = allow_smem(k_bun_units<uint32_t>, units_smem<uint32_t>(), done32);
        if (e != cudaSuccess) return e;
        k_bun_units<uint32_t><<<(unsigned)m.nbun, UT, units_smem<uint32_t>(), st>>>(m, vbits, vox, tv, tb, td, nunit, ndist, err);
    } else {
        const cudaError_t e = allow_smem(k_bun_units<uint64_t>, units_smem<uint64_t>(), done64);
        if (e != cudaSuccess) return e;
        k_bun_units<uint64_t><<<(unsigned)m.nbun, UT, units_smem<uint64_t>(), st>>>(m, vbits, vox, tv, tb, td, nunit, ndist, err);
    }
    return cudaGetLastError();
}

cudaError_t bun_ub(int nbun, const int64_t *uoff, const int64_t *doff, int2 *ub, int32_t *mx, cudaStream_t st)
{
    k_bun_ub<<<cap_grid(nbun + 1), 256, 0, st>>>(nbun, uoff, doff, ub, mx);
    return cudaGetLastError();
}

cudaError_t bun_compact(const Bun32 &m, const uint32_t *tv, const uint32_t *tb, const uint32_t *td,
                        uint32_t *uvox, cudaStream_t st)
{
    k_bun_compact<<<(unsigned)m.nbun, 256, 0, st>>>(m, tv, tb, td, uvox);
    return cudaGetLastError();
}

cudaError_t bun_coef(const Bun32 &m, const uint32_t *vox, const double *len64, const double *chi,
                     const int32_t *ray_angle, const double *wt, const double *invL, int nvox, cudaStream_t st)
{
    if (m.r_hi <= m.r_lo) return cudaSuccess;
    k_bun_coef<<<(unsigned)((m.r_hi - m.r_lo + 7) / 8), 256, 0, st>>>(m, vox, len64, chi, ray_angle, wt, invL, nvox);
    return cudaGetLastError();
}

template <typename OUT>
static cudaError_t bun_march_as(const Bun32 &m, const double *S, const double *B, float I_outer, int homog, OUT *out,
                                cudaStream_t st)
{
    static std::atomic<uint64_t> done{0};
    const cudaError_t e = allow_smem(k_march_bun<OUT>, sizeof(float) * (PLACES + 1 + BUN_CAP), done);
    if (e != cudaSuccess) return e;
    const size_t bytes = sizeof(float) * (size_t)(PLACES + 1 + m.dmax);
    k_march_bun<OUT><<<(unsigned)m.nbun, 32 * NW, bytes, st>>>(m, S, B, I_outer, homog, out);
    return cudaGetLastError();
}

cudaError_t bun_march(const Bun32 &m, const double *S, const double *B, float I_outer, int homog, void *out, bool pair,
                      cudaStream_t st)
{
    return pair ? bun_march_as(m, S, B, I_outer, homog, static_cast<float2 *>(out), st)
                : bun_march_as(m, S, B, I_outer, homog, static_cast<float *>(out), st);
}

}  // namespace rtk
