// geom_fast.cuh -- the voxels a characteristic crosses, found in FP32 with an
// error bound on every comparison and in FP64 where a bound is not enough.
// Included by geom.cu after the exact walk, whose cell sequence it reproduces.
//
// The FP64 pipe is narrow on this GPU (an FP64 instruction of a warp takes an SM
// about 19 cycles), and a step of the exact walk evaluates surfaces in FP64 with
// square roots and divisions, in a branch per kind of surface: about 13 000 cycles
// for a warp.  The launch set only needs the order of the crossings, so here a
// step evaluates the cell's faces in FP32, each crossing with a margin that
// bounds its distance from the parameter the exact walk would compute, and takes
// the nearest one if its interval overlaps neither another candidate's nor the
// current parameter's.  Otherwise (grazing lines, crossings closer than FP32
// resolves, ties) the step is the exact walk's, from the exact current
// parameter, which is evaluated again from the surface that was crossed last.
//
// Parameters are measured from the line's closest approach to the origin (to
// the axis on the cylindrical grid): s = t - tm, X = P + s d with P . d = 0, so
// that P and s are as small as the geometry around the cell and FP32 resolves
// about 1e-6 of a cell's distance from the centre.  Lengths and parameters are
// multiplied by the power of two F.scale, which changes no rounding.
//
// Margins.  u = 2^-24 bounds the relative rounding of an operation and of a
// table entry.  With |x| the size of the terms of a sum, first order in u:
//   shell      h2 = (r - p)(r + p):  E = 4 u (r + p)^2,  ds = E / (2 sqrt h2)
//   cone       f(s) = A s^2 + 2 B s + C, A = dz^2 - c^2, B = Pz dz, C = Pz^2 - c^2 p^2:
//              df = u (4 |A| s^2 + 8 |B| |s| + 6 |C|) with |A|, |C| the sums of sizes,
//              ds = df / |f'| = df / (2 sqrt disc); valid while ds |A| is small against
//              sqrt disc
//   half-plane s = -num / den:  ds = (dnum + |s| dden) / |den|
//   z-plane    ds = 2 u (|z_m| + |Pz|) / |dz|
// plus a few u |s| (quotients and roots are the hardware's, good to 2 ulp = 4 u);
// every margin is doubled.  The FP64 rounding of P (about 2^-52 of
// |x0| + |tm|, whatever is left of them) and of the exact walk's own products of x0
// is added through fl = 2e-8 (|x0| + |tm|) in the sizes of P's components and c64 =
// 1e-14 |x0|^2 in squares: far below the rest unless radii differ by more than 1e4.

constexpr float U24 = 5.9604645e-8f;

struct FastLine {
    double tm;                       // closest approach (unscaled)
    float px, py, pz, dx, dy, dz;    // P and the direction
    float p, p2;                     // |P| (of x, y on the cylindrical grid) and its square
    float pm, pzm, pxy, adz, dxy;    // sizes: |P|, |Pz|, |Px| + |Py| with the FP64 rounding; |dz|, |dx| + |dy|
    float isa, rdz;                  // 1 / sqrt(a), 1 / dz
    float fl, c64;
    int zs;                          // sign of dz
    bool usable;
};

__device__ __forceinline__ FastLine fast_line(const GeomDev &G, const Line &L, double scale)
{
    FastLine f;
    const bool sph = G.coord == RT_SPHERICAL;
    f.usable = L.a > 1e-8;
    f.tm = f.usable ? -(L.b / L.a) : 0.0;
    const double x = (L.x + f.tm * L.dx) * scale, y = (L.y + f.tm * L.dy) * scale, z = (L.z + f.tm * L.dz) * scale;
    const float tm = fabsf((float)(f.tm * scale));
    const double p2 = sph ? (x * x + y * y) + z * z : x * x + y * y;
    f.px = (float)x;
    f.py = (float)y;
    f.pz = (float)z;
    f.dx = (float)L.dx;
    f.dy = (float)L.dy;
    f.dz = (float)L.dz;
    f.p2 = (float)p2;
    f.p = sqrtf(f.p2);
    const float x2 = (float)((sph ? L.p2 : L.p2 + L.z2) * scale * scale);
    f.fl = 2e-8f * (sqrtf(x2) + tm);
    f.c64 = 1e-14f * x2;
    f.pm = f.p + f.fl;
    f.pzm = fabsf(f.pz) + f.fl;
    f.pxy = fabsf(f.px) + fabsf(f.py) + 2.0f * f.fl;
    f.adz = fabsf(f.dz);
    f.dxy = fabsf(f.dx) + fabsf(f.dy);
    f.isa = f.usable ? rsqrtf((float)L.a) : 0.0f;
    f.zs = (L.dz > 0.0) - (L.dz < 0.0);
    f.rdz = __fdividef(1.0f, f.dz);
    // squares within FP32's range
    f.usable = f.usable && x2 < 1e16f && x2 > 1e-16f && tm < 1e8f;
    return f;
}

// The root of a surface the walk crossed last: 0 the start (t = 0), 1 shell lo,
// 2 shell hi, 3 and 4 cone ra and rb, 5 half-plane, 6 z-plane.
enum { R_START = 0, R_SHLO, R_SHHI, R_CONEA, R_CONEB, R_HALF, R_ZPL };

__device__ __forceinline__ double exact_root(const GeomDev &G, const Line &L, int kind, int m)
{
    double a = 0.0, b = 0.0;
    if (kind == R_SHLO || kind == R_SHHI) {
        shell_roots(G, L, m, a, b);
        return kind == R_SHLO ? a : b;
    }
    if (kind == R_CONEA || kind == R_CONEB) {
        cone_roots(G, L, m, a, b);
        return kind == R_CONEA ? a : b;
    }
    if (kind == R_HALF) return halfplane_root(G, L, m);
    if (kind == R_ZPL) return zplane_root(G, L, m);
    return 0.0;
}

// One step of the exact walk from parameter t in cell (i, j, k): how it ends (0:
// it goes on), the next cell and parameter, and the root that was crossed.
__device__ __noinline__ int exact_step(const GeomDev &G, const Line &L, double t, int &i, int &j, int &k, double &tn,
                                       int &kind, int &surf)
{
    const bool sph = G.coord == RT_SPHERICAL;
    const long long INFB = bits(dinf()), tb = bits(t);
    long long c[6] = {INFB, INFB, INFB, INFB, INFB, INFB};
    int kd[6] = {R_SHLO, R_SHHI, 0, 0, 0, 0}, sf[6] = {i, i + 1, 0, 0, 0, 0};
    double lo, hi;
    if (!(i == 0 && G.e1[0] == 0.0)) {
        shell_roots(G, L, i, lo, hi);
        if (bits(lo) > tb && bits(lo) < bits(hi)) c[0] = bits(lo);
    }
    shell_roots(G, L, i + 1, lo, hi);
    if (bits(hi) > tb) c[1] = bits(hi);
    double ra, rb;
    auto cone = [&](int q, int m) {
        cone_roots(G, L, m, ra, rb);
        c[q] = after(ra, rb, tb, INFB);
        sf[q] = m;
        kd[q] = c[q] == bits(ra) ? R_CONEA : R_CONEB;
    };
    auto half = [&](int q, int m) {
        ra = halfplane_root(G, L, m);
        c[q] = bits(ra) > tb ? bits(ra) : INFB;
        sf[q] = m;
        kd[q] = R_HALF;
    };
    auto zpl = [&](int q, int m) {
        ra = zplane_root(G, L, m);
        c[q] = bits(ra) > tb ? bits(ra) : INFB;
        sf[q] = m;
        kd[q] = R_ZPL;
    };
    if (sph) {
        if (j >= 1) cone(2, j);
        if (j + 1 <= G.n2 - 1) cone(3, j + 1);
        if (G.n3 > 1) {
            half(4, k);
            half(5, (k + 1 == G.n3) ? 0 : k + 1);
        }
    } else {
        if (G.n2 > 1) {
            half(2, j);
            half(3, (j + 1 == G.n2) ? 0 : j + 1);
        }
        if (L.dz < 0.0) zpl(4, k);
        if (L.dz > 0.0) zpl(5, k + 1);
    }
    long long best = INFB;
    for (int q = 0; q < 6; ++q)
        if (c[q] < best) {
            best = c[q];
            kind = kd[q];
            surf = sf[q];
        }
    if (best == INFB) return RTK_END_LOST;
    int ni = i, nj = j, nk = k;
    bool ex = false, core = false;
    if (c[0] == best) { if (i == 0) core = true; else ni = i - 1; }
    if (c[1] == best) { if (i == G.n1 - 1) ex = true; else ni = i + 1; }
    if (sph) {
        if (c[2] == best) nj = nj - 1;
        if (c[3] == best) nj = nj + 1;
        if (c[4] == best) nk = (nk == 0) ? G.n3 - 1 : nk - 1;
        if (c[5] == best) nk = (nk + 1 == G.n3) ? 0 : nk + 1;
    } else {
        if (c[2] == best) nj = (nj == 0) ? G.n2 - 1 : nj - 1;
        if (c[3] == best) nj = (nj + 1 == G.n2) ? 0 : nj + 1;
        if (c[4] == best) { if (k == 0) ex = true; else nk = k - 1; }
        if (c[5] == best) { if (k == G.n3 - 1) ex = true; else nk = k + 1; }
    }
    tn = __longlong_as_double(best);
    if (ex) return RTK_END_EXIT;
    if (core) {
        if (G.inner_bc == RT_CORE_B) return RTK_END_CORE;
        shell(G, L, 0, lo, hi);
        tn = hi;
        if (!sph) {
            double tz = dinf();
            if (L.dz > 0.0) tz = (G.e3[G.n3] - L.z) / L.dz;
            if (L.dz < 0.0) tz = (G.e3[0] - L.z) / L.dz;
            if (tz <= tn) return RTK_END_EXIT;
        }
        locate(G, L, tn, nj, nk);
        ni = 0;
        kind = R_SHHI;
        surf = 0;
    }
    i = ni;
    j = nj;
    k = nk;
    return 0;
}

// The nearest crossing ahead of the current one, and how near anything that is
// not resolved may be.
struct Nearest {
    float s, m;      // best candidate and its margin
    float next;      // lower end of the nearest other candidate
    float unsure;    // lower end of the nearest crossing that FP32 cannot place
    int face;
    int kind;
    float cur, mcur;
    __device__ __forceinline__ void start(float c, float mc)
    {
        s = next = unsure = HUGE_VALF;
        m = 0.0f;
        face = -1;
        kind = 0;
        cur = c;
        mcur = mc;
    }
    // a crossing at x +- d through face q; crossed: the very root the walk stands on
    __device__ __forceinline__ void add(float x, float d, int q, int kd, bool crossed)
    {
        if (crossed) return;
        if (!(x + d >= cur - mcur)) {
            if (x + d < cur - mcur) return;  // behind
            unsure = -HUGE_VALF;             // not a number: the exact step decides
            return;
        }
        if (x - d <= cur + mcur) {
            unsure = fminf(unsure, cur);
        } else if (x < s) {
            if (s - m < next) next = s - m;
            s = x;
            m = d;
            face = q;
            kind = kd;
        } else if (x - d < next) {
            next = x - d;
        }
    }
    __device__ __forceinline__ void doubt(float from) { unsure = fminf(unsure, from); }
    __device__ __forceinline__ bool clear() const { return face >= 0 && s + m < next && s + m < unsure; }
};

__device__ __forceinline__ void fast_cone(const FastLine &f, float c, int q, bool last_here, int last_kind, Nearest &N)
{
    if (c == 0.0f) {  // the plane z = 0
        if (f.zs == 0) return;
        if (f.adz < 1e-30f) {
            N.doubt(-HUGE_VALF);
            return;
        }
        const float s = -f.pz * f.rdz;
        N.add(s, 8.0f * U24 * (3.0f * fabsf(s) + f.pzm * fabsf(f.rdz)) + 1e-37f, q, R_CONEA, last_here && last_kind == R_CONEA);
        return;
    }
    const float cc = c * c, d2 = f.dz * f.dz;
    const float A = d2 - cc, B = f.pz * f.dz, C = f.pz * f.pz - cc * f.p2;
    const float Am = d2 + cc, Bm = f.pzm * f.adz + cc * f.fl, Cm = f.pzm * f.pzm + cc * f.pm * f.pm + f.c64 / U24;
    const float disc = B * B - A * C;
    const float E = 24.0f * U24 * (Bm * Bm + fabsf(A) * Cm + fabsf(C) * Am) + 1e-37f;
    if (disc < -E) return;
    if (!(disc > E)) {
        N.doubt(-HUGE_VALF);
        return;
    }
    const float isq = rsqrtf(disc), sq = disc * isq, i2 = 0.5f * isq;
    const float qq = (B >= 0.0f) ? -(B + sq) : (sq - B);
    const float r1 = __fdividef(qq, A), r2 = __fdividef(C, qq);
    const bool up = r1 <= r2;  // r1 is the smaller root (ra)
    bool far1 = false;         // A is all but zero: r1 is far away, on a side FP32 cannot tell
#pragma unroll
    for (int w = 0; w < 2; ++w) {
        const float s = w ? r2 : r1, as = fabsf(s);
        const int kd = (w == 0) == up ? R_CONEA : R_CONEB;
        const float d = 2.0f * (U24 * (4.0f * Am * as * as + 8.0f * Bm * as + 6.0f * Cm) * i2 * 1.5f + 12.0f * U24 * as);
        if (!(d * fabsf(A) <= 0.25f * sq)) {
            far1 = true;
            const float lb = 0.4f * __fdividef(fabsf(qq), fabsf(A) + 8.0f * U24 * Am);
            N.doubt(w == 0 && lb > fabsf(N.cur) + N.mcur ? lb : -HUGE_VALF);
            continue;
        }
        if (s + d < N.cur - N.mcur) continue;  // behind
        const float z = f.pz + s * f.dz;
        const float dzv = 4.0f * U24 * (f.pzm + as * f.adz) + d * f.adz;
        const bool here = last_here && last_kind == kd;
        if (!here && (fabsf(z) <= dzv || far1)) {
            N.doubt(s - d);
            continue;
        }
        if (!here && (c > 0.0f) != (z > 0.0f)) continue;
        N.add(s, d, q, kd, here && !far1);
    }
}

__device__ __forceinline__ void fast_half(const FastLine &f, float c, float s, int q, bool last_here, Nearest &N)
{
    const float den = c * f.dy - s * f.dx, num = c * f.py - s * f.px;
    const float dnum = 6.0f * U24 * f.pxy + 1e-37f, dden = 6.0f * U24 * f.dxy + 1e-37f;
    if (fabsf(den) <= 4.0f * dden) {
        const float lb = 0.9f * __fdividef(fabsf(num) - dnum, fabsf(den) + dden);
        N.doubt(lb > fabsf(N.cur) + N.mcur ? lb : -HUGE_VALF);
        return;
    }
    const float rden = __fdividef(1.0f, den);
    const float r = -num * rden, ar = fabsf(r);
    const float d = 1.4f * (dnum + ar * dden) * fabsf(rden) + 16.0f * U24 * ar;
    const float h = c * (f.px + r * f.dx) + s * (f.py + r * f.dy);
    const float dh = 8.0f * U24 * (f.pxy + ar * f.dxy) + d * f.dxy;
    if (fabsf(h) <= dh) {
        if (r + d >= N.cur - N.mcur && !last_here) N.doubt(r - d);
        return;
    }
    if (h < 0.0f) return;
    N.add(r, d, q, R_HALF, last_here);
}

// Cells from the centre of voxel (i, j, k) along (dx, dy, dz): vis.cell(vox) for
// each, as walk() reports them; returns how the characteristic ended.
template <class Visit>
__device__ __forceinline__ int fast_walk(const GeomDev &G, const GeomF &F, double x0, double y0, double z0, double dx, double dy, double dz, int i,
                         int j, int k, Visit &vis)
{
    const Line L = make_line(G, x0, y0, z0, dx, dy, dz);
    const FastLine f = fast_line(G, L, F.scale);
    const bool sph = G.coord == RT_SPHERICAL;
    const int nsteps = max_steps(G);
    int kind = R_START, surf = 0;
    float cur = (float)(-f.tm * F.scale), mcur = 8.0f * U24 * fabsf(cur) + 1e-37f;
    for (int step = 0; step < nsteps; ++step) {
        const int v = vid(G, i, j, k);
        Nearest N;
        N.start(cur, mcur);
        if (!f.usable) {
            N.doubt(-HUGE_VALF);
        } else {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                if (q == 0 && i == 0 && F.r0_zero) continue;
                const float r = F.e1[i + q], sm = r + f.p;
                const float h2 = (r - f.p) * sm;
                const float E = 8.0f * U24 * sm * sm + f.c64;
                if (h2 < -E) {  // missed: the inner face; the outer one cannot be
                    if (q) N.doubt(-HUGE_VALF);
                    continue;
                }
                if (!(h2 > 4.0f * E)) {
                    N.doubt(-HUGE_VALF);
                    continue;
                }
                const float ih = rsqrtf(h2), s = h2 * ih * f.isa;
                const float d = E * ih * f.isa + 24.0f * U24 * s;
                if (q) N.add(s, d, 1, R_SHHI, kind == R_SHHI && surf == i + 1);
                else N.add(-s, d, 0, R_SHLO, kind == R_SHLO && surf == i);
            }
            if (sph) {
                if (j >= 1)
                    fast_cone(f, F.ct[j], 2, surf == j, kind, N);
                if (j + 1 <= G.n2 - 1)
                    fast_cone(f, F.ct[j + 1], 3, surf == j + 1, kind, N);
                if (G.n3 > 1) {
                    const int k1 = (k + 1 == G.n3) ? 0 : k + 1;
                    fast_half(f, F.cp[k], F.sp[k], 4, kind == R_HALF && surf == k, N);
                    fast_half(f, F.cp[k1], F.sp[k1], 5, kind == R_HALF && surf == k1, N);
                }
            } else {
                if (G.n2 > 1) {
                    const int j1 = (j + 1 == G.n2) ? 0 : j + 1;
                    fast_half(f, F.cp[j], F.sp[j], 2, kind == R_HALF && surf == j, N);
                    fast_half(f, F.cp[j1], F.sp[j1], 3, kind == R_HALF && surf == j1, N);
                }
                if (f.zs != 0) {
                    const int m = f.zs > 0 ? k + 1 : k;
                    const float e = F.e3[m];
                    if (f.adz < 1e-30f) N.doubt(-HUGE_VALF);
                    const float s = (e - f.pz) * f.rdz;
                    const float d = 4.0f * U24 * ((fabsf(e) + f.pzm) * fabsf(f.rdz) + 6.0f * fabsf(s)) + 1e-37f;
                    N.add(s, d, f.zs > 0 ? 5 : 4, R_ZPL, kind == R_ZPL && surf == m);
                }
            }
        }
        if (N.clear() && !(N.face == 0 && i == 0 && G.inner_bc != RT_CORE_B)) {
            vis.cell(v);
            cur = N.s;
            mcur = N.m;
            kind = N.kind;
            const int q = N.face;
            if (q == 0) {
                if (i == 0) return RTK_END_CORE;
                surf = i;
                i = i - 1;
            } else if (q == 1) {
                if (i == G.n1 - 1) return RTK_END_EXIT;
                i = i + 1;
                surf = i;
            } else if (sph) {
                if (q == 2) { surf = j; j = j - 1; }
                else if (q == 3) { j = j + 1; surf = j; }
                else if (q == 4) { surf = k; k = (k == 0) ? G.n3 - 1 : k - 1; }
                else { k = (k + 1 == G.n3) ? 0 : k + 1; surf = k; }
            } else {
                if (q == 2) { surf = j; j = (j == 0) ? G.n2 - 1 : j - 1; }
                else if (q == 3) { j = (j + 1 == G.n2) ? 0 : j + 1; surf = j; }
                else if (q == 4) { if (k == 0) return RTK_END_EXIT; surf = k; k = k - 1; }
                else { if (k == G.n3 - 1) return RTK_END_EXIT; k = k + 1; surf = k; }
            }
        } else {
            double tn = 0.0;
            const int end = exact_step(G, L, exact_root(G, L, kind, surf), i, j, k, tn, kind, surf);
            if (end != RTK_END_LOST) vis.cell(v);
            if (end) return end;
            cur = (float)((tn - f.tm) * F.scale);
            mcur = 8.0f * U24 * fabsf(cur) + 1e-37f;
        }
    }
    return RTK_END_LOST;
}
