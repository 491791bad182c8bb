// mg_march.cuh -- FP64 stencils of a whole 3D level on the integer pipe: a block
// marches a 32 x 8 column of cells through a range of planes.
//
// The residual and the forces of a DRAM-resident level are bound by the FP64
// pipe when written with doubles (9 and 12 instructions a cell of 64 cycles a
// warp) and by the instruction count when every cell aligns all its neighbours
// to integers (mg_fix.cuh, about 16 instructions each).  Here every value is
// aligned once, by the thread that loads it (1.3 times with the tile's halo, 1.7
// times for two rings): the neighbours in the plane come from shared memory, those
// along z from a window in registers.  All values of a block share one
// exponent, the largest seen so far plus a bit; a plane that exceeds it shifts
// what the block holds (the test rides on the barrier that each plane needs
// anyway).  Cells for which that exponent is too large take the FP64
// instructions: residuals whose centre is below 2^-6 of it (else the truncation
// of the terms is of the size of FP64's own rounding, 12 units of 2^-53 of the
// centre at most), forces of which a term lost a bit (else their sum is exact
// and rounded once).  Two planes are in flight ahead of the one being aligned,
// and the functor's own loads one plane ahead.
#pragma once

#include "mg_fix.cuh"

struct MarchGrid {
    int n[3];         // active cells per axis; storage extents are n + 2 R
    int nx, ny, zc;   // tiles along x and y, planes per block
    int sy;           // words per row
    long long sz;     // words per plane
};

// Tiles and z ranges: of the splits with at least 8 planes a block and at most
// MG_MARCH_BLOCKS blocks, the one whose waves of 152 x 5 resident blocks march the
// fewest planes in all (each block also loads 2 R planes around its own).
// Five blocks an SM is what the residual kernels keep; the force kernels keep four
// but gain from the longer split: counting four, mg_forces takes 61.0 -> 56.8 us at
// 160^3 and 209 -> 204 at 256^3, but 49.7 -> 51.1 at 144^3 and 403 -> 490 at 512x256x256.
inline MarchGrid march_grid(int n0, int n1, int n2, long long sy, long long sz, int R, int *blocks)
{
    MarchGrid m;
    m.n[0] = n0;
    m.n[1] = n1;
    m.n[2] = n2;
    m.nx = (n0 + 31) / 32;
    m.ny = (n1 + 7) / 8;
    m.sy = (int)sy;
    m.sz = sz;
    m.zc = n2;
    const int tiles = m.nx * m.ny;
    long best = 0;
    for (int c = 1; c == 1 || (c * 8 <= n2 && (long)tiles * c <= MG_MARCH_BLOCKS); c++) {
        const int zc = (n2 + c - 1) / c;
        const long cost = (((long)tiles * c + 759) / 760) * (zc + 2 * R);
        if (best == 0 || cost < best) {
            best = cost;
            m.zc = zc;
        }
    }
    *blocks = tiles * ((n2 + m.zc - 1) / m.zc);
    return m;
}

// v * 2^-d, the last bit set where bits are lost
__device__ __forceinline__ long long fx_shift_mark(long long v, int d)
{
    const long long r = v >> d;
    return (long long)((unsigned long long)r << d) == v ? r : r | 1;
}
// fx_align, the last bit set where x has bits there or below (it is clear otherwise)
template <int P>
__device__ __forceinline__ long long fx_align_mark(double x, int emax)
{
    const bool lost = emax - fx_exp(x) >= P && ((__double2hiint(x) << 1) | __double2loint(x)) != 0;
    return fx_align<P>(x, emax) | (lost ? 1 : 0);
}

// R rings; fn.prefetch(i, j, k) a plane ahead and fn(i, j, k, b, w, bound) for every active cell
// (storage indices): b points at the cell in its aligned plane of row pitch
// 32 + 2 R, w[0..2R] is its column, both multiples of 2^(bound - 1023 - 52 - P)
// and below 2^(52 + P) of them; with MARK the last bit says that bits were lost.
template <int R, int P, bool MARK, class Fn>
__device__ __forceinline__ void march(const double *__restrict__ src, const MarchGrid &g, Fn &fn)
{
    constexpr int TX = 32, TY = 8, W = TX + 2 * R, H = TY + 2 * R, NB = R + 1, HALO = 2 * R * (TX + TY);
    static_assert(HALO <= TX * TY, "one halo cell per thread");
    __shared__ long long buf[NB][H * W];
    __shared__ int s_e[TX * TY / 32];
    const int t = threadIdx.x, tx = t % TX, ty = t / TX;
    int q = blockIdx.x;
    const int bx = q % g.nx;
    q /= g.nx;
    const int by = q % g.ny, z0 = q / g.ny * g.zc + R, z1 = min(z0 + g.zc, g.n[2] + R);
    const int x = bx * TX + tx + R, y = by * TY + ty + R;
    const bool in = x < g.n[0] + 2 * R && y < g.n[1] + 2 * R, active = x < g.n[0] + R && y < g.n[1] + R;
    // this thread's halo cell
    int hx = 0, hy = 0;
    if (t < 2 * R * TX) {
        const int r = t / TX;
        hx = R + tx;
        hy = r < R ? r : TY + r;
    } else if (t < HALO) {
        const int u = t - 2 * R * TX, c = u / TY;
        hx = c < R ? c : TX + c;
        hy = R + u % TY;
    }
    const int gx = bx * TX + hx, gy = by * TY + hy;
    const bool halo = t < HALO && gx < g.n[0] + 2 * R && gy < g.n[1] + 2 * R;
    const double *pc = src + (long long)(z0 - R) * g.sz + (long long)y * g.sy + x;
    const double *ph = src + (long long)(z0 - R) * g.sz + (long long)gy * g.sy + gx;
    const int at = (ty + R) * W + tx + R, hat = hy * W + hx;
    const int last = z1 - 1 + R;   // last plane loaded
    double c0 = in ? pc[0] : 0.0, h0 = halo ? ph[0] : 0.0;
    double c1 = in ? pc[g.sz] : 0.0, h1 = halo ? ph[g.sz] : 0.0;
    long long w[2 * R + 1] = {};
    if (active)
        fn.prefetch(x, y, z0);
    int bound = 0, cur = 0;
    bool first = true;
    for (int p = z0 - R; p <= last; p++) {
        pc += g.sz;
        ph += g.sz;
        double c2 = 0.0, h2 = 0.0;
        if (p + 2 <= last) {
            if (in)
                c2 = pc[g.sz];
            if (halo)
                h2 = ph[g.sz];
        }
        const int k = p - R;
        const int e = max(fx_exp(c0), fx_exp(h0));
        if (__syncthreads_or(first || e > bound)) {
            // a larger exponent: the block's new common one
            const int m = __reduce_max_sync(0xffffffffu, e);
            if (tx == 0)
                s_e[ty] = m;
            __syncthreads();
            int nb = s_e[0];
#pragma unroll
            for (int u = 1; u < TX * TY / 32; u++)
                nb = max(nb, s_e[u]);
            nb++;
            if (!first) {
                const int d = min(nb - bound, 63);
#pragma unroll
                for (int u = 0; u <= 2 * R; u++)
                    w[u] = MARK ? fx_shift_mark(w[u], d) : w[u] >> d;
                for (int u = t; u < NB * H * W; u += TX * TY) {
                    long long &v = (&buf[0][0])[u];
                    v = MARK ? fx_shift_mark(v, d) : v >> d;
                }
            }
            bound = nb;
            first = false;
            __syncthreads();
        }
#pragma unroll
        for (int u = 0; u < 2 * R; u++)
            w[u] = w[u + 1];
        w[2 * R] = MARK ? fx_align_mark<P>(c0, bound) : fx_align<P>(c0, bound);
        buf[cur][at] = w[2 * R];
        if (t < HALO)
            buf[cur][hat] = MARK ? fx_align_mark<P>(h0, bound) : fx_align<P>(h0, bound);
        cur = cur == NB - 1 ? 0 : cur + 1;   // now the plane k = p - R: written R planes ago
        if (k >= z0 && active) {
            const auto ahead = fn.taken();
            if (k + 1 < z1)
                fn.prefetch(x, y, k + 1);
            fn(x, y, k, &buf[cur][at], w, bound, ahead);
        }
        c0 = c1;
        h0 = h1;
        c1 = c2;
        h1 = h2;
    }
}

// h-scaled differences of a column: 8 (a - b) - (c - d) of aligned values
__device__ __forceinline__ long long fx_d4(long long a, long long b, long long c, long long d)
{
    return 8 * (a - b) - (c - d);
}

// Residual f - ih2 (sum of the neighbours - 6 Phi) of every active cell of a
// finest multigrid level (one ring): |r|^2 summed into r2 and, with r32, r into
// the FP32 defect and zero into the correction, at the index idx(i, j, k) of
// those arrays; with b, |b|^2 (the residual of a zero potential inside) into b2.
template <class Idx>
struct MarchResidual {
    const double *phi, *f;
    int sy;
    long long sz;
    int n0, n1, n2;
    double ih2;
    bool want_b;
    float *r32, *e32;
    Idx idx;
    double b2, r2, fnext;

    __device__ __forceinline__ void prefetch(int i, int j, int k) { fnext = f[k * sz + (long long)j * sy + i]; }
    __device__ __forceinline__ double taken() const { return fnext; }

    __device__ __noinline__ static double plain_lap(const double *c, int sy, long long sz)
    {
        return ((c[-1] + c[1]) + (c[-sy] + c[sy])) + (c[-sz] + c[sz]) - 6.0 * c[0];
    }
    __device__ __noinline__ static double ring_sum(const double *c, int sy, long long sz, int bits)
    {
        double o = 0.0;
        if (bits & 1) o += c[-1];
        if (bits & 2) o += c[1];
        if (bits & 4) o += c[-sy];
        if (bits & 8) o += c[sy];
        if (bits & 16) o += c[-sz];
        if (bits & 32) o += c[sz];
        return o;
    }

    __device__ __forceinline__ void operator()(int i, int j, int k, const long long *b, const long long (&w)[3], int bound,
                                               double fv)
    {
        constexpr int W = 34;
        double lap;
        // a centre below 2^-6 of the block's exponent: truncation could exceed FP64's own rounding
        if (fx_ok(bound) && (unsigned long long)(w[1] + (1ll << 53)) >= (1ull << 54))
            lap = fx_round<6>((w[0] + w[2]) + (b[-1] + b[1]) + (b[-W] + b[W]) - 6 * w[1], bound);
        else
            lap = plain_lap(phi + (k * sz + (long long)j * sy + i), sy, sz);
        const double r = fma(-lap, ih2, fv);
        r2 = fma(r, r, r2);
        if (r32) {
            const long long q = idx(i, j, k);
            r32[q] = fx_to_float(r);
            e32[q] = 0.0f;
        }
        if (want_b) {
            const int bits = (i == 1 ? 1 : 0) | (i == n0 ? 2 : 0) | (j == 1 ? 4 : 0) | (j == n1 ? 8 : 0) |
                             (k == 1 ? 16 : 0) | (k == n2 ? 32 : 0);
            double v = fv;
            if (bits)
                v = fma(-ring_sum(phi + (k * sz + (long long)j * sy + i), sy, sz, bits), ih2, fv);
            b2 = fma(v, v, b2);
        }
    }
};

// F = -grad(Phi) (Eq. 2, or the two-point difference) and the potential on
// Omega of a block with two rings; component a at F[a cells + cell].
struct MarchForces {
    const double *phi;
    int sy;
    long long sz, cells;
    int n0, n1, stencil;
    double c;   // -1 / (12 h) or -1 / (2 h)
    double *F, *out;
    double pnext;

    __device__ __forceinline__ void prefetch(int i, int j, int k)
    {
        if (out)
            pnext = phi[k * sz + (long long)j * sy + i];
    }
    __device__ __forceinline__ double taken() const { return pnext; }
    __device__ __noinline__ static double plain(const double *p, long long st, int stencil)
    {
        return stencil == 0 ? 8.0 * (p[st] - p[-st]) - (p[2 * st] - p[-2 * st]) : p[st] - p[-st];
    }
    __device__ __forceinline__ void operator()(int i, int j, int k, const long long *b, const long long (&w)[5], int bound,
                                               double pv)
    {
        constexpr int W = 36;
        const double *p = phi + (k * sz + (long long)j * sy + i);
        const long long t = ((long long)(k - 2) * n1 + (j - 2)) * n0 + (i - 2);
        double d[3];
        {
            // the differences of aligned terms, and whether one of these lost bits (march)
            long long s[3];
            int lost[3];
            if (stencil == 0) {
                auto diff = [&](int a, long long p1, long long m1, long long p2, long long m2) {
                    s[a] = fx_d4(p1, m1, p2, m2);
                    lost[a] = ((int)p1 | (int)m1 | (int)p2 | (int)m2) & 1;
                };
                diff(0, b[1], b[-1], b[2], b[-2]);
                diff(1, b[W], b[-W], b[2 * W], b[-2 * W]);
                diff(2, w[3], w[1], w[4], w[0]);
            } else {
                auto diff = [&](int a, long long p1, long long m1) {
                    s[a] = p1 - m1;
                    lost[a] = ((int)p1 | (int)m1) & 1;
                };
                diff(0, b[1], b[-1]);
                diff(1, b[W], b[-W]);
                diff(2, w[3], w[1]);
            }
            const bool ok = fx_ok(bound);
#pragma unroll
            for (int a = 0; a < 3; a++) {
                d[a] = fx_round<6>(s[a], bound);
                if (!ok || lost[a])
                    d[a] = plain(p, a == 0 ? 1 : a == 1 ? sy : sz, stencil);
            }
        }
        if (F) {
#pragma unroll
            for (int a = 0; a < 3; a++)
                F[a * cells + t] = c * d[a];
        }
        if (out)
            out[t] = pv;
    }
};
