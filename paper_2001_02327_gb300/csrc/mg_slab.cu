// mg_slab.cu -- the coarse part of the V-cycle (Sec. 2.3 steps 2-13 on the
// multigrid levels from a size limit down) in one launch of one thread-block
// cluster.  Every array of those levels lives on chip: the potentials in the
// shared memory of the cluster's CTAs (the larger levels as slabs of planes
// along the outermost axis, z in 3D and y in 2D, the smaller ones whole in CTA
// 0), the right-hand sides and coefficients with the threads that use them.
//
// What bounds these levels is latency, not arithmetic or bandwidth: a level of
// 33^3 cells has 18k updates per colour, less than a microsecond of work for
// the whole GPU, but one launch per phase costs about 2.2 us (a graph node with
// programmatic dependent launch about 0.9 us, the loads' round trip to L2 the
// rest).  So everything here removes steps from the dependent chain of a phase:
//   - a thread owns fixed pairs of neighbouring cells (2x+1, 2x+2) of a row on
//     every level; where they are, which boundary class they have and where
//     their children and parents are comes packed from a plan image in global
//     memory, written once per level configuration and copied to shared memory
//     before the kernel waits for its predecessor, so no phase divides;
//   - each CTA keeps copies of its neighbours' boundary planes, and the owner
//     pushes every new value into the copies, so that sweeps load locally only;
//     a colour pass waits for its two neighbours' values alone (asynchronous
//     stores that count their bytes on an mbarrier, about 300 cycles) and not at
//     a barrier of the whole cluster (about 600 with its stores);
//   - a thread holds its cells' right-hand sides and coefficients in registers
//     from sweep to sweep;
//   - the first red half-sweep on a level (whose correction starts from zero)
//     is done with the restriction into it, the potential that a finer level
//     interpolates is copied to where it reads it right after the level's last
//     sweep, and the pair sums of the restriction come from the residual pass;
//   - from the first level of at most 64 cells down, one V-cycle from a zero
//     correction is a fixed linear map of that level's right-hand side: its
//     matrix is built once (in FP64) and applied as a matrix-vector product,
//     one phase in place of the 25 or so of those levels;
//   - an FP64 level that fits whole is solved by one launch: the V-cycles of its
//     loop, the residual norm and the decision after each.  Loading the level
//     (4 us), its norm kernel, the control kernel and the turn of the graph's
//     loop then happen once per solve and not once per cycle: a hierarchy of
//     three 16^3 levels 2.05 -> 1.28 ms, of three 64^2 levels 1.35 -> 0.90 ms
//     (one launch per phase: 2.73 and 2.34 ms).
//
// One V-cycle, launch to launch: 33^3 31 us in FP32 and 48 us in FP64, 17^3 15
// us (FP32), 18^3 30 us and 66^2 28 us (FP64).
//
// FP64 V-cycles run in 64-bit fixed point.  The part issues one FP64
// instruction per sub-partition every 64 cycles but a 64-bit integer addition
// every 2.3 (measured), so an update of the 7-point stencil (five additions,
// one FMA, one product) takes 450 cycles a warp in FP64 and about 45 as
// integers: the neighbour sum and the right-hand side are exact, the product
// by the reciprocal diagonal is a 64 x 64 bit high product.  Every level has a
// power-of-two scale of its own, taken from the largest right-hand side (and
// potential) it starts from; a coarse correction too large for the finer
// level's scale, or a potential that has outgrown it, lowers that scale first
// (prolong_scale).  So a potential stays below 2^57 + 2^57 and what the sweeps
// add, the sum of a pair's residuals (f + 12 Phi at most, twice) below 2^63.
//
// What that costs in accuracy: a level's arrays share a scale, so a value far
// below the level's largest keeps fewer bits of its own than a double would.
// What a finest level keeps from cycle to cycle has 56 to 57 bits for the
// largest potential (ring included) and, without a potential that outweighs
// it, 54 to 57 for the largest right-hand side; a level that is a correction
// of a finer one starts from 50 to 57 bits.  Largest error of the converged
// potential over its largest value, V(2,2), against a solution in 128 bits,
// FP64 launches -> here: a sphere with its potential on the ring, 32^3 1.6e-15
// -> 7.5e-17, 160^2 1.6e-14 -> 1.6e-16; random density and ring 3.0e-16 ->
// 2.6e-16 and 5.7e-16 -> 2.9e-16; an amplitude growing by 2^30 across the level
// 4.0e-16 -> 1.6e-16 and 5.4e-16 -> 4.9e-16.  There the cells of the median,
// 2^-15 of the largest, are 1.9e-15 (32^3, launches 7e-16) and 2e-14 (160^2,
// launches 4.6e-15) of their own value off.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <type_traits>
#include <vector>

#include <math_constants.h>

#include "mg_internal.h"

namespace {

constexpr int kT = MG_SLAB_THREADS;
constexpr int kWaitUnits = 954;                   // bound of one wait in 2^21 cycles (1 ms), about 1 s
constexpr long long kDrainCycles = 1ll << 19;     // time that values sent before a failure have to arrive

typedef long long fix;   // fixed-point value: real * 2^scale

__device__ __forceinline__ unsigned cluster_rank_()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// every thread of every CTA of the cluster, from converged code
__device__ __forceinline__ void cluster_sync_()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Shared memory by 32-bit address: the same location in CTA `rank` of the
// cluster, and loads and stores there
__device__ __forceinline__ unsigned cluster_addr(unsigned a, int rank)
{
    unsigned out;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(out) : "r"(a), "r"(rank));
    return out;
}
__device__ __forceinline__ void st_cluster(unsigned a, float v)
{
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void st_cluster(unsigned a, long long v)
{
    asm volatile("st.shared::cluster.b64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
}
__device__ __forceinline__ void st_cluster(unsigned a, unsigned v)
{
    asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void ld_cluster(float &v, unsigned a)
{
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
}
__device__ __forceinline__ void ld_cluster(long long &v, unsigned a)
{
    asm volatile("ld.shared::cluster.b64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
}
// a store that counts its bytes on the mbarrier `mb` of the same CTA
__device__ __forceinline__ void st_async(unsigned a, float v, unsigned mb)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(a),
                 "r"(__float_as_uint(v)), "r"(mb)
                 : "memory");
}
__device__ __forceinline__ void st_async(unsigned a, long long v, unsigned mb)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(a), "l"(v), "r"(mb)
                 : "memory");
}
__device__ __forceinline__ void mbar_init(unsigned mb, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mb), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect(unsigned mb, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(unsigned mb, unsigned parity)
{
    unsigned ok;
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok)
                 : "r"(mb), "r"(parity)
                 : "memory");
    return ok != 0;
}
template <typename T>
__device__ __forceinline__ unsigned shared_addr(const T *p)
{
    return (unsigned)__cvta_generic_to_shared(p);
}

// Everything that a level keeps is rounded to nearest: a rounding that leans to
// one side adds up over the level.  With floors, half a unit on every
// right-hand side moved the potential by N^2 / 16 units.

// (v * K) >> (32 + S) for |v|, |K| < 2^62, K = kh 2^32 + kl with kl signed; the
// product of the low words (below one unit) is dropped.  It leans by half a unit
// and more: update() rounds, the others scale corrections, whose last bits the
// next cycle corrects.
template <int S>
__device__ __forceinline__ fix qmul(fix v, fix K)
{
    const int kl = (int)K, kh = (int)((K - kl) >> 32);
    const int vh = (int)(v >> 32);
    const unsigned vl = (unsigned)v;
    const fix mid = (fix)vh * kl + (fix)vl * kh;
    return (((fix)vh * kh) << (32 - S)) + (mid >> S);
}

__device__ __forceinline__ fix shift_by(fix v, int s)   // v * 2^s, |v| < 2^62
{
    if (s >= 0)
        return v << min(s, 63);
    s = min(-s, 63);
    return (v + (1ll << (s - 1))) >> s;
}

// v * 2^-s, ties to even: where the dropped bits are few, ties are many and
// must not lean either (0 <= v < 2^63 or |v| < 2^62; s >= 0)
template <typename V>
__device__ __forceinline__ V shift_even(V v, int s)
{
    return s == 0 ? v : s > 63 ? V(0) : (v + ((V(1) << (s - 1)) - 1) + ((v >> s) & 1)) >> s;
}

// x * 2^scale (|result| < 2^62 by the choice of the scale; x finite)
__device__ __forceinline__ fix to_fix(double x, int scale)
{
    const int hi = __double2hiint(x);
    const unsigned lo = (unsigned)__double2loint(x);
    const int e = (hi >> 20) & 0x7ff;
    if (e == 0)
        return 0;   // zero or denormal
    const unsigned long long m = ((unsigned long long)((hi & 0xfffff) | 0x100000) << 32) | lo;
    const int s = e - 1075 + scale;
    const fix a = (fix)(s >= 0 ? m << min(s, 63) : shift_even(m, -s));
    return hi < 0 ? -a : a;
}

// x * k * 2^(scale - 62) for 2^61 <= k < 2^62 (|result| < 2^58), rounded once
__device__ __forceinline__ fix to_fix_times(double x, fix k, int scale)
{
    const int hi = __double2hiint(x);
    const unsigned lo = (unsigned)__double2loint(x);
    const int e = (hi >> 20) & 0x7ff;
    if (e == 0)
        return 0;
    const unsigned long long m = ((unsigned long long)((hi & 0xfffff) | 0x100000) << 43) | ((unsigned long long)lo << 11);
    const unsigned long long k2 = (unsigned long long)k << 1;
    // the product's upper 64 bits, the last one set where lower ones are: 2^61 .. 2^63
    const unsigned long long p = __umul64hi(m, k2) | (m * k2 ? 1 : 0);
    const fix a = (fix)shift_even(p, 1085 - e - scale);
    return hi < 0 ? -a : a;
}

// v * 2^-scale rounded to nearest (ties away from zero)
__device__ __forceinline__ double from_fix(fix v, int scale)
{
    if (v == 0)
        return 0.0;
    const unsigned long long a = v < 0 ? (unsigned long long)(-v) : (unsigned long long)v;
    const int lz = __clzll((fix)a);
    const unsigned long long n = a << lz;
    const unsigned long long q = (n >> 11) + ((n >> 10) & 1);   // 2^52 .. 2^53
    const int e = 63 - lz - scale + 1023;
    unsigned long long bits;
    if (e <= 0)
        bits = 0;
    else if (e >= 2047)
        bits = 0x7ffull << 52;
    else
        bits = ((unsigned long long)(e - 1) << 52) + q;         // the carry of q = 2^53 reaches the exponent
    if (v < 0)
        bits |= 1ull << 63;
    return __longlong_as_double((long long)bits);
}

// Working precision: storage type T of the shared-memory arrays and G of the
// global ones; words per boundary class of the coefficient tables.
struct PrecF32 {
    typedef float T;
    typedef float G;
    static constexpr bool kFix = false;
    static constexpr int kTab = 2;   // negated reciprocal diagonal, diagonal
};
struct PrecFix {
    typedef fix T;
    typedef double G;
    static constexpr bool kFix = true;
    static constexpr int kTab = 3;   // reciprocal of -diagonal * 2^63, floor(-diagonal), its fraction * 2^62
};

// The plan image: per item (a pair of cells of a thread) four words.
//   A  bits 0-13 b, the index of the odd cell 2x+1 within its colour (the even
//      cell is at b + 1 of the other colour); 14 colour of the odd cell; 15, 16
//      odd, even cell exists; 17-18, 19-20 boundary class along the second and
//      third axis (bit 0 first, bit 1 last cell); 21-22 the odd cell's along x;
//      23 even cell last along x; 24, 25 the plane before, after is another CTA's
//   B  bits 0-13 index of (near plane, near row, column x) among the staged
//      coarse planes; 14, 15 the far row, plane is the next one (else previous)
//   C  bits 0-13 index of the first child pair in the finer level's pair sums;
//      14-17 CTA of the first child plane, 18-21 of the second; 22 the second
//      plane, 23 the second row exists; 24 the second plane is the first of its
//      CTA; 25-28 the first plane's index within its CTA
//   D  level 0: x (bits 0-9), row (10-19), plane (20-29); other levels: bits
//      0-12 index of the odd cell within a staged plane, 13-16 the first CTA
//      that interpolates from this plane, 17-20 how many do, 21-30 the plane
// In the image (and in shared memory) the A words of all slots come first,
// then B, C, D of the slots of the levels with one pair per thread; those of
// the other levels follow and stay in global memory (read once per V-cycle).
// Then, per level of the plan but the last, the ghost cells of the staged
// planes: bits 0-12 the cell, 13-25 the cell it comes from, and two bits per
// axis (x lowest) for the factor: 0 one, 1 minus one, 2 cR.
constexpr int kA = 0, kB = 1, kC = 2, kD = 3;

// One level as one CTA sees it.  Colour c of plane k, row j, storage half
// index m at ph[c cs + ((k - k0 + 1) R + j) H + m].
struct Shape {
    int N, H, R, cs, rows, ha, k0, k1, total;
};

// planes 1..N of a distributed level over the C CTAs: CTA r owns [plane_first(r), plane_first(r + 1)),
// and plane k belongs to CTA plane_owner(k); the other levels are CTA 0's
__host__ __device__ __forceinline__ bool slab_dist(const MgSlabPlan &p, int q) { return q < p.nclu; }
__host__ __device__ __forceinline__ int plane_first(const MgSlabPlan &p, int q, int r)
{
    return slab_dist(p, q) ? 1 + ((r * p.g[q].N) >> p.lgc) : (r == 0 ? 1 : p.g[q].N + 1);
}
__host__ __device__ __forceinline__ int plane_owner(const MgSlabPlan &p, int q, int k)
{
    return slab_dist(p, q) ? ((k << p.lgc) - 1) / p.g[q].N : 0;
}
// first and last staged plane of level q + 1 in CTA r: those around its planes
// of level q (and the source of the right ghost plane where x_N = 1)
__host__ __device__ __forceinline__ int staged_first(const MgSlabPlan &p, int q, int r)
{
    const int K = plane_first(p, q, r) >> 1;
    const MgGeom &c = p.g[q + 1];
    return c.tie && plane_first(p, q, r + 1) > p.g[q].N && K > c.N - 1 ? c.N - 1 : K;
}
__host__ __device__ __forceinline__ int staged_last(const MgSlabPlan &p, int q, int r)
{
    return ((plane_first(p, q, r + 1) - 1) >> 1) + 1;
}

template <int DIM>
__host__ __device__ __forceinline__ Shape shape_of(const MgSlabPlan &p, int q, int rank)
{
    Shape s;
    s.N = p.g[q].N;
    s.H = (s.N + 3) >> 1;
    s.R = DIM == 3 ? s.N + 2 : 1;
    s.cs = (p.po[q] + 2) * s.R * s.H;
    s.rows = DIM == 3 ? s.N : 1;
    s.ha = (s.N + 1) >> 1;
    s.k0 = plane_first(p, q, rank);
    s.k1 = plane_first(p, q, rank + 1);
    s.total = s.ha * s.rows * (s.k1 - s.k0);
    return s;
}

// Item t of level q in CTA `rank` (t = thread + 512 slot; the pair sums of the
// residual pass are stored at t)
template <int DIM>
__host__ __device__ void plan_item(const MgSlabPlan &p, int q, int rank, int t, int (&w)[4])
{
    const Shape s = shape_of<DIM>(p, q, rank);
    w[0] = w[1] = w[2] = w[3] = 0;
    if (t >= s.total) {
        w[kA] = s.R * s.H + (DIM == 3 ? s.H : 0);   // inside the slab
        return;
    }
    const int x = t % s.ha, r = t / s.ha;
    const int j = DIM == 3 ? r % s.rows + 1 : 0, kk = r / s.rows, k = s.k0 + kk;
    const int b = ((kk + 1) * s.R + j) * s.H + x;
    const bool even = 2 * x + 2 <= s.N;
    auto cls = [&](int v) { return (v == 1 ? 1 : 0) | (v == s.N ? 2 : 0); };
    const bool ring = p.g[q].L == 0;
    const int c2 = ring ? 0 : DIM == 3 ? cls(j) : cls(k), c3 = ring || DIM == 2 ? 0 : cls(k);
    w[kA] = b | (((1 + j + k) & 1) << 14) | (1 << 15) | ((even ? 1 : 0) << 16) | (c2 << 17) | (c3 << 19) |
            ((ring ? 0 : cls(2 * x + 1)) << 21) | ((!ring && 2 * x + 2 == s.N ? 1 : 0) << 23) |
            ((slab_dist(p, q) && kk == 0 && k > 1 ? 1 : 0) << 24) |
            ((slab_dist(p, q) && k == s.k1 - 1 && k < s.N ? 1 : 0) << 25);
    w[kD] = x | (j << 10) | (k << 20);
    if (q > 0) {
        // the CTAs with planes 2 k - 2 .. 2 k + 1 of the finer level (and its last plane, whose
        // right ghost comes from cell N - 1 where x_N = 1)
        const int Nf = p.g[q - 1].N, ka = max(2 * k - 2, 1);
        const int kb = p.g[q].tie && k == s.N - 1 ? Nf : min(2 * k + 1, Nf);
        const int oa = plane_owner(p, q - 1, ka), ob = plane_owner(p, q - 1, kb);
        w[kD] = (j * (s.N + 2) + 2 * x + 1) | (oa << 13) | ((ob - oa + 1) << 17) | (k << 21);
    }
    if (q + 1 < p.nlev) {
        const int Ec = p.g[q + 1].N + 2, Ra = DIM == 3 ? Ec : 1;
        const int zn = (k + 1) >> 1, yn = DIM == 3 ? (j + 1) >> 1 : 0;
        w[kB] = (((zn - staged_first(p, q, rank)) * Ra + yn) * Ec + x) | ((DIM == 3 && !(j & 1) ? 1 : 0) << 14) |
                ((!(k & 1) ? 1 : 0) << 15);
    }
    if (q > 0) {
        const int Nf = p.g[q - 1].N, haf = (Nf + 1) >> 1, rowsf = DIM == 3 ? Nf : 1;
        const int k1 = 2 * k - 1, o1 = plane_owner(p, q - 1, k1);
        const int row = DIM == 3 ? 2 * j - 2 : 0;
        const bool pl2 = k1 + 1 <= Nf, row2 = DIM == 3 && 2 * j <= Nf;
        const int o2 = pl2 ? plane_owner(p, q - 1, k1 + 1) : o1;
        w[kC] = (((k1 - plane_first(p, q - 1, o1)) * rowsf + row) * haf + 2 * x) | (o1 << 14) | (o2 << 18) |
                ((pl2 ? 1 : 0) << 22) | ((row2 ? 1 : 0) << 23) | ((o2 != o1 ? 1 : 0) << 24) |
                (((k1 - plane_first(p, q - 1, o1)) & 15) << 25);
    }
}

// Ghost cell t of the staged planes of level q + 1 in CTA `rank` (-1: none)
template <int DIM>
__host__ __device__ int plan_ghost(const MgSlabPlan &p, int q, int rank, int t)
{
    const MgGeom &g = p.g[q + 1];
    const int N = g.N, Ec = N + 2, Ra = DIM == 3 ? Ec : 1;
    const int Ka = staged_first(p, q, rank), Kb = staged_last(p, q, rank);
    if (plane_first(p, q, rank) >= plane_first(p, q, rank + 1))
        return -1;
    // the active index a ghost index comes from (itself where active), and the factor's kind
    auto from = [&](int v, int &kind) {
        kind = 0;
        if (v >= 1 && v <= N)
            return v;
        if (v == 0) {
            kind = 1;
            return 1;
        }
        if (g.tie) {
            kind = N >= 2 ? 1 : 0;
            return N >= 2 ? N - 1 : 1;
        }
        kind = 2;
        return N;
    };
    int n = 0;
    for (int K = Ka; K <= Kb; K++) {
        const bool kg = K < 1 || K > N;
        const int in_plane = kg ? Ra * Ec : DIM == 3 ? Ec * Ec - N * N : 2;
        if (t >= n + in_plane) {
            n += in_plane;
            continue;
        }
        int r = t - n, I, J = 0;
        if (kg) {
            J = r / Ec;
            I = r - J * Ec;
        } else if (DIM == 2) {
            I = r ? N + 1 : 0;
        } else if (r < 2 * Ec) {       // first and last row
            J = r < Ec ? 0 : N + 1;
            I = r < Ec ? r : r - Ec;
        } else {                       // two columns of the other rows
            r -= 2 * Ec;
            J = 1 + (r >> 1);
            I = r & 1 ? N + 1 : 0;
        }
        int kx, ky = 0, kz;
        const int i = from(I, kx), j = DIM == 3 ? from(J, ky) : 0, k = from(K, kz);
        const int dst = ((K - Ka) * Ra + J) * Ec + I, src = ((k - Ka) * Ra + j) * Ec + i;
        return dst | (src << 13) | ((kx | (ky << 2) | (kz << 4)) << 26);
    }
    return -1;
}

template <int DIM>
__global__ void __launch_bounds__(kT) k_slab_plan(const __grid_constant__ MgSlabPlan p, int *img)
{
    const int rank = blockIdx.x;
    int *o = img + (size_t)rank * p.words * kT + threadIdx.x;
    for (int q = 0; q < p.nlev; q++) {
        for (int u = 0; u < p.K[q]; u++) {
            int w[4];
            plan_item<DIM>(p, q, rank, (int)threadIdx.x + u * kT, w);
            o[(p.slot[q] + u) * kT] = w[kA];
            for (int a = kB; a <= kD; a++)
                o[(p.bcd[q] + 3 * u + a - 1) * kT] = w[a];
        }
        for (int u = 0; u < p.KG[q]; u++)
            o[(p.ghost[q] + u) * kT] = plan_ghost<DIM>(p, q, rank, (int)threadIdx.x + u * kT);
    }
    const int t = threadIdx.x;
    o[p.dpos * kT] = 0;
    if (t < p.dn) {
        const Shape s = shape_of<DIM>(p, p.nlev - 1, 0);
        const int i = t % s.N + 1, r = t / s.N, j = DIM == 3 ? r % s.N + 1 : 0, k = DIM == 3 ? r / s.N + 1 : r + 1;
        o[p.dpos * kT] = ((i + j + k) & 1) * s.cs + (k * s.R + j) * s.H + (i >> 1);
    }
}

template <class P, int DIM>
struct Engine {
    typedef typename P::T T;
    static constexpr bool kFix = P::kFix;
    static constexpr int kW = sizeof(T);
    const MgSlabPlan &pl;
    int rank, tid;
    unsigned npass = 0;     // colour passes on distributed levels so far (the same in every CTA)
    // phase bits of the four mbarriers: [from the previous, next CTA][even, odd pass]; kDead: this thread
    // has left a wait that had not ended
    unsigned phase = 0;
    static constexpr unsigned kDead = 16;

    __device__ explicit Engine(const MgSlabPlan &p) : pl(p), rank((int)cluster_rank_()), tid((int)threadIdx.x) {}

    // ---- shared memory: word arrays (potentials, scratch = pair sums or
    // staged coarse planes, right-hand sides, dense matrix, tables), then the
    // control words, then the plan words
    __device__ __forceinline__ static T *W()
    {
        extern __shared__ __align__(16) unsigned char smem_raw[];
        return reinterpret_cast<T *>(smem_raw);
    }
    __device__ __forceinline__ T *scratch() const { return W() + pl.scratch; }
    __device__ __forceinline__ T *fs() const { return W() + pl.fs; }
    __device__ __forceinline__ T *tab(int q) const { return W() + pl.tabs + P::kTab * 64 * q; }
    __device__ __forceinline__ int *ctrl() const { return reinterpret_cast<int *>(W() + pl.ctrl); }
    __device__ __forceinline__ int *sc() const { return ctrl(); }                       // fixed point: scale of every level
    __device__ __forceinline__ int *psc() const { return ctrl() + MG_SLAB_MAXLEV; }     // ... of its published potential
    // OR of magnitudes, [2 MAXLEV] pairs: residuals of level q at q, published
    // potentials at MAXLEV + q (level 0's, which is not published, in a solve);
    // orw: over this CTA, slots: of every CTA
    __device__ __forceinline__ unsigned *orw() const { return reinterpret_cast<unsigned *>(ctrl() + 2 * MG_SLAB_MAXLEV); }
    __device__ __forceinline__ unsigned *slots() const { return orw() + 4 * MG_SLAB_MAXLEV; }
    // per level, of the CTAs with the planes before and after its own: byte
    // address of their copies of its first and last plane, and of their
    // mbarriers for this CTA's values (0: none)
    __device__ __forceinline__ unsigned *nbr() const { return slots() + 64 * MG_SLAB_MAXLEV; }
    // this CTA's mbarriers: values from the previous (dir 0) and the next CTA, even and odd passes
    __device__ __forceinline__ unsigned mbar(int dir, int par) const
    {
        return shared_addr(nbr() + 4 * MG_SLAB_MAXLEV) + 8 * (2 * dir + par);
    }
    __device__ __forceinline__ int *failed() const { return reinterpret_cast<int *>(nbr() + 4 * MG_SLAB_MAXLEV + 8); }
    // bound of a wait (here, not in a register or the parameters: either cost 1.5 % of an FP64 V-cycle)
    __device__ __forceinline__ volatile int *wait_units() const { return failed() + 1; }
    // norm of the residual: 16 warps' and 16 CTAs' sums, the total
    __device__ __forceinline__ double *sums() const { return reinterpret_cast<double *>(nbr() + 4 * MG_SLAB_MAXLEV + 10); }
    __device__ __forceinline__ int *img() const { return ctrl() + MG_SLAB_CTRL; }
    __device__ __forceinline__ const int *gimg() const { return pl.img + (size_t)rank * pl.words * kT; }

    __device__ __forceinline__ bool dist(int q) const { return q < pl.nclu; }
    __device__ __forceinline__ int word_a(int slot) const { return img()[slot * kT + tid]; }
    // word B, C or D of pair u of level q
    __device__ __forceinline__ int word(int q, int u, int a) const
    {
        const int i = (pl.bcd[q] + 3 * u + a - 1) * kT + tid;
        return pl.K[q] == 1 ? img()[i] : gimg()[i];
    }
    // barrier between two phases: the cluster's, or this block's when the level lives in CTA 0
    __device__ __forceinline__ void sync(bool cluster) const
    {
        if (cluster)
            cluster_sync_();
        else
            __syncthreads();
    }

    // where this CTA keeps level q (word offset) and its neighbours keep the
    // copies of its first and last plane (byte address of the same word)
    struct Lev {
        int ph, cs, H, RH;
        unsigned prev, next, mprev, mnext;
        bool tie;
    };
    __device__ __forceinline__ Lev level(int q) const
    {
        Lev L;
        L.ph = pl.off[q];
        L.H = (pl.g[q].N + 3) >> 1;
        L.RH = (DIM == 3 ? pl.g[q].N + 2 : 1) * L.H;
        L.cs = (pl.po[q] + 2) * L.RH;
        L.tie = pl.g[q].L > 0 && pl.g[q].tie && pl.g[q].N >= 2;
        L.prev = nbr()[4 * q];
        L.next = nbr()[4 * q + 1];
        L.mprev = nbr()[4 * q + 2];
        L.mnext = nbr()[4 * q + 3];
        return L;
    }
    // the addresses level() reads, and the neighbours' mbarriers beside them (one thread per level)
    __device__ __forceinline__ void find_neighbours(int q) const
    {
        const Shape s = shape_of<DIM>(pl, q, rank);
        unsigned *n = nbr() + 4 * q;
        n[0] = n[1] = n[2] = n[3] = 0u;
        if (!dist(q) || s.total == 0)
            return;
        const unsigned w0 = shared_addr(W());
        const int RH = s.R * s.H;
        if (s.k0 > 1) {
            const int o = plane_owner(pl, q, s.k0 - 1);
            n[0] = cluster_addr(w0, o) + (s.k0 - plane_first(pl, q, o)) * RH * kW;
            n[2] = cluster_addr(mbar(1, 0), o);
        }
        if (s.k1 <= s.N) {
            const int o = plane_owner(pl, q, s.k1);
            n[1] = cluster_addr(w0, o) - (s.k1 - s.k0) * RH * kW;
            n[3] = cluster_addr(mbar(0, 0), o);
        }
    }
    // bytes of colour c of plane k that a neighbour sends
    __device__ __forceinline__ unsigned plane_bytes(int q, int c, int k) const
    {
        const int N = pl.g[q].N, cells = DIM == 3 ? N * N : N;
        // 3D: i + j even for half of the cells and the odd one; 2D: i odd
        const bool more = DIM == 3 ? ((c + k) & 1) == 0 : ((c + k) & 1) == 1;
        return (unsigned)(kW * ((cells + (more ? 1 : 0)) >> 1));
    }
    __device__ __forceinline__ bool has_failed() const { return *(volatile int *)failed() != 0; }
    // After a colour pass on level q: the neighbours' new values have arrived
    // and every thread of this CTA has written its own.  The wait is bounded;
    // after one that ran out this CTA waits for nothing more, sends what its
    // neighbours wait for, and the launch runs to its end and reports the
    // failure (k_slab).  Thread 0 no longer arrives then: no phase gets a second
    // arrival.  (Its test is of a register: this step is on the critical path, a
    // load from shared memory here cost 1 to 2 % of a V-cycle.)
    __device__ __forceinline__ void pass_sync(int q, const Lev &L, int c)
    {
        if (!dist(q)) {
            __syncthreads();
            return;
        }
        const int par = npass & 1;
        npass++;
        if (tid == 0 && !(phase & kDead)) {
            if (L.mprev)
                mbar_expect(mbar(0, par), plane_bytes(q, c, plane_first(pl, q, rank) - 1));
            if (L.mnext)
                mbar_expect(mbar(1, par), plane_bytes(q, c, plane_first(pl, q, rank + 1)));
        }
#pragma unroll
        for (int dir = 0; dir < 2; dir++)
            if (dir ? L.mnext : L.mprev) {
                const unsigned bit = 1u << (2 * dir + par);
                if (!mbar_try(mbar(dir, par), phase & bit ? 1u : 0u)) {
                    const long long t0 = clock64();
                    while (!mbar_try(mbar(dir, par), phase & bit ? 1u : 0u))
                        if (has_failed() || (int)((clock64() - t0) >> 21) >= *wait_units()) {
                            *(volatile int *)failed() = 1;
                            phase |= kDead;
                            break;
                        }
                }
                phase ^= bit;
            }
        __syncthreads();
    }

    __device__ __forceinline__ static int cls_odd(int A) { return ((A >> 21) & 3) | ((A >> 15) & 0x3c); }
    __device__ __forceinline__ static int cls_even(int A) { return ((A >> 22) & 2) | ((A >> 15) & 0x3c); }
    // the pair's cell of colour c: 0 the odd one, 1 the even one; whether it exists
    __device__ __forceinline__ static int s_of(int A, int c) { return ((A >> 14) & 1) ^ c; }
    __device__ __forceinline__ static bool has(int A, int c) { return (A >> (15 + s_of(A, c))) & 1; }

    // a new value into this CTA's slab and (plain stores, completed by a
    // cluster barrier) the neighbours' copies
    __device__ __forceinline__ void put(const Lev &L, int A, int i, T v) const
    {
        W()[i] = v;
        if ((A >> 24) & 3) {
            if ((A >> 24) & 1)
                st_cluster(L.prev + i * kW, v);
            if ((A >> 25) & 1)
                st_cluster(L.next + i * kW, v);
        }
    }
    // the same in a colour pass, the copies by stores that pass_sync waits for
    __device__ __forceinline__ void put_async(const Lev &L, int A, int i, T v, unsigned mb) const
    {
        W()[i] = v;
        if ((A >> 24) & 3) {
            if ((A >> 24) & 1)
                st_async(L.prev + i * kW, v, L.mprev + mb);
            if ((A >> 25) & 1)
                st_async(L.next + i * kW, v, L.mnext + mb);
        }
    }

    // neighbour sum of a pair's cell of colour c (s = 0: the odd, 1: the even
    // cell).  Ghost layers read zero on coarse levels; where x_N = 1 the ghost
    // cancels the left neighbour of the last cell (Sec. 2.4).
    __device__ __forceinline__ T nsum(const Lev &L, int A, int c, int s) const
    {
        const T *o = W() + L.ph + (1 - c) * L.cs + (A & 0x3fff);
        T sx = o[0] + o[1];
        o += s;
        T sy = T(0), sz;
        if (DIM == 3) {
            sy = o[-L.H] + o[L.H];
            sz = o[-L.RH] + o[L.RH];
        } else {
            sz = o[-L.H] + o[L.H];
        }
        if (L.tie) {
            if (s ? (A >> 23) & 1 : (A >> 22) & 1)
                sx = T(0);
            if (DIM == 3) {
                if ((A >> 18) & 1)
                    sy = T(0);
                if ((A >> 20) & 1)
                    sz = T(0);
            } else if ((A >> 18) & 1) {
                sz = T(0);
            }
        }
        return DIM == 3 ? (sx + sy) + sz : sx + sz;
    }

    // What a thread keeps of K of its pairs of a level while it sweeps: per
    // pair the plan word, and per colour the right-hand side and the reciprocal
    // diagonal.  Pairs that do not exist point at a cell inside the slab, so
    // everything but the stores is done for all of them without a branch, and
    // the loads of several pairs are in flight together.
    template <int K>
    struct Items {
        int A[K];
        T f[2][K], n[2][K];
    };
    template <int K>
    __device__ __forceinline__ void load_items(int q, int u0, Items<K> &it, bool with_f) const
    {
        const int slot = pl.slot[q] + u0;
        const T *tb = tab(q);
#pragma unroll
        for (int u = 0; u < K; u++) {
            const int A = word_a(slot + u);
            it.A[u] = A;
#pragma unroll
            for (int c = 0; c < 2; c++) {
                it.n[c][u] = tb[s_of(A, c) ? cls_even(A) : cls_odd(A)];
                it.f[c][u] = with_f ? fs()[(2 * (slot + u) + c) * kT + tid] : T(0);
            }
        }
    }
    // All K pairs of a thread on a level: held in registers from phase to
    // phase, or (more than two in 64 bits) read two at a time in each phase:
    // the kernel's shared memory leaves the L1 cache no room for spills.  A warp
    // without pairs skips the phases.
    template <int K>
    struct Held {
        static constexpr bool kStream = kFix && K > 2;
        Items<kStream ? 1 : K> it;
        bool on;
    };
    template <int K>
    __device__ __forceinline__ void hold(int q, Held<K> &h, bool with_f) const
    {
        if constexpr (!Held<K>::kStream)
            load_items(q, 0, h.it, with_f);
        h.on = K > 1 || __any_sync(0xffffffffu, (h.it.A[0] >> 15) & 1);
    }
    template <int K, typename Fn>
    __device__ __forceinline__ void each(int q, Held<K> &h, Fn &&fn) const
    {
        if constexpr (Held<K>::kStream) {
#pragma unroll 1
            for (int u = 0; u < K; u += 2) {
                Items<2> it;
                load_items(q, u, it, true);
                if (__any_sync(0xffffffffu, (it.A[0] >> 15) & 1))
                    fn(it, u);
            }
        } else if (h.on) {
            fn(h.it, 0);
        }
    }

    __device__ __forceinline__ T update(int q, T s, T f, T n) const
    {
        // rounded by what is added before the product: half of an inner cell's diagonal, and twice the
        // mean of what qmul drops, kl / 2^32 = 1/3 for K = 2^63 / 6 (one addition of three terms)
        if constexpr (kFix)
            return qmul<31>(s - f + (DIM == 3 ? 5 : 2), n);
        else
            return (s - pl.g[q].h2f * f) * n;
    }

    // colour c of a red-black sweep; send: the neighbours need the new values
    template <int c, int K>
    __device__ __forceinline__ void pass(int q, const Lev &L, const Items<K> &it, bool send) const
    {
        const unsigned mb = 8 * (npass & 1);
        T v[K];
#pragma unroll
        for (int u = 0; u < K; u++)
            v[u] = update(q, nsum(L, it.A[u], c, s_of(it.A[u], c)), it.f[c][u], it.n[c][u]);
#pragma unroll
        for (int u = 0; u < K; u++)
            if (has(it.A[u], c)) {
                const int i = L.ph + c * L.cs + (it.A[u] & 0x3fff) + s_of(it.A[u], c);
                if (send)
                    put_async(L, it.A[u], i, v[u], mb);
                else
                    W()[i] = v[u];
            }
    }

    // OR of the magnitudes m over this CTA into word pair w of orw
    __device__ __forceinline__ void block_or(fix m, int w) const
    {
        const unsigned hi = __reduce_or_sync(0xffffffffu, (unsigned)((unsigned long long)m >> 32));
        const unsigned lo = __reduce_or_sync(0xffffffffu, (unsigned)m);
        if ((tid & 31) == 0) {
            if (hi)
                atomicOr(orw() + 2 * w, hi);
            else if (lo)
                atomicOr(orw() + 2 * w + 1, lo);
        }
    }
    // ... and to every CTA of the cluster; also that of word pair w2 (-1: none)
    __device__ __forceinline__ void share_or(int w, int w2 = -1) const
    {
        __syncthreads();
        if (w2 >= 0 && tid >= 32)
            w = w2;
        const int to = tid & 31;
        if (to < pl.csize && tid < (w2 >= 0 ? 64 : 32)) {
            const unsigned dst = cluster_addr(shared_addr(slots() + (w * 16 + rank) * 2), to);
            st_cluster(dst, orw()[2 * w]);
            st_cluster(dst + 4, orw()[2 * w + 1]);
            if (w >= MG_SLAB_MAXLEV && rank == 0)
                st_cluster(cluster_addr(shared_addr(psc() + (w - MG_SLAB_MAXLEV)), to),
                           (unsigned)sc()[w - MG_SLAB_MAXLEV]);
        }
    }
    __device__ __forceinline__ void clear_or(int w) const
    {
        if (tid == 0)
            orw()[2 * w] = orw()[2 * w + 1] = 0u;
    }
    // bits of the largest magnitude, after the barrier that follows block_or (and share_or)
    __device__ __forceinline__ int or_bits(int w, bool cluster) const
    {
        unsigned hi = 0, lo = 0;
        if (cluster) {
            for (int t = 0; t < pl.csize; t++) {
                hi |= slots()[(w * 16 + t) * 2];
                lo |= slots()[(w * 16 + t) * 2 + 1];
            }
        } else {
            hi = orw()[2 * w];
            lo = orw()[2 * w + 1];
        }
        return hi ? 64 - __clz(hi) : 32 - __clz(lo);
    }
    __device__ __forceinline__ static fix mag(fix v) { return v < 0 ? ~v : v; }

    // Residual (step 4) of both cells of every pair, summed over the pair; the
    // OR of the sums' magnitudes, and in `pot` that of the potentials'.
    template <int K>
    __device__ __forceinline__ fix residual(int q, const Lev &L, const Items<K> &it, int u0, fix &pot) const
    {
        const T *tb = tab(q);
        const float ih2 = pl.g[q].inv_h2f;
        fix big = 0;
#pragma unroll
        for (int u = 0; u < K; u++) {
            const int A = it.A[u];
            T sum = T(0);
#pragma unroll
            for (int c = 0; c < 2; c++) {
                const int s = s_of(A, c), cls = s ? cls_even(A) : cls_odd(A);
                const T ns = nsum(L, A, c, s);
                const T v = W()[L.ph + c * L.cs + (A & 0x3fff) + s];
                T d;
                if constexpr (kFix) {
                    d = (2 * DIM) * v;
                    if (cls)
                        d = tb[64 + cls] * v + qmul<30>(v, tb[128 + cls]);
                    d = it.f[c][u] - ns + d;
                    pot |= mag(v);
                } else {
                    d = it.f[c][u] - (ns + tb[64 + cls] * v) * ih2;
                }
                sum += has(A, c) ? d : T(0);
            }
            if ((A >> 15) & 1)
                scratch()[tid + (u0 + u) * kT] = sum;
            if constexpr (kFix)
                big |= mag(sum);
        }
        return big;
    }

    // The scale of level q from the largest residual of level q - 1; the shift
    // of its pair sums into it (h_c^2 = 4 h_f^2, 2^-d average).
    __device__ __forceinline__ int restrict_scale(int q) const
    {
        const int bits = or_bits(q - 1, dist(q - 1)), s0 = sc()[q - 1];
        const int s1 = bits ? s0 + pl.tb[q] - (bits + 1) : s0;
        if (tid == 0)
            sc()[q] = s1;
        return s1 - s0 - (DIM == 3 ? 1 : 0);
    }

    // The right-hand sides of K pairs of level q: the 2^d-child average (step
    // 5) of level q - 1's residual.
    template <int K>
    __device__ __forceinline__ void restrict_into(int q, Items<K> &it, int u0, int sh, bool keep) const
    {
        const bool dup = dist(q - 1);
        const int slot = pl.slot[q] + u0;
        const int Nf = pl.g[q - 1].N, haf = (Nf + 1) >> 1, planef = haf * (DIM == 3 ? Nf : 1);
        const unsigned r0 = shared_addr(scratch());
#pragma unroll
        for (int u = 0; u < K; u++) {
            const int A = it.A[u];
            T o = T(0), e = T(0);
            if ((A >> 15) & 1) {
                const int w = word(q, u0 + u, kC);
                const bool even = (A >> 16) & 1, row2 = DIM == 3 && ((w >> 23) & 1), pl2 = (w >> 22) & 1;
                const int i1 = w & 0x3fff, i2 = (w >> 24) & 1 ? i1 - ((w >> 25) & 15) * planef : i1 + planef;
                T a0 = T(0), a1 = T(0), b0 = T(0), b1 = T(0), c0 = T(0), c1 = T(0), d0 = T(0), d1 = T(0);
                auto quad = [&](auto &&ld) {
                    ld(a0, 0, i1);
                    if (even)
                        ld(a1, 0, i1 + 1);
                    if (row2) {
                        ld(b0, 0, i1 + haf);
                        if (even)
                            ld(b1, 0, i1 + haf + 1);
                    }
                    if (pl2) {
                        ld(c0, 1, i2);
                        if (even)
                            ld(c1, 1, i2 + 1);
                        if (row2) {
                            ld(d0, 1, i2 + haf);
                            if (even)
                                ld(d1, 1, i2 + haf + 1);
                        }
                    }
                };
                if (dup) {
                    const unsigned r1 = cluster_addr(r0, (w >> 14) & 15), r2 = cluster_addr(r0, (w >> 18) & 15);
                    quad([&](T &v, int p, int i) { ld_cluster(v, (p ? r2 : r1) + i * kW); });
                } else {
                    quad([&](T &v, int, int i) { v = scratch()[i]; });
                }
                o = (a0 + b0) + (c0 + d0);
                e = (a1 + b1) + (c1 + d1);
            }
            if constexpr (kFix) {
                o = shift_by(o, sh);
                e = shift_by(e, sh);
            } else {
                o *= DIM == 3 ? 0.125f : 0.25f;
                e *= DIM == 3 ? 0.125f : 0.25f;
            }
            const bool odd0 = s_of(A, 0) == 0;   // the odd cell is red
            it.f[0][u] = odd0 ? o : e;
            it.f[1][u] = odd0 ? e : o;
            if (keep) {
                fs()[(2 * (slot + u)) * kT + tid] = it.f[0][u];
                fs()[(2 * (slot + u) + 1) * kT + tid] = it.f[1][u];
            }
        }
    }

    // The potential of a level that starts from zero after its first red
    // half-sweep, which sees zero neighbours
    template <int K>
    __device__ __forceinline__ void first_red(int q, const Lev &L, const Items<K> &it) const
    {
        const bool on = pl.nu_pre > 0;
#pragma unroll
        for (int u = 0; u < K; u++) {
            const int A = it.A[u], i = L.ph + (A & 0x3fff);
            if (has(A, 0))
                put(L, A, i + s_of(A, 0), on ? update(q, T(0), it.f[0][u], it.n[0][u]) : T(0));
            if (has(A, 1))
                put(L, A, i + L.cs + s_of(A, 1), T(0));
        }
    }

    // The last level of the plan and everything below it: the matrix of one
    // V-cycle times the right-hand side.  CTA 0; pl.dn cells, cell t at word
    // dpos[t] of the level; eight partial sums per cell.
    __device__ __forceinline__ void dense_solve(int q, const Lev &L, const Items<1> &it) const
    {
        const int n = pl.dn;
        T *vec = W() + pl.dvec, *part = vec + 64;
        const T *mat = W() + pl.dmat;
        const int *pos = img() + pl.dpos * kT;
        // right-hand sides by cell number (x fastest)
        const int A = it.A[0];
        if ((A >> 15) & 1) {
            const int w = 2 * tid - (pl.g[q].N & 1) * (tid / ((pl.g[q].N + 1) >> 1));
            const bool odd0 = s_of(A, 0) == 0;
            T o = odd0 ? it.f[0][0] : it.f[1][0], e = odd0 ? it.f[1][0] : it.f[0][0];
            if constexpr (!kFix) {
                o *= pl.g[q].h2f;
                e *= pl.g[q].h2f;
            }
            vec[w] = o;
            if ((A >> 16) & 1)
                vec[w + 1] = e;
        }
        __syncthreads();
        const int i = tid & 63, p = tid >> 6;
        T s = T(0);
        if (i < n)
            for (int j = p; j < n; j += 8) {
                if constexpr (kFix)
                    s += qmul<28>(vec[j], mat[j * n + i]);
                else
                    s += mat[j * n + i] * vec[j];
            }
        part[tid] = s;
        __syncthreads();
        if (tid < n) {
            T v = T(0);
#pragma unroll
            for (int k = 0; k < 8; k++)
                v += part[tid + 64 * k];
            W()[L.ph + pos[tid]] = v;
        }
        __syncthreads();
    }

    // The potential of level q into the staged planes of the CTAs that
    // interpolate from it.
    __device__ __forceinline__ void publish(int q, const Lev &L) const
    {
        const int Ec = pl.g[q].N + 2, ps = (DIM == 3 ? Ec : 1) * Ec;
        const bool dup = dist(q - 1);
        const unsigned s0 = shared_addr(scratch());
        fix big = 0;
        const int K = pl.K[q];
#pragma unroll 1
        for (int u = 0; u < K; u++) {
            const int A = word_a(pl.slot[q] + u), d = word(q, u, kD);
            if (!((A >> 15) & 1))
                continue;
            const int c1 = (A >> 14) & 1, b = L.ph + (A & 0x3fff), k = d >> 21;
            const bool even = (A >> 16) & 1;
            const T vo = W()[b + c1 * L.cs], ve = even ? W()[b + (1 - c1) * L.cs + 1] : T(0);
            if constexpr (kFix)
                big |= mag(vo) | mag(ve);
            if (!dup) {
                T *dst = scratch() + k * ps + (d & 0x1fff);
                dst[0] = vo;
                if (even)
                    dst[1] = ve;
                continue;
            }
            const int o1 = (d >> 13) & 15, n = (d >> 17) & 15;
            for (int o = o1; o < o1 + n; o++) {
                if (plane_first(pl, q - 1, o) == plane_first(pl, q - 1, o + 1))
                    continue;
                const unsigned dst = cluster_addr(s0, o) + ((k - staged_first(pl, q - 1, o)) * ps + (d & 0x1fff)) * kW;
                st_cluster(dst, vo);
                if (even)
                    st_cluster(dst + kW, ve);
            }
        }
        if constexpr (kFix) {
            block_or(big, MG_SLAB_MAXLEV + q);
            if (dup)
                share_or(MG_SLAB_MAXLEV + q);
        }
    }

    // The ghost cells of the staged planes of level q + 1 by the rule of Sec.
    // 2.4: left ghost -Phi_1, right ghost cR Phi_N, or -Phi_{N-1} where x_N = 1.
    __device__ __forceinline__ void fill_ghosts(int q) const
    {
        const int K = pl.KG[q];
#pragma unroll 1
        for (int u = 0; u < K; u++) {
            const int w = img()[(pl.ghost[q] + u) * kT + tid];
            if (w == -1)
                continue;
            T v = scratch()[(w >> 13) & 0x1fff];
#pragma unroll
            for (int a = 0; a < DIM; a++) {
                const int kind = (w >> (26 + 2 * (DIM == 2 && a ? 2 : a))) & 3;
                if (kind == 1)
                    v = -v;
                if (kind == 2) {
                    if constexpr (kFix)
                        v = pl.cri[q + 1] * v + qmul<30>(v, pl.crf[q + 1]);
                    else
                        v = pl.g[q + 1].cRf * v;
                }
            }
            scratch()[w & 0x1fff] = v;
        }
    }

    // The shift of level q + 1's potential to level q's scale, which is lowered
    // first if the correction is beyond its range, or (level 0 of a solve, whose
    // potential stays from cycle to cycle; every other starts from the range of
    // its right-hand side) the potential.
    __device__ __forceinline__ int prolong_scale(int q, const Lev &L) const
    {
        const bool cl = dist(q);
        const int bits = or_bits(MG_SLAB_MAXLEV + q + 1, cl), s1 = cl ? psc()[q + 1] : sc()[q + 1], s0 = sc()[q];
        const int pot = q == 0 && pl.solve ? or_bits(MG_SLAB_MAXLEV, cl) : 0;
        const int low = max(0, max(bits ? bits + s0 - s1 : 0, pot) - pl.top[q]);
        if (low) {
            __syncthreads();   // every thread has read the scale
            if (tid == 0)
                sc()[q] = s0 - low;
            for (int t = tid; t < 2 * L.cs; t += kT)
                W()[L.ph + t] = shift_even(W()[L.ph + t], low);
            T *f = fs() + 2 * pl.slot[q] * kT + tid;
            for (int u = 0; u < 2 * pl.K[q]; u++)
                f[u * kT] = shift_even(f[u * kT], low);
            sync(cl);
        }
        return s0 - low - s1;
    }

    // Prolongation and correction (step 10) of K pairs of level q from the
    // staged planes of level q + 1.
    template <int K>
    __device__ __forceinline__ void prolong_from(int q, const Lev &L, const Items<K> &it, int u0, int sh) const
    {
        const int Ec = pl.g[q + 1].N + 2, ps = (DIM == 3 ? Ec : 1) * Ec;
        // 3/4 - 1/4 interpolation along one axis
        auto mix = [](T near, T far) -> T {
            if constexpr (kFix)
                return (3 * near + far + 2) >> 2;
            else
                return 0.75f * near + 0.25f * far;
        };
#pragma unroll
        for (int u = 0; u < K; u++) {
            const int A = it.A[u];
            if (!((A >> 15) & 1))
                continue;
            const int bw = word(q, u0 + u, kB);
            const T *b = scratch() + (bw & 0x3fff);
            const int dy = (bw >> 14) & 1 ? Ec : -Ec, dz = (bw >> 15) & 1 ? ps : -ps;
            auto plane = [&](const T *z, T &o, T &e) {
                o = mix(z[1], z[0]);
                e = mix(z[1], z[2]);
                if (DIM == 3) {
                    const T *y = z + dy;
                    o = mix(o, mix(y[1], y[0]));
                    e = mix(e, mix(y[1], y[2]));
                }
            };
            T o0, e0, o1, e1;
            plane(b, o0, e0);
            plane(b + dz, o1, e1);
            T po = mix(o0, o1), pe = mix(e0, e1);
            if constexpr (kFix) {
                po = shift_by(po, sh);
                pe = shift_by(pe, sh);
            }
            const int c1 = (A >> 14) & 1, i = L.ph + (A & 0x3fff), io = i + c1 * L.cs, ie = i + (1 - c1) * L.cs + 1;
            put(L, A, io, W()[io] + po);
            if ((A >> 16) & 1)
                put(L, A, ie, W()[ie] + pe);
        }
    }

    // descent on level q: its right-hand side from the finer level (q > 0),
    // pre-smoothing, residual; the last level is solved
    template <int K>
    __device__ __forceinline__ void descend(int q, bool fresh)
    {
        const Lev L = level(q);
        const bool cl = dist(q);
        Held<K> h;
        if constexpr (kFix)
            clear_or(MG_SLAB_MAXLEV + q);
        const bool red = q > 0 || fresh, last = q + 1 == pl.nlev;
        hold(q, h, q == 0);
        int sh = 0;
        if constexpr (kFix)
            if (q > 0)
                sh = restrict_scale(q);
        if constexpr (K == 1)
            if (last) {
                if (h.on)
                    restrict_into(q, h.it, 0, sh, false);
                dense_solve(q, L, h.it);
                return;
            }
        if (red) {
            each(q, h, [&](auto &it, int u0) {
                if (q > 0)
                    restrict_into(q, it, u0, sh, true);
                first_red(q, L, it);
            });
            sync(cl);
        }
        auto colour = [&](auto c) {
            each(q, h, [&](auto &it, int) { this->template pass<decltype(c)::value>(q, L, it, true); });
            pass_sync(q, L, decltype(c)::value);
        };
#pragma unroll 1
        for (int s = 0; s < pl.nu_pre; s++) {
            if (s > 0 || !red)
                colour(std::integral_constant<int, 0>());
            colour(std::integral_constant<int, 1>());
        }
        fix big = 0, pot = 0;
        each(q, h, [&](auto &it, int u0) { big |= residual(q, L, it, u0, pot); });
        if constexpr (kFix) {
            const bool both = q == 0 && pl.solve;
            block_or(big, q);
            if (both)
                block_or(pot, MG_SLAB_MAXLEV);
            if (cl)
                share_or(q, both ? MG_SLAB_MAXLEV : -1);
        }
        sync(cl);
    }

    // ascent on level q: correction from level q + 1, post-smoothing (the
    // last sweep of a level that publishes is read by its own thread alone: no
    // barrier, nothing sent)
    template <int K>
    __device__ __forceinline__ void ascend(int q, bool last)
    {
        const Lev L = level(q);
        const bool cl = dist(q);
        Held<K> h;
        int sh = 0;
        if constexpr (kFix) {
            clear_or(q);
            sh = prolong_scale(q, L);
        }
        fill_ghosts(q);
        hold(q, h, true);
        __syncthreads();
        each(q, h, [&](auto &it, int u0) { prolong_from(q, L, it, u0, sh); });
        const bool fin = q > 0 || last;
        sync(cl);   // also: no CTA may publish into staged planes that another still reads
#pragma unroll 1
        for (int s = 0; s < pl.nu_post; s++) {
            const bool end = fin && s + 1 == pl.nu_post;
            each(q, h, [&](auto &it, int) { this->template pass<0>(q, L, it, true); });
            pass_sync(q, L, 0);
            each(q, h, [&](auto &it, int) { this->template pass<1>(q, L, it, !end); });
            if (!end)
                pass_sync(q, L, 1);
        }
    }

    __device__ __forceinline__ void descend_any(int q, bool fresh)
    {
        if (pl.K[q] == 1)
            descend<1>(q, fresh);
        else if (pl.K[q] == 2)
            descend<2>(q, fresh);
        else
            descend<4>(q, fresh);
    }
    __device__ __forceinline__ void ascend_any(int q, bool last)
    {
        if (pl.K[q] == 1)
            ascend<1>(q, last);
        else if (pl.K[q] == 2)
            ascend<2>(q, last);
        else
            ascend<4>(q, last);
    }

    // One V-cycle on the levels of the plan
    __device__ __forceinline__ void cycle(bool fresh, bool last)
    {
        // a level in CTA 0 alone: the other CTAs wait for its staged planes
        int q = 0;
        for (;; q++) {
            if (dist(q) || rank == 0)
                descend_any(q, fresh);
            if (q + 1 == pl.nlev)
                break;
        }
        for (; q > 0; q--) {
            if (dist(q) || rank == 0)
                publish(q, level(q));
            if (dist(q - 1))
                cluster_sync_();
            else if (rank == 0)
                __syncthreads();
            if (dist(q - 1) || rank == 0)
                ascend_any(q - 1, last);
        }
    }

    // x 2^e (e any)
    __device__ __forceinline__ static double scaled(double x, int e) { return scalbn(scalbn(x, e / 2), e - e / 2); }
    // The CTAs' parts of the norm, two sets in turn: a CTA without a share in the
    // level waits for nobody between two norms, so a part may arrive while
    // another still reads the last norm's.  The second set takes the slots of
    // the residual of the last possible level, which is solved and has none.
    __device__ __forceinline__ double *parts(int odd) const
    {
        return odd ? reinterpret_cast<double *>(slots() + 32 * (MG_SLAB_MAXLEV - 1)) : sums() + 16;
    }
    // |h^2 r|^2 over level 0 after cycle n: every CTA gets the same sum, added
    // in a fixed order.  A CTA scales its own part: a level that CTA 0 holds
    // alone changes its scale there alone (prolong_scale).
    __device__ __forceinline__ double square_sum(int K, int n) const
    {
        const Lev L = level(0);
        double acc = 0.0;
#pragma unroll 1
        for (int u = 0; u < K; u++) {
            Items<1> it;
            load_items(0, u, it, true);
            const int A = it.A[0];
#pragma unroll
            for (int c = 0; c < 2; c++)
                if (has(A, c)) {
                    const int s = s_of(A, c);
                    const fix v = W()[L.ph + c * L.cs + (A & 0x3fff) + s];
                    const double r = from_fix(it.f[c][0] - nsum(L, A, c, s) + (2 * DIM) * v, 0);
                    acc = fma(r, r, acc);
                }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            acc += __shfl_down_sync(0xffffffffu, acc, o);
        double *sm = sums();
        if ((tid & 31) == 0)
            sm[tid >> 5] = acc;
        __syncthreads();
        if (tid < 32) {
            acc = tid < kT / 32 ? sm[tid] : 0.0;
#pragma unroll
            for (int o = 8; o > 0; o >>= 1)
                acc += __shfl_down_sync(0xffffffffu, acc, o);
            acc = has_failed() ? CUDART_NAN : scaled(__shfl_sync(0xffffffffu, acc, 0), -2 * sc()[0]);
            if (tid < pl.csize)
                st_cluster(cluster_addr(shared_addr(parts(n & 1) + rank), tid), __double_as_longlong(acc));
        }
        cluster_sync_();
        if (tid < 32) {
            acc = tid < pl.csize ? parts(n & 1)[tid] : 0.0;
#pragma unroll
            for (int o = 8; o > 0; o >>= 1)
                acc += __shfl_down_sync(0xffffffffu, acc, o);
            if (tid == 0)
                sm[32] = acc;
        }
        __syncthreads();
        return sm[32];
    }

    // coefficient tables of every level, the dense matrix
    __device__ __forceinline__ void fill_tables() const
    {
        for (int t = tid; t < 64 * pl.nlev; t += kT) {
            const int q = t >> 6, c = t & 63;
            const MgGeom &g = pl.g[q];
            T *tb = tab(q);
            double d = -2.0 * DIM, nid = 1.0 / (2 * DIM);
            if (c && g.tab64) {
                d = g.tab64[c];
                nid = g.tab64[64 + c];
            }
            if constexpr (kFix) {
                // an inner cell's to the last bit: the double 1 / 6 is 2^-55 of it off, half a unit of 2^54
                tb[c] = c ? (fix)(nid * 9223372036854775808.0) : (fix)(((1ull << 63) + DIM) / (2 * DIM));
                const double fl = floor(-d);
                tb[64 + c] = (fix)fl;
                tb[128 + c] = (fix)((-d - fl) * 4611686018427387904.0);
            } else {
                tb[c] = (float)nid;
                tb[64 + c] = (float)d;
            }
        }
        if (rank == 0) {
            const T *src = static_cast<const T *>(pl.dense);
            T *dst = W() + pl.dmat;
            const int n = pl.dn * pl.dn;
#pragma unroll 4
            for (int t = tid; t < n; t += kT)
                dst[t] = src[t];
        }
    }
};

// exponent bound: |x| < 2^result for the largest magnitude with this high word
__device__ __forceinline__ int exp_bound(unsigned hi) { return hi ? (int)(hi >> 20) - 1022 : -4000; }

template <class P, int DIM>
__global__ void __launch_bounds__(kT, 1) k_slab(const __grid_constant__ MgSlabPlan pl)
{
    typedef typename P::T T;
    typedef typename P::G G;
    __shared__ unsigned s_max[2], s_all[2][16];
    Engine<P, DIM> en(pl);
    const int tid = threadIdx.x, rank = en.rank, C = pl.csize;
    const int wid = tid >> 5, lane = tid & 31, nw = kT / 32;
    // before the predecessor has finished: the plan image, the tables, the
    // potentials to zero (their ghost layers stay zero)
    {
        const int nw16 = pl.nimg * (kT / 4);
        const uint4 *src = reinterpret_cast<const uint4 *>(en.gimg());
        uint4 *dst = reinterpret_cast<uint4 *>(en.img());
#pragma unroll 4
        for (int t = tid; t < nw16; t += kT)
            dst[t] = src[t];
    }
    for (int t = tid; t < pl.zero16; t += kT)
        reinterpret_cast<uint4 *>(en.W())[t] = make_uint4(0, 0, 0, 0);
    en.fill_tables();
    for (int t = tid; t < MG_SLAB_CTRL; t += kT)
        en.ctrl()[t] = 0;
    if (tid < 2)
        s_max[tid] = 0u;
    __syncthreads();
    if (tid == 0)
        *en.wait_units() = pl.fault ? 1 : kWaitUnits;
    if (tid < 4) {
        // (pl.fault: CTA 1's even passes wait for an arrival that does not come)
        mbar_init(en.mbar(tid >> 1, tid & 1), pl.fault && rank == 1 && !(tid & 1) ? 2 : 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < pl.nlev)
        en.find_neighbours(tid);
    cluster_sync_();   // every CTA has started: its shared memory may be written
    pdl_begin();
    const Shape S = shape_of<DIM>(pl, 0, rank);
    const MgGeom &g0 = pl.g[0];
    const int N = g0.N, E = N + 2;
    T *ph0 = en.W() + pl.off[0];
    const G *gphi = static_cast<const G *>(pl.phi), *gf = static_cast<const G *>(pl.f);
    auto gidx = [&](int i, int j, int k) { return (size_t)(DIM == 3 ? k * E + j : k) * E + i; };
    // level 0 of the plan from global memory: the right-hand side to its
    // threads, the potential (with its ring) to the slab, a warp per row
    unsigned mphi = 0, mf = 0;
    G fo[MG_SLAB_MAXK], fe[MG_SLAB_MAXK];
#pragma unroll
    for (int u = 0; u < MG_SLAB_MAXK; u++) {
        fo[u] = fe[u] = G(0);
        if (u < pl.K[0] && ((en.word_a(u) >> 15) & 1)) {
            const int d = en.word(0, u, kD);
            const G *src = gf + gidx(2 * (d & 0x3ff) + 1, (d >> 10) & 0x3ff, d >> 20);
            fo[u] = src[0];
            if ((en.word_a(u) >> 16) & 1)
                fe[u] = src[1];
        }
    }
    if (!pl.zero_start && S.total > 0) {
        const int rows = DIM == 3 ? E : 1, ka = S.k0 - 1, nr = rows * (S.k1 - S.k0 + 2);
        constexpr int U = 4;
        for (int i0 = 0; i0 < E; i0 += 32)
            for (int r0 = wid; r0 < nr; r0 += nw * U) {
                const int i = i0 + lane;
                G v[U];
#pragma unroll
                for (int u = 0; u < U; u++) {
                    const int r = r0 + u * nw, kz = r / rows;
                    v[u] = G(0);
                    if (r < nr && i < E)
                        v[u] = gphi[gidx(i, r - kz * rows, ka + kz)];
                }
#pragma unroll
                for (int u = 0; u < U; u++) {
                    const int r = r0 + u * nw, kz = r / rows, j = r - kz * rows;
                    if (r < nr && i < E) {
                        T &d = ph0[((i + j + ka + kz) & 1) * S.cs + (kz * S.R + j) * S.H + (i >> 1)];
                        if constexpr (P::kFix) {
                            d = __double_as_longlong(v[u]);
                            mphi = max(mphi, (unsigned)__double2hiint(v[u]) & 0x7fffffffu);
                        } else {
                            d = v[u];
                        }
                    }
                }
            }
    }
    // right-hand sides by colour to their threads' words
    auto keep = [&](auto &&conv) {
#pragma unroll
        for (int u = 0; u < MG_SLAB_MAXK; u++)
            if (u < pl.K[0]) {
                const bool odd0 = ((en.word_a(u) >> 14) & 1) == 0;
                en.fs()[(2 * u) * kT + tid] = conv(odd0 ? fo[u] : fe[u]);
                en.fs()[(2 * u + 1) * kT + tid] = conv(odd0 ? fe[u] : fo[u]);
            }
    };
    bool bad = false;
    if constexpr (P::kFix) {
        // the scale of the plan's first level from the largest magnitudes over
        // the cluster; infinities and NaN make every result NaN
#pragma unroll
        for (int u = 0; u < MG_SLAB_MAXK; u++)
            mf = max(mf, max((unsigned)__double2hiint(fo[u]) & 0x7fffffffu, (unsigned)__double2hiint(fe[u]) & 0x7fffffffu));
        mphi = __reduce_max_sync(0xffffffffu, mphi);
        mf = __reduce_max_sync(0xffffffffu, mf);
        if (lane == 0) {
            atomicMax(&s_max[0], mphi);
            atomicMax(&s_max[1], mf);
        }
        __syncthreads();
        if (tid < C) {
            st_cluster(cluster_addr(shared_addr(&s_all[0][rank]), tid), s_max[0]);
            st_cluster(cluster_addr(shared_addr(&s_all[1][rank]), tid), s_max[1]);
        }
        cluster_sync_();
        mphi = mf = 0;
        for (int t = 0; t < C; t++) {
            mphi = max(mphi, s_all[0][t]);
            mf = max(mf, s_all[1][t]);
        }
        bad = mphi >= 0x7ff00000u || mf >= 0x7ff00000u;
        const int gb = mf ? exp_bound(mf) + pl.h2e : -4000;   // h^2 = h2k 2^(h2e - 62)
        const int s0 = mf || mphi ? min(pl.tb[0] - gb, pl.top[0] - exp_bound(mphi)) : 0;
        if (tid == 0)
            en.sc()[0] = s0;
        if (!pl.zero_start)
            for (int t = tid; t < 2 * S.cs; t += kT)
                ph0[t] = to_fix(__longlong_as_double(ph0[t]), s0);
        keep([&](double f) { return to_fix_times(f, pl.h2k, s0 + pl.h2e); });
    } else {
        keep([](float f) { return f; });
    }
    cluster_sync_();
    // V-cycles: `cycles` of them, or (solve; the loop of Sec. 2.3 step 14)
    // until |r| < tol |b|, both in FP64, |b| and the first |r| from the norm
    // kernel before this launch.  Compared as squares; r = 0 meets any tol > 0.
    const bool solve = P::kFix && pl.solve;
    double bb = 0.0, r2 = 0.0, goal = 0.0;
    int n = 0;
    auto more = [&]() { return n < pl.cycles && (!solve || (isfinite(r2) && !(r2 < goal) && !(r2 == 0.0 && goal >= 0.0 && pl.tol > 0.0))); };
    bool go = pl.cycles > 0;
    if (solve) {
        bb = pl.scal[0];
        r2 = pl.scal[1];
        goal = pl.tol * pl.tol * bb;
        // (a first |r| that is not finite: one step finds that out, as in the loop of launches)
        go = isfinite(bb) && bb > 0.0 && (more() || (!isfinite(r2) && go));
    }
    while (go) {
        if (!bad)
            en.cycle(pl.zero_start && n == 0, !solve && n + 1 == pl.cycles);
        n++;
        if constexpr (P::kFix)
            if (solve) {
                r2 = CUDART_NAN;
                if (!bad)
                    r2 = en.square_sum(pl.K[0], n) * g0.inv_h2 * g0.inv_h2;
            }
        go = more();
    }
    if (solve && rank == 0 && tid == 0) {
        MgSolveCtl c{};
        c.cycles = c.outer = n;
        c.bnorm = sqrt(bb);
        c.rel = c.bnorm > 0.0 ? sqrt(r2) / c.bnorm : 0.0;
        c.status = isfinite(c.bnorm) && (n == 0 || isfinite(c.rel)) ? 0 : 6;
        *pl.ctl = c;
    }
    // the potential of the plan's first level back to global memory
    if (n > 0) {
        G *out = static_cast<G *>(pl.phi);
        int s0 = 0;
        if constexpr (P::kFix)
            s0 = en.sc()[0];
#pragma unroll
        for (int u = 0; u < MG_SLAB_MAXK; u++) {
            if (u >= pl.K[0])
                break;
            const int A = en.word_a(u);
            if (!((A >> 15) & 1))
                continue;
            const int d = en.word(0, u, kD), c1 = (A >> 14) & 1, b = A & 0x3fff;
            G *dst = out + gidx(2 * (d & 0x3ff) + 1, (d >> 10) & 0x3ff, d >> 20);
            auto value = [&](T v) -> G {
                if constexpr (P::kFix)
                    return bad ? __longlong_as_double(0x7ff8000000000000ll) : from_fix(v, s0);
                else
                    return v;
            };
            dst[0] = value(ph0[c1 * S.cs + b]);
            if ((A >> 16) & 1)
                dst[1] = value(ph0[(1 - c1) * S.cs + b + 1]);
        }
    }
    if (pl.ctl && !solve && rank == 0 && tid == 0)
        inner_step_count(pl.ctl, pl.hi);
    if (tid < C && en.has_failed())
        st_cluster(cluster_addr(shared_addr(en.failed()), tid), 1u);
    cluster_sync_();   // no CTA leaves while another may still write to its shared memory
    // A wait ran out, in whichever CTA: the potential becomes NaN, and what was
    // sent but never waited for gets time to arrive before its destination
    // leaves.
    if (en.has_failed()) {
        for (int u = 0; u < pl.K[0]; u++) {
            const int A = en.word_a(u), d = en.word(0, u, kD);
            G *dst = static_cast<G *>(pl.phi) + gidx(2 * (d & 0x3ff) + 1, (d >> 10) & 0x3ff, d >> 20);
            if ((A >> 15) & 1)
                dst[0] = G(CUDART_NAN);
            if ((A >> 16) & 1)
                dst[1] = G(CUDART_NAN);
        }
        if (rank == 0 && tid == 0) {
            if (pl.err)
                *pl.err = 7;   // MG_ETIMEOUT
            if (solve)
                pl.ctl->status = 6;
        }
        const long long t0 = clock64();
        while (clock64() - t0 < kDrainCycles)
            ;
    }
}

template <class P, int DIM>
cudaError_t slab_prepare()
{
    cudaError_t e = cudaFuncSetAttribute(k_slab<P, DIM>, cudaFuncAttributeMaxDynamicSharedMemorySize, MG_SLAB_SMEM_MAX);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_slab<P, DIM>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

void slab_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute *at, int csize, size_t smem, cudaStream_t s)
{
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3(csize);
    cfg.blockDim = dim3(kT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = csize;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = mg_pdl_enabled() ? 2 : 1;
}

}  // namespace

// The largest cluster (16 CTAs, else 8) that the device can hold at the
// largest shared-memory size, 0 if none.
int mg_slab_prepare()
{
    if (slab_prepare<PrecF32, 2>() || slab_prepare<PrecF32, 3>() || slab_prepare<PrecFix, 2>() ||
        slab_prepare<PrecFix, 3>()) {
        cudaGetLastError();
        return 0;
    }
    for (int cs : {16, 8}) {
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute at[2];
        slab_config(cfg, at, cs, MG_SLAB_SMEM_MAX, nullptr);
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, k_slab<PrecFix, 3>, &cfg) == cudaSuccess && n > 0)
            return cs;
        cudaGetLastError();
    }
    return 0;
}

// Shared-memory layout of levels g[0..nlev-1]; the levels of more than `cut`
// cells per edge are distributed.  False when it does not fit.
bool mg_slab_layout(int dim, bool fp32, int csize, const MgGeom *g, int nlev, int cut, int nu_pre, int nu_post,
                    MgSlabPlan &p)
{
    // the plan ends with the first level of at most 64 cells
    int last = 1;
    while (last < nlev && std::pow((double)g[last].N, dim) > 64.5)
        last++;
    if ((csize != 8 && csize != 16) || last >= nlev || last >= MG_SLAB_MAXLEV)
        return false;
    nlev = last + 1;
    p = MgSlabPlan{};
    p.nlev = nlev;
    p.csize = csize;
    p.lgc = csize == 16 ? 4 : 3;
    p.nu_pre = nu_pre;
    p.nu_post = nu_post;
    int e2 = 0;
    p.h2k = std::llrint(std::ldexp(std::frexp(g[0].h2, &e2), 62));
    p.h2e = e2;
    const size_t w = fp32 ? 4 : 8;
    size_t off = 0, scratch = 0;
    const int lognu = (int)std::ceil(std::log2(1.0 + nu_pre + nu_post));
    auto align = [](size_t v) { return (v + 3) & ~(size_t)3; };
    for (int q = 0; q < nlev; q++) {
        p.g[q] = g[q];
        if (g[q].N > cut && q == p.nclu && q + 1 < nlev)
            p.nclu = q + 1;
    }
    for (int q = 0; q < nlev; q++) {
        const int N = g[q].N, H = (N + 3) >> 1, R = dim == 3 ? N + 2 : 1, ha = (N + 1) >> 1, rows = dim == 3 ? N : 1;
        p.po[q] = q < p.nclu ? (N + csize - 1) / csize : N;
        const size_t cs = (size_t)(p.po[q] + 2) * R * H, items = (size_t)p.po[q] * rows * ha;
        if (cs > 0x3fff || items > 0x3fff || N > 1020 || (q < p.nclu && p.po[q] > 16))   // fields of the plan words
            return false;
        p.off[q] = (int)off;
        off = align(off + 2 * cs);
        const int k = (int)((items + kT - 1) / kT);
        if (k > MG_SLAB_MAXK)
            return false;
        p.K[q] = k <= 2 ? k : 4;
        p.slot[q] = p.nslot;
        p.nslot += p.K[q];
        scratch = std::max(scratch, items);
        if (q + 1 < nlev) {
            const size_t Ec = g[q + 1].N + 2, planes = q < p.nclu ? (size_t)p.po[q] / 2 + 5 : Ec + 1;
            const size_t staged = planes * Ec * (dim == 3 ? Ec : 1);
            if (staged > 0x1fff)
                return false;
            scratch = std::max(scratch, staged);
            for (int r = 0; r < csize; r++) {
                if (plane_first(p, q, r) >= plane_first(p, q, r + 1))
                    continue;
                size_t cells = 0;   // ghost cells of this CTA's staged planes
                for (int K = staged_first(p, q, r); K <= staged_last(p, q, r); K++) {
                    const bool whole = K < 1 || K > g[q + 1].N;
                    const size_t Nc = Ec - 2;
                    cells += dim == 3 ? Ec * Ec - (whole ? 0 : Nc * Nc) : whole ? Ec : 2;
                }
                p.KG[q] = std::max(p.KG[q], (int)((cells + kT - 1) / kT));
            }
        }
        const double fl = std::floor(g[q].cR);
        p.cri[q] = (int)fl;
        p.crf[q] = (long long)((g[q].cR - fl) * 4611686018427387904.0);
        // fixed point: the boundary cells' diagonals can be larger than 2 d
        double dmax = 2.0 * dim;
        for (int c = 0; c < 64; c++) {
            double d = mg_axis_diag(c & 3, g[q]) + mg_axis_diag((c >> 2) & 3, g[q]);
            if (dim == 3)
                d += mg_axis_diag((c >> 4) & 3, g[q]);
            if (g[q].L > 0)
                dmax = std::max(dmax, -d);
        }
        const int db = (int)std::ceil(std::log2(dmax / 6.0 > 1.0 ? dmax / 6.0 : 1.0));
        p.tb[q] = std::min(57 - db - lognu, q + 1 == nlev ? 54 : 57);
        p.top[q] = 57 - db;
        // the finest level of a refinement level keeps its right-hand side and potential from cycle to
        // cycle and their bits are those of the result: with a potential of 2^57, as much again from a
        // correction and nu f / dim from the sweeps, 2 (f + 4 dim Phi) stays below 2^63
        if (g[q].L == 0) {
            const double room = (std::ldexp(1.0, 62) - std::ldexp(1.0, 57)) / (4 * dim) - std::ldexp(1.0, 58);
            p.tb[q] = std::min(57, (int)std::floor(std::log2(room * dim / (nu_pre + nu_post))));
        }
    }
    // plan words: A of every slot, B C D of the levels with one pair per thread, ghosts (copied to
    // shared memory), then B C D of the other levels
    p.words = p.nslot;
    for (int q = 0; q < nlev; q++)
        if (p.K[q] == 1) {
            p.bcd[q] = p.words;
            p.words += 3;
        }
    for (int q = 0; q < nlev; q++) {
        p.ghost[q] = p.words;
        p.words += p.KG[q];
    }
    p.dpos = p.words++;          // word offset of every cell of the last level
    p.nimg = p.words;
    for (int q = 0; q < nlev; q++)
        if (p.K[q] > 1) {
            p.bcd[q] = p.words;
            p.words += 3 * p.K[q];
        }
    p.zero16 = (int)(off * w / 16);
    p.scratch = (int)off;
    off = align(off + scratch);
    p.fs = (int)off;
    off += (size_t)2 * (p.nslot - 1) * kT;   // the last level's right-hand side is used at once
    p.dn = 1;
    for (int a = 0; a < dim; a++)
        p.dn *= g[nlev - 1].N;
    p.dmat = (int)off;
    off = align(off + (size_t)p.dn * p.dn);
    p.dvec = (int)off;
    off += 64 + kT;
    p.tabs = (int)off;
    off = align(off + (size_t)(fp32 ? 2 : 3) * 64 * nlev);
    p.ctrl = (int)off;
    p.smem = off * w + (size_t)MG_SLAB_CTRL * 4 + (size_t)p.nimg * kT * 4;
    return p.K[nlev - 1] == 1 && p.smem <= MG_SLAB_SMEM_MAX;
}

// Matrix of one V-cycle from a zero potential on levels g[0..nlev-1] (all of
// them, down to one cell): column j holds the potential of level 0 for the
// right-hand side h^2 f = unit vector j, cells x fastest.  FP64 on the host,
// at most 64 cells.  The columns go through each step side by side (a row of n0
// values per cell), along lists of neighbours made once: creating a handle
// waits for this (4^3, V(2,2): 0.4 ms one column at a time).
void mg_slab_dense(int dim, const MgGeom *g, int nlev, int nu_pre, int nu_post, double *mat)
{
    struct Cell {
        int nb[6], nn, parent, colour;   // neighbours in the order of the stencil's sum
        double d;                        // diagonal with the ghost rule folded in
        int at[8];                       // the coarse cells that it is interpolated from
        double w[8];
    };
    struct Level {
        std::vector<Cell> cell;
        std::vector<double> phi, f;      // f as h^2 f
    };
    auto cells = [&](int q) { return (dim == 3 ? g[q].N : 1) * g[q].N * g[q].N; };
    const int n0 = cells(0), corners = 1 << dim;
    // coarse index with ghosts -> active index, factor
    auto ghost = [&](int q, int I, double &c) {
        const int N = g[q].N;
        c = 1.0;
        if (I >= 1 && I <= N)
            return I;
        if (I == 0) {
            c = -1.0;
            return 1;
        }
        if (g[q].tie) {
            c = N >= 2 ? -1.0 : 1.0;
            return N >= 2 ? N - 1 : 1;
        }
        c = g[q].cR;
        return N;
    };
    std::vector<Level> lev(nlev);
    for (int q = 0; q < nlev; q++) {
        Level &l = lev[q];
        const int N = g[q].N, Nc = q + 1 < nlev ? g[q + 1].N : 0;
        l.cell.resize(cells(q));
        l.phi.assign((size_t)cells(q) * n0, 0.0);
        l.f.assign((size_t)cells(q) * n0, 0.0);
        for (int t = 0; t < cells(q); t++) {
            Cell &c = l.cell[t];
            const int a[3] = {t % N + 1, t / N % N + 1, dim == 3 ? t / (N * N) + 1 : 0}, st[3] = {1, N, N * N};
            c.colour = (a[0] + a[1] + a[2]) & 1;
            c.nn = 0;
            c.d = 0.0;
            for (int x = 0; x < dim; x++) {
                const bool lo = a[x] == 1, hi = a[x] == N;
                c.d += mg_axis_diag((lo ? 1 : 0) | (hi ? 2 : 0), g[q]);
                if (!lo && !(hi && g[q].tie && N >= 2))
                    c.nb[c.nn++] = t - st[x];
                if (!hi)
                    c.nb[c.nn++] = t + st[x];
            }
            c.parent = -1;
            if (!Nc)
                continue;
            const int P[3] = {(a[0] + 1) / 2, (a[1] + 1) / 2, (a[2] + 1) / 2};
            if (P[0] <= Nc && P[1] <= Nc && P[2] <= Nc)
                c.parent = (dim == 3 ? (P[2] - 1) * Nc * Nc : 0) + (P[1] - 1) * Nc + P[0] - 1;
            for (int m = 0; m < corners; m++) {
                c.w[m] = 1.0;
                int at[3] = {1, 1, 1};
                for (int x = 0; x < dim; x++) {
                    const int near = (a[x] + 1) / 2, far = near + (a[x] & 1 ? -1 : 1);
                    double k;
                    at[x] = ghost(q + 1, (m >> x) & 1 ? far : near, k);
                    c.w[m] *= k * ((m >> x) & 1 ? 0.25 : 0.75);
                }
                c.at[m] = (at[2] - 1) * Nc * Nc + (at[1] - 1) * Nc + at[0] - 1;
            }
        }
    }
    std::vector<double> sum(n0);
    auto neighbours = [&](const Level &l, const Cell &c) {
        std::fill(sum.begin(), sum.end(), 0.0);
        for (int e = 0; e < c.nn; e++) {
            const double *v = &l.phi[(size_t)c.nb[e] * n0];
            for (int k = 0; k < n0; k++)
                sum[k] += v[k];
        }
    };
    auto smooth = [&](int q, int sweeps) {
        Level &l = lev[q];
        for (int sw = 0; sw < (g[q].N == 1 && sweeps > 0 ? 1 : sweeps); sw++)
            for (int colour = 0; colour < 2; colour++)
                for (size_t t = 0; t < l.cell.size(); t++) {
                    const Cell &c = l.cell[t];
                    if (c.colour != colour)
                        continue;
                    neighbours(l, c);
                    for (int k = 0; k < n0; k++)
                        l.phi[t * n0 + k] = (sum[k] - l.f[t * n0 + k]) / -c.d;
                }
    };
    for (int k = 0; k < n0; k++)
        lev[0].f[(size_t)k * n0 + k] = 1.0;
    smooth(0, nu_pre);
    for (int q = 0; q + 1 < nlev; q++) {
        Level &l = lev[q];
        for (size_t t = 0; t < l.cell.size(); t++) {   // h_c^2 = 4 h_f^2, 2^-d average
            const Cell &c = l.cell[t];
            if (c.parent < 0)
                continue;
            neighbours(l, c);
            double *fc = &lev[q + 1].f[(size_t)c.parent * n0];
            for (int k = 0; k < n0; k++)
                fc[k] += (dim == 3 ? 0.5 : 1.0) * (l.f[t * n0 + k] - sum[k] - c.d * l.phi[t * n0 + k]);
        }
        smooth(q + 1, nu_pre);
    }
    for (int q = nlev - 2; q >= 0; q--) {
        Level &l = lev[q];
        for (size_t t = 0; t < l.cell.size(); t++) {
            const Cell &c = l.cell[t];
            std::fill(sum.begin(), sum.end(), 0.0);
            for (int m = 0; m < corners; m++) {
                const double *v = &lev[q + 1].phi[(size_t)c.at[m] * n0];
                for (int k = 0; k < n0; k++)
                    sum[k] += c.w[m] * v[k];
            }
            for (int k = 0; k < n0; k++)
                l.phi[t * n0 + k] += sum[k];
        }
        smooth(q, nu_post);
    }
    for (int t = 0; t < n0; t++)
        for (int k = 0; k < n0; k++)
            mat[(size_t)k * n0 + t] = lev[0].phi[(size_t)t * n0 + k];
}

size_t mg_slab_image_bytes(const MgSlabPlan &p) { return (size_t)p.csize * p.words * kT * sizeof(int); }

cudaError_t mg_launch_slab_plan(int dim, const MgSlabPlan &p, int *img, cudaStream_t s)
{
    if (dim == 3)
        k_slab_plan<3><<<p.csize, kT, 0, s>>>(p, img);
    else
        k_slab_plan<2><<<p.csize, kT, 0, s>>>(p, img);
    return cudaGetLastError();
}

cudaError_t mg_launch_slab(int dim, bool fp32, const MgSlabPlan &p, cudaStream_t s)
{
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[2];
    slab_config(cfg, at, p.csize, p.smem, s);
    if (fp32)
        return dim == 3 ? cudaLaunchKernelEx(&cfg, k_slab<PrecF32, 3>, p) : cudaLaunchKernelEx(&cfg, k_slab<PrecF32, 2>, p);
    return dim == 3 ? cudaLaunchKernelEx(&cfg, k_slab<PrecFix, 3>, p) : cudaLaunchKernelEx(&cfg, k_slab<PrecFix, 2>, p);
}
