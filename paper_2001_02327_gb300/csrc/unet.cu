// unet.cu -- the learned initial guess: a small 3D U-Net that predicts the
// correction of a refinement level's interpolated initial potential, with
// hand-written BF16 tensor-core convolutions (FP32 accumulate), its backward
// pass, AdamW training and the hook into the solver.
//
// Network (channels-last BF16 activations, n = 2^k spatial edge, 4 scales):
//   x0 = [4 pi G rho h^2 / s, Phi_interp / s, h^2 r / s_r]   on Omega, with
//        r = 4 pi G rho - lap(Phi_interp) the residual of the interpolated
//        potential, s = max |Phi_interp|, s_r = max |h^2 r|
//   a0 = relu(c3(x0; 3->16))      s0 = relu(c3(a0; 16->16))          n
//   a1 = relu(c3(pool s0; 16->32)) s1 = relu(c3(a1; 32->32))         n/2
//   s2 = relu(c3(pool s1; 32->64))                                   n/4
//   a3 = relu(c3(pool s2; 64->64))                                   n/8
//   d2 = relu(c3([up a3, s2]; 128->32))                              n/4
//   d1 = relu(c3([up d2, s1]; 64->16))                               n/2
//   d0 = relu(c3([up d1, s0]; 32->16))                               n
//   y  = c1(d0; 16->1);   Phi_guess = Phi_interp + (s_r n^2 / 16) y  on Omega
// (the inverse 7-point Laplacian amplifies smooth residuals by ~n^2: the
// factor keeps y of order one across level sizes).
// c3: 3x3x3 convolution, zero padding, bias; pool: 2x2x2 mean; up: nearest.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/unet.h"

namespace {

typedef __nv_bfloat16 bf16;

constexpr int kT = 256;

inline int blocks_for(long n, int cap = 152 * 32)
{
    long b = (n + kT - 1) / kT;
    return (int)(b < 1 ? 1 : (b > cap ? cap : b));
}

__device__ __forceinline__ uint32_t pack2(float a, float b)
{
    __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t *>(&v);
}
// the 8 BF16 values of a 16-byte word
__device__ __forceinline__ void unpack8(uint4 q, float *f)
{
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int i = 0; i < 4; i++) {
        f[2 * i] = __uint_as_float(w[i] << 16);
        f[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
    }
}

__device__ __forceinline__ uint32_t ld2(const bf16 *p) { return *reinterpret_cast<const uint32_t *>(p); }
__device__ __forceinline__ uint32_t ld2(const float *p)
{
    const float2 f = *reinterpret_cast<const float2 *>(p);
    return pack2(f.x, f.y);
}

// D += A (16x16, row) * B (16x8, col), BF16 in, FP32 accumulate
__device__ __forceinline__ void mma16816(float *d, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};\n"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// 3x3x3 convolution as an implicit GEMM on the tensor cores.
//   out[v][nn] = sum_{tap, c} in[v +/- off(tap)][c] * W[tap][nn][c]  (+ bias, relu)
// in: [V][CK] (CK a multiple of 16), W: [27][NT*8][CK] BF16, V = batch * n^3
// with n = 2^lg.  FLIP = true gathers at v - off (the transpose convolution of
// the backward data pass).  A block of 4 warps covers 64 voxels; a warp owns
// 16 voxels and all NT*8 output channels.
template <int NT, bool FLIP, typename TIn>
__global__ void __launch_bounds__(128) k_conv3(const TIn *__restrict__ in, int CK, const bf16 *__restrict__ W,
                                               const float *__restrict__ bias, void *__restrict__ out, int out_bf16,
                                               int relu, int lg, int V)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int n = 1 << lg, msk = n - 1;
    const int r0 = blockIdx.x * 64 + warp * 16 + g, r1 = r0 + 8;
    const bool ok0 = r0 < V, ok1 = r1 < V;
    const int x0 = r0 & msk, y0 = (r0 >> lg) & msk, z0 = (r0 >> (2 * lg)) & msk, b0 = r0 >> (3 * lg);
    const int x1 = r1 & msk, y1 = (r1 >> lg) & msk, z1 = (r1 >> (2 * lg)) & msk, b1 = r1 >> (3 * lg);
    float acc[NT][4];
#pragma unroll
    for (int q = 0; q < NT; q++)
        acc[q][0] = acc[q][1] = acc[q][2] = acc[q][3] = 0.f;
    constexpr int N = NT * 8;
    for (int tap = 0; tap < 27; tap++) {
        int dz = tap / 9 - 1, dy = (tap / 3) % 3 - 1, dx = tap % 3 - 1;
        if (FLIP) {
            dz = -dz;
            dy = -dy;
            dx = -dx;
        }
        int q0 = -1, q1 = -1;
        {
            const int zz = z0 + dz, yy = y0 + dy, xx = x0 + dx;
            if (ok0 && (unsigned)zz < (unsigned)n && (unsigned)yy < (unsigned)n && (unsigned)xx < (unsigned)n)
                q0 = (((b0 << lg | zz) << lg | yy) << lg) | xx;
        }
        {
            const int zz = z1 + dz, yy = y1 + dy, xx = x1 + dx;
            if (ok1 && (unsigned)zz < (unsigned)n && (unsigned)yy < (unsigned)n && (unsigned)xx < (unsigned)n)
                q1 = (((b1 << lg | zz) << lg | yy) << lg) | xx;
        }
        const bf16 *Wt = W + (size_t)tap * N * CK;
        for (int c0 = 0; c0 < CK; c0 += 16) {
            const uint32_t a0 = q0 >= 0 ? ld2(in + (size_t)q0 * CK + c0 + 2 * t) : 0u;
            const uint32_t a1 = q1 >= 0 ? ld2(in + (size_t)q1 * CK + c0 + 2 * t) : 0u;
            const uint32_t a2 = q0 >= 0 ? ld2(in + (size_t)q0 * CK + c0 + 2 * t + 8) : 0u;
            const uint32_t a3 = q1 >= 0 ? ld2(in + (size_t)q1 * CK + c0 + 2 * t + 8) : 0u;
#pragma unroll
            for (int q = 0; q < NT; q++) {
                const bf16 *wp = Wt + (size_t)(q * 8 + g) * CK + c0 + 2 * t;
                mma16816(acc[q], a0, a1, a2, a3, ld2(wp), ld2(wp + 8));
            }
        }
    }
#pragma unroll
    for (int q = 0; q < NT; q++) {
        const int c = q * 8 + 2 * t;
        float v[4] = {acc[q][0], acc[q][1], acc[q][2], acc[q][3]};
        if (bias) {
            v[0] += bias[c];
            v[1] += bias[c + 1];
            v[2] += bias[c];
            v[3] += bias[c + 1];
        }
        if (relu)
            for (int e = 0; e < 4; e++)
                v[e] = fmaxf(v[e], 0.f);
        if (out_bf16) {
            bf16 *o = reinterpret_cast<bf16 *>(out);
            if (ok0)
                *reinterpret_cast<uint32_t *>(o + (size_t)r0 * N + c) = pack2(v[0], v[1]);
            if (ok1)
                *reinterpret_cast<uint32_t *>(o + (size_t)r1 * N + c) = pack2(v[2], v[3]);
        } else {
            float *o = reinterpret_cast<float *>(out);
            if (ok0)
                *reinterpret_cast<float2 *>(o + (size_t)r0 * N + c) = make_float2(v[0], v[1]);
            if (ok1)
                *reinterpret_cast<float2 *>(o + (size_t)r1 * N + c) = make_float2(v[2], v[3]);
        }
    }
}

// ---------------------------------------------------------------------------
// 5th-generation tensor cores (tcgen05): the same implicit GEMM with the
// accumulator in tensor memory.  Inline PTX after the PTX ISA's tcgen05
// section: TMEM allocation by one warp, tcgen05.mma issued by one thread
// from shared-memory matrix descriptors, completion through tcgen05.commit
// on an mbarrier, tcgen05.ld for the epilogue.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void tc_alloc(uint32_t slot, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tc_relinquish()
{
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tc_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// generic-proxy stores to shared memory made visible to the tensor core's reads
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// D[tmem] (+)= A * B^T, kind::f16 (BF16 operands, FP32 accumulate)
__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n"
                 ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
                 : "memory");
}
// arrive once on the mbarrier when every tcgen05.mma this thread issued so far has completed
__device__ __forceinline__ void tc_commit(uint32_t mbar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar)
                 : "memory");
}
// 16 consecutive FP32 columns of this warp's 32 TMEM lanes (one lane per thread)
__device__ __forceinline__ void tc_ld16(uint32_t taddr, float *v)
{
    uint32_t r[16];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
                 "[%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                   "=r"(r[15])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; i++)
        v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void mbar_init1(uint32_t mbar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mbar) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ bool mbar_test(uint32_t mbar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}\n"
                 : "=r"(ok)
                 : "r"(mbar), "r"(parity)
                 : "memory");
    return ok != 0;
}
// wait for completion `parity` of the mbarrier; false when the clock budget ran out first
__device__ __forceinline__ bool mbar_wait_for(uint32_t mbar, uint32_t parity, long long budget)
{
    const long long t0 = clock64();
    while (!mbar_test(mbar, parity))
        if (clock64() - t0 > budget)
            return false;
    return true;
}

// Shared-memory matrix descriptor, no swizzle: start address, leading-dimension
// byte offset (between core matrices adjacent along K), stride-dimension byte
// offset (between 8-row groups along M or N), the fixed 0b001 at bits 46-48.
__device__ __forceinline__ uint64_t tc_sdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// Instruction descriptor of kind::f16: FP32 D, BF16 A and B, both K-major,
// N >> 3 at bits 17-22, M >> 4 at bits 24-28.
__host__ __device__ constexpr uint32_t tc_idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// Operand tiles in shared memory, K-major without swizzle: K in slabs of 16
// (one MMA each); within a slab, core matrices of 8 rows x 8 BF16 (128
// contiguous bytes, rows 16 B apart), the two core matrices of a row group
// 128 B apart (LBO), row groups 256 B apart (SBO).  Byte offset of the
// 16-byte chunk holding elements k8*8..k8*8+7 of row m in a tile of `rows`
// rows:
__device__ __forceinline__ uint32_t tc_chunk(int rows, int m, int k8)
{
    return (uint32_t)((k8 >> 1) * rows * 32 + (m >> 3) * 256 + (k8 & 1) * 128 + (m & 7) * 16);
}

// 16-byte asynchronous copy global -> shared through L1, zero-filled when
// `valid` is false (a padding voxel); groups committed and waited on per tap
__device__ __forceinline__ void cp16(uint32_t dst, const void *src, bool valid)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int K> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(K) : "memory"); }

constexpr long long kTcBudget = 1ll << 31;   // clock cycles an mbarrier wait may take (about 1 s)
constexpr int kTcStages = 4;                  // taps in flight

// 3x3x3 convolution on tcgen05: a block of 128 threads computes 128 voxels
// (thread m gathers voxel m's rows and owns its outputs) x N output channels.
// Taps run through kTcStages shared-memory stages: the 128 gathered input
// rows (CK channels, zero rows at the padding) and the tap's N x CK weights
// arrive by cp.async kTcStages - 2 taps ahead; once a tap's copies have
// landed, thread 0 issues CK/16 MMAs into the TMEM accumulator and commits
// them to the stage's mbarrier, which the stage's next fill (two taps later)
// waits on.
// Epilogue: each warp reads its 32 TMEM lanes, adds the bias, applies relu,
// stores.  FLIP and the operand layouts as in k_conv3 (BF16 input).  A wait
// that outlasts kTcBudget sets *err and stops issuing; the block still waits
// (bounded) for what it issued and frees its TMEM.
template <int N, bool FLIP>
__global__ void __launch_bounds__(128) k_conv3_tc(const bf16 *__restrict__ in, int CK, const bf16 *__restrict__ W,
                                                  const float *__restrict__ bias, void *__restrict__ out,
                                                  int out_bf16, int relu, int lg, int V, int *__restrict__ err)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t mbar[kTcStages];
    __shared__ uint32_t tslot;
    constexpr int NCOL = N < 32 ? 32 : N;
    constexpr uint32_t IDESC = tc_idesc_bf16(128, N);
    const int tid = threadIdx.x, warp = tid >> 5;
    const int abytes = 128 * CK * 2, bbytes = N * CK * 2, sbytes = abytes + bbytes;
    const uint32_t sm0 = smem_u32(smem), mb0 = smem_u32(&mbar[0]);   // stage s: tiles at sm0 + s sbytes, mbarrier mb0 + 8 s
    if (warp == 0) {
        tc_alloc(smem_u32(&tslot), NCOL);
        tc_relinquish();
    }
    if (tid == 0) {
        for (int q = 0; q < kTcStages; q++)
            mbar_init1(mb0 + 8 * q);
        fence_mbar_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tslot;
    const int n = 1 << lg, msk = n - 1;
    const int r = blockIdx.x * 128 + tid;
    const bool ok = r < V;
    const int x = r & msk, y = (r >> lg) & msk, z = (r >> (2 * lg)) & msk, b = r >> (3 * lg);
    const int nk8 = CK >> 3;
    // the copies of one tap into stage s
    auto fill = [&](int tap, int s) {
        int dz = tap / 9 - 1, dy = (tap / 3) % 3 - 1, dx = tap % 3 - 1;
        if (FLIP) {
            dz = -dz;
            dy = -dy;
            dx = -dx;
        }
        const int zz = z + dz, yy = y + dy, xx = x + dx;
        const bool inside = ok && (unsigned)zz < (unsigned)n && (unsigned)yy < (unsigned)n && (unsigned)xx < (unsigned)n;
        const bf16 *src = inside ? in + (size_t)((((b << lg | zz) << lg | yy) << lg) | xx) * CK : in;
        const uint32_t As = sm0 + s * sbytes, Bs = As + abytes;
        for (int k8 = 0; k8 < nk8; k8++)
            cp16(As + tc_chunk(128, tid, k8), src + k8 * 8, inside);
        const bf16 *Wt = W + (size_t)tap * N * CK;
        for (int e = tid; e < N * nk8; e += 128) {
            const int row = e / nk8, k8 = e - row * nk8;
            cp16(Bs + tc_chunk(N, row, k8), Wt + (size_t)row * CK + k8 * 8, true);
        }
    };
    for (int t = 0; t < kTcStages - 2; t++) {
        fill(t, t);
        cp_commit();
    }
    uint32_t phases = 0u;    // bit s: parity of stage s's next completion
    int issued = 0;          // taps whose MMAs were issued (uniform)
    bool bad = false;
    for (int tap = 0; tap < 27; tap++) {
        const int s = tap % kTcStages;
        // refill the stage of tap - 2 with tap + kTcStages - 2, once tap - 2's MMAs are done with it
        // (a tap's MMAs get one tap of slack; the copies of two taps stay in flight)
        const int tn = tap + kTcStages - 2;
        if (tn < 27) {
            const int sn = tn % kTcStages;
            if (tap >= 2) {
                const bool done = mbar_wait_for(mb0 + 8 * sn, (phases >> sn) & 1u, kTcBudget);
                if (__syncthreads_or(!done)) {   // the final wait covers tap - 2 and what followed it
                    bad = true;
                    break;
                }
                phases ^= 1u << sn;
            }
            fill(tn, sn);
        }
        cp_commit();                 // (an empty group past the last tap keeps the count)
        cp_wait<kTcStages - 2>();    // this thread's copies of `tap` have landed
        fence_async_smem();
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (tid == 0) {
            const uint32_t a0 = sm0 + s * sbytes, b0 = a0 + abytes;
            for (int k = 0; k < CK / 16; k++)
                tc_mma(tmem, tc_sdesc(a0 + k * 128 * 32, 128, 256), tc_sdesc(b0 + k * N * 32, 128, 256), IDESC,
                       (tap > 0 || k > 0) ? 1u : 0u);
            tc_commit(mb0 + 8 * s);
        }
        issued = tap + 1;
    }
    cp_wait<0>();
    // the last commit covers every MMA issued before it
    bool done = true;
    if (issued > 0) {
        const int s = (issued - 1) % kTcStages;
        done = mbar_wait_for(mb0 + 8 * s, (phases >> s) & 1u, kTcBudget);
    }
    done = !__syncthreads_or(!done);
    tc_fence_after();
    if (done && !bad) {
        const uint32_t lane_base = tmem + ((uint32_t)(warp * 32) << 16);
        for (int c0 = 0; c0 < N; c0 += 16) {
            float v[16];
            tc_ld16(lane_base + c0, v);
            if (bias)
#pragma unroll
                for (int i = 0; i < 16; i++)
                    v[i] += bias[c0 + i];
            if (relu)
#pragma unroll
                for (int i = 0; i < 16; i++)
                    v[i] = fmaxf(v[i], 0.f);
            if (!ok)
                continue;
            if (out_bf16) {
                uint4 *o = reinterpret_cast<uint4 *>(reinterpret_cast<bf16 *>(out) + (size_t)r * N + c0);
                o[0] = make_uint4(pack2(v[0], v[1]), pack2(v[2], v[3]), pack2(v[4], v[5]), pack2(v[6], v[7]));
                o[1] = make_uint4(pack2(v[8], v[9]), pack2(v[10], v[11]), pack2(v[12], v[13]), pack2(v[14], v[15]));
            } else {
                float4 *o = reinterpret_cast<float4 *>(reinterpret_cast<float *>(out) + (size_t)r * N + c0);
#pragma unroll
                for (int i = 0; i < 4; i++)
                    o[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0)
        tc_dealloc(tmem, NCOL);
    if ((bad || !done) && tid == 0)
        atomicExch(err, 1);
}

// Weight gradients of a 3x3x3 convolution on tcgen05 (bias gradient apart):
//   dW[tap][ci][co] += sum_v in[v + off(tap)][ci] * bf16(d[v][co])
// as D = A B^T with the voxels as K: a block takes TG = 128 / CK taps (rows
// m = tap_local * CK + ci; rows of taps past 26 stay zero) and a run of
// `vchunk` voxels, gathers 64 voxels per stage -- A[m][k] from the voxels'
// shifted input rows, B[co][k] from their output gradients rounded to BF16,
// both transposed into the K-major tiles of k_conv3_tc -- issues 4 MMAs per
// stage into its TMEM accumulator (two stages, a stage refilled once its
// MMAs of two stages back have completed), and adds its 128 x N partial sums
// into dW (FP32 atomics, real channels only).  Waits bounded as in
// k_conv3_tc.
template <int CK, int N>
__global__ void __launch_bounds__(128) k_wgrad_tc(const bf16 *__restrict__ in, int Cin, const float *__restrict__ d,
                                                  float *__restrict__ dW, int lg, int V, int vchunk,
                                                  int *__restrict__ err)
{
    constexpr int TG = 128 / CK, KB = 64, NS = 2;
    constexpr int NCOL = N < 32 ? 32 : N;
    constexpr uint32_t IDESC = tc_idesc_bf16(128, N);
    constexpr int ABYTES = 128 * KB * 2, BBYTES = N * KB * 2, SBYTES = ABYTES + BBYTES;
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t mbar[NS];
    __shared__ uint32_t tslot;
    const int tid = threadIdx.x, warp = tid >> 5;
    const uint32_t sm0 = smem_u32(smem), mb0 = smem_u32(&mbar[0]);
    if (warp == 0) {
        tc_alloc(smem_u32(&tslot), NCOL);
        tc_relinquish();
    }
    if (tid == 0) {
        for (int q = 0; q < NS; q++)
            mbar_init1(mb0 + 8 * q);
        fence_mbar_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tslot;
    const int n = 1 << lg, msk = n - 1;
    const int tap0 = blockIdx.y * TG;
    const int v0 = blockIdx.x * vchunk, v1 = min(v0 + vchunk, V);
    const int nst = (v1 - v0 + KB - 1) / KB;
    // rows of the tap `tap` shifted from voxel v, or NULL (padding, past the run, or no such tap)
    auto row_of = [&](int v, int tap) -> const bf16 * {
        if (v >= v1 || tap >= 27)
            return nullptr;
        const int x = v & msk, y = (v >> lg) & msk, z = (v >> (2 * lg)) & msk, b = v >> (3 * lg);
        const int zz = z + tap / 9 - 1, yy = y + (tap / 3) % 3 - 1, xx = x + tap % 3 - 1;
        if ((unsigned)zz >= (unsigned)n || (unsigned)yy >= (unsigned)n || (unsigned)xx >= (unsigned)n)
            return nullptr;
        return in + (size_t)((((b << lg | zz) << lg | yy) << lg) | xx) * CK;
    };
    auto fill = [&](int j, int s) {
        unsigned char *As = smem + s * SBYTES, *Bs = As + ABYTES;
        const int vb = v0 + j * KB;
        // A: (voxel pair p, tap_local) items; a pair of voxels k = 2p, 2p + 1 makes one 32-bit word per row
        for (int it = tid; it < (KB / 2) * TG; it += 128) {
            const int p = it % (KB / 2), tl = it / (KB / 2), k = 2 * p;
            const bf16 *ra = row_of(vb + k, tap0 + tl), *rb = row_of(vb + k + 1, tap0 + tl);
#pragma unroll 2
            for (int k8 = 0; k8 < CK / 8; k8++) {
                const uint4 qa = ra ? *reinterpret_cast<const uint4 *>(ra + 8 * k8) : make_uint4(0u, 0u, 0u, 0u);
                const uint4 qb = rb ? *reinterpret_cast<const uint4 *>(rb + 8 * k8) : make_uint4(0u, 0u, 0u, 0u);
                const uint32_t wa[4] = {qa.x, qa.y, qa.z, qa.w}, wb[4] = {qb.x, qb.y, qb.z, qb.w};
#pragma unroll
                for (int e = 0; e < 8; e++) {
                    const uint32_t lo = (wa[e >> 1] >> (16 * (e & 1))) & 0xFFFFu;
                    const uint32_t hi = (wb[e >> 1] >> (16 * (e & 1))) & 0xFFFFu;
                    const int m = tl * CK + 8 * k8 + e;
                    *reinterpret_cast<uint32_t *>(As + tc_chunk(128, m, k >> 3) + (k & 7) * 2) = lo | (hi << 16);
                }
            }
        }
        // B: (voxel pair p, 4 output channels) items from the FP32 gradient rows
        for (int it = tid; it < (KB / 2) * (N / 4); it += 128) {
            const int p = it % (KB / 2), c4 = it / (KB / 2), k = 2 * p;
            const int va = vb + k, vbb = vb + k + 1;
            const float4 ga = va < v1 ? *reinterpret_cast<const float4 *>(d + (size_t)va * N + 4 * c4)
                                      : make_float4(0.f, 0.f, 0.f, 0.f);
            const float4 gb = vbb < v1 ? *reinterpret_cast<const float4 *>(d + (size_t)vbb * N + 4 * c4)
                                       : make_float4(0.f, 0.f, 0.f, 0.f);
            const float fa[4] = {ga.x, ga.y, ga.z, ga.w}, fb[4] = {gb.x, gb.y, gb.z, gb.w};
#pragma unroll
            for (int e = 0; e < 4; e++)
                *reinterpret_cast<uint32_t *>(Bs + tc_chunk(N, 4 * c4 + e, k >> 3) + (k & 7) * 2) = pack2(fa[e], fb[e]);
        }
    };
    uint32_t phases = 0u;
    int issued = 0;
    bool bad = false;
    for (int j = 0; j < nst; j++) {
        const int s = j % NS;
        if (j >= NS) {       // the stage's MMAs of stage j - 2 have finished reading it
            const bool done = mbar_wait_for(mb0 + 8 * s, (phases >> s) & 1u, kTcBudget);
            if (__syncthreads_or(!done)) {
                bad = true;
                break;
            }
            phases ^= 1u << s;
        }
        fill(j, s);
        fence_async_smem();
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (tid == 0) {
            const uint32_t a0 = sm0 + s * SBYTES, b0 = a0 + ABYTES;
            for (int k = 0; k < KB / 16; k++)
                tc_mma(tmem, tc_sdesc(a0 + k * 128 * 32, 128, 256), tc_sdesc(b0 + k * N * 32, 128, 256), IDESC,
                       (j > 0 || k > 0) ? 1u : 0u);
            tc_commit(mb0 + 8 * s);
        }
        issued = j + 1;
    }
    bool done = true;
    if (issued > 0) {
        const int s = (issued - 1) % NS;
        done = mbar_wait_for(mb0 + 8 * s, (phases >> s) & 1u, kTcBudget);
    }
    done = !__syncthreads_or(!done);
    tc_fence_after();
    if (done && !bad && issued > 0) {
        const int tl = tid / CK, ci = tid - tl * CK, tap = tap0 + tl;
        const bool mine = tap < 27 && ci < Cin;
        const uint32_t lane_base = tmem + ((uint32_t)(warp * 32) << 16);
        for (int c0 = 0; c0 < N; c0 += 16) {
            float v[16];
            tc_ld16(lane_base + c0, v);
            if (mine)
#pragma unroll
                for (int i = 0; i < 16; i++)
                    atomicAdd(&dW[((size_t)tap * Cin + ci) * N + c0 + i], v[i]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0)
        tc_dealloc(tmem, NCOL);
    if ((bad || !done) && tid == 0)
        atomicExch(err, 1);
}

// The same gradients on grids of at least 8^3 voxels, without a transposition:
// with the voxels as K, both operands lie in memory with M and N fastest, so
// they go to shared memory as they are (16-byte rows of 8 channels) and the
// MMAs read them M- and N-major.  A stage holds 8 grid rows (y0 .. y0 + 7 of
// one plane z, all x) of the output gradient and the rows y0 - 1 .. of plane
// z + dz of the input, per row one line of voxels per 8 channels.  A start
// address 16 bytes on is a shift by one voxel (dx), and the lines of
// consecutive rows are evenly spaced, so one MMA takes the input rows of all
// three dy (M = row, channel; 128 / CK rows, what is past the third ignored)
// over 16 voxels of x (two rows on the 8^3 grid).  A block keeps the ndx
// shifts of one dz in TMEM over its stages, two in flight, and adds its sums
// into dW with 16-byte reductions.  With NZ = 3 (planes of at least
// kWgradChain voxels) a stage holds 4 rows of an input plane and of the gradient planes z
// - dz of all three dz, side by side in N, which an MMA takes in the time of
// one: a third of the MMAs.
// The tensor core rounds each sum in its FP32 accumulators towards zero, an
// error that grows with the number of MMAs that an accumulator takes.  A block
// takes kWgradChain voxels in memory order, the products of k_wgrad_tc's
// accumulators in the same order: the sums are equal bit for bit up to the
// order of the reductions into dW.  Two or four gradient rows in N would need
// as many times fewer MMAs, but other sums (up to 3e-5 relative off).
// The gather by tap (k_wgrad_tc) spent its time in the transposing stores,
// eight-way bank conflicts among them, once per tap.
// Training step of 4 samples of 64^3: 5538 us with the gather, 1998 us with
// NZ = 1 everywhere, 1679 us with NZ = 3 at 64^3 (1416 us with two or four
// gradient rows in N).  What bounds it is the MMAs, 32 cycles each for the 4
// KB of A that they read.
// Grids of less than 8^3 voxels and layers whose stages do not fit stay with
// k_wgrad_tc.
constexpr int kWgradChain = 4096;   // voxels per accumulator

template <int CK, int N, int NZ>
struct WgradTile {
    static constexpr int kRA = 128 / CK;              // input rows of one MMA
    static constexpr int kMA = (3 + kRA - 1) / kRA;   // MMAs for the three dy
    static constexpr int kTY = NZ == 3 ? 4 : 8;
    static constexpr int kRows = kTY - 1 + kRA * kMA; // input rows an MMA may read
    static constexpr int kCols = 3 * kMA * NZ * N;
    static constexpr int kAlloc = kCols <= 64 ? 64 : kCols <= 128 ? 128 : kCols <= 256 ? 256 : 512;
    // voxels per line: x = -1 .. n and one more (odd: lines of different channels in different banks)
    __host__ __device__ static int pa(int n) { return n + 3; }
    __host__ __device__ static int pb(int n) { return n + 1; }
    __host__ __device__ static int a_bytes(int n) { return kRows * (CK / 8) * pa(n) * 16; }
    __host__ __device__ static int stage(int n) { return a_bytes(n) + kTY * NZ * (N / 8) * pb(n) * 16; }
    static constexpr int kSmemMax = 226 * 1024;
    static bool applies(int lg)
    {
        return kCols <= 512 && lg >= 3 && (NZ == 1 || 1 << 2 * lg >= kWgradChain) && kTY << lg <= kWgradChain &&
               2 * stage(1 << lg) <= kSmemMax;
    }
};

__device__ __forceinline__ void red_add4(float *p, const float *v)
{
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3])
                 : "memory");
}

template <int CK, int N, int NZ>
__global__ void __launch_bounds__(256) k_wgrad_rows(const bf16 *__restrict__ in, int Cin, const bf16 *__restrict__ d,
                                                    float *__restrict__ dW, int lg, int B, int ndx, int *__restrict__ err)
{
    typedef WgradTile<CK, N, NZ> W;
    constexpr int CG = CK / 8, NG = N / 8, TY = W::kTY, LTY = TY == 4 ? 2 : 3;
    // BF16 operands, both M- / N-major
    constexpr uint32_t IDESC = tc_idesc_bf16(128, NZ * N) | (1u << 15) | (1u << 16);
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t mbar[2];
    __shared__ uint32_t tslot;
    const int tid = threadIdx.x, warp = tid >> 5;
    const uint32_t sm0 = smem_u32(smem), mb0 = smem_u32(&mbar[0]);
    if (warp == 0) {
        tc_alloc(smem_u32(&tslot), W::kAlloc);
        tc_relinquish();
    }
    if (tid == 0) {
        mbar_init1(mb0);
        mbar_init1(mb0 + 8);
        fence_mbar_init();
    }
    const int n = 1 << lg, PA = W::pa(n), PB = W::pb(n), sbytes = W::stage(n), abytes = W::a_bytes(n);
    // the padding voxels x = -1 and x = n of every line stay zero
    for (int e = tid; e < 2 * W::kRows * CG * 2; e += 256) {
        const int line = (e >> 1) % (W::kRows * CG), st = (e >> 1) / (W::kRows * CG);
        *reinterpret_cast<uint4 *>(smem + st * sbytes + (line * PA + (e & 1 ? n + 1 : 0)) * 16) = make_uint4(0, 0, 0, 0);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tslot;
    // blockIdx.y: dz (NZ = 1) and the first dx (ndx = 3: all of them; else ndx = 1)
    const int dz = NZ == 3 ? 0 : (int)blockIdx.y % 3 - 1, dx0 = NZ == 3 ? (int)blockIdx.y : (int)blockIdx.y / 3;
    const int lgt = lg - LTY, chain = kWgradChain >> (lg + LTY);
    const int it0 = blockIdx.x * chain, nitem = min(it0 + chain, B << (lg + lgt));   // items: (sample, z, TY rows)
    auto next_item = [&](int it) {
        for (; it < nitem; it++) {
            const int z = ((it >> lgt) & (n - 1)) + dz;
            if ((unsigned)z < (unsigned)n)
                break;
        }
        return it;
    };
    auto fill = [&](int it, int st) {
        const int y0 = (it & ((1 << lgt) - 1)) * TY, z = (it >> lgt) & (n - 1), b = it >> (lgt + lg);
        const uint32_t As = sm0 + st * sbytes, Bs = As + abytes;
        const bf16 *pa = in + ((size_t)(((b << lg) + z + dz) << lg) << lg) * CK;
        for (int e = tid; e < (TY + 2) * n * CG; e += 256) {
            const int cg = e & (CG - 1), x = (e / CG) & (n - 1), row = (e / CG) >> lg, y = y0 - 1 + row;
            const bool ok = (unsigned)y < (unsigned)n;
            cp16(As + ((row * CG + cg) * PA + x + 1) * 16, ok ? pa + ((size_t)(y << lg) + x) * CK + 8 * cg : pa, ok);
        }
#pragma unroll
        for (int q = 0; q < NZ; q++) {   // gradient planes z - dz (NZ = 3: dz = q - 1)
            const int zg = NZ == 3 ? z - q + 1 : z;
            const bool ok = (unsigned)zg < (unsigned)n;
            const bf16 *pd = ok ? d + ((size_t)((((b << lg) + zg) << lg) + y0) << lg) * N : d;
            for (int e = tid; e < TY * n * NG; e += 256) {
                const int ng = e & (NG - 1), x = (e / NG) & (n - 1), row = (e / NG) >> lg;
                cp16(Bs + (((row * NZ + q) * NG + ng) * PB + x) * 16,
                     ok ? pd + ((size_t)(row << lg) + x) * N + 8 * ng : d, ok);
            }
        }
    };
    const uint32_t lboA = n == 8 ? CG * PA * 16 : 128, lboB = n == 8 ? NG * PB * 16 : 128;
    const int ystep = n == 8 ? 2 : 1;
    int it = next_item(it0), issued = 0;
    uint32_t phases = 0u;
    bool bad = false;
    if (it < nitem)
        fill(it, 0);
    cp_commit();
    while (it < nitem) {
        const int nx = next_item(it + 1), s = issued & 1;
        if (nx < nitem) {
            if (issued > 0) {   // the other stage's MMAs have finished reading it
                const bool done = mbar_wait_for(mb0 + 8 * (s ^ 1), (phases >> (s ^ 1)) & 1u, kTcBudget);
                if (__syncthreads_or(!done)) {
                    bad = true;
                    break;
                }
                phases ^= 1u << (s ^ 1);
            }
            fill(nx, s ^ 1);
        }
        cp_commit();
        cp_wait<1>();
        fence_async_smem();
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (tid == 0) {
            const uint64_t da0 = tc_sdesc(sm0 + s * sbytes, lboA, PA * 16);
            const uint64_t db0 = tc_sdesc(sm0 + s * sbytes + abytes, lboB, PB * 16);
            const uint32_t lines = W::kRA * CG * PA;
            bool first = issued == 0;
            for (int yb = 0; yb < TY; yb += ystep) {
                uint64_t da = da0 + yb * CG * PA + dx0, db = db0 + yb * NZ * NG * PB;
                for (int x0 = 0; x0 < n; x0 += 16, da += 16, db += 16) {
#pragma unroll
                    for (int dx = 0; dx < 3; dx++)
                        if (dx < ndx)
#pragma unroll
                            for (int ma = 0; ma < W::kMA; ma++)
                                tc_mma(tmem + (dx * W::kMA + ma) * NZ * N, da + dx + ma * lines, db, IDESC,
                                       first ? 0u : 1u);
                    first = false;
                }
            }
            tc_commit(mb0 + 8 * s);
        }
        issued++;
        it = nx;
    }
    cp_wait<0>();
    bool done = true;
    if (issued > 0) {
        const int s = (issued - 1) & 1;   // the last commit covers every MMA issued before it
        done = mbar_wait_for(mb0 + 8 * s, (phases >> s) & 1u, kTcBudget);
    }
    done = !__syncthreads_or(!done);
    tc_fence_after();
    if (done && !bad && issued > 0) {
        const int m = (warp & 3) * 32 + (tid & 31), ci = m & (CK - 1);
        const uint32_t lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        for (int q = warp >> 2; q < ndx * W::kMA * NZ; q += 2) {   // column blocks (dx, group of dy, dz)
            const int ma = q / NZ % W::kMA, dx = dx0 + q / (NZ * W::kMA), dy = ma * W::kRA + m / CK;
            const int tz = NZ == 3 ? q % NZ : dz + 1;
            float *o = dW + ((size_t)(tz * 9 + dy * 3 + dx) * Cin + ci) * N;
            for (int c0 = 0; c0 < N; c0 += 16) {
                float v[16];
                tc_ld16(lane_base + q * N + c0, v);
                if (dy < 3 && ci < Cin)
#pragma unroll
                    for (int i = 0; i < 16; i += 4)
                        red_add4(o + c0 + i, v + i);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0)
        tc_dealloc(tmem, W::kAlloc);
    if ((bad || !done) && tid == 0)
        atomicExch(err, 1);
}

// What the weight and data gradients of a convolution read, in one pass over
// its output gradient d (N channels, V voxels): d where the activation is
// positive, else 0, as BF16 (out) and, for grids of less than 8^3 voxels, in
// FP32 in place; db[c] += its sums.  A thread keeps one group of 8 channels.
// Bound by memory; as three kernels (mask, sums, rounding) the gradient of 4 x
// 64^3 x 16 took 77 us, here 22 us.
__global__ void __launch_bounds__(256) k_grad_prep(float *__restrict__ d, const bf16 *__restrict__ act, int N, long n8,
                                                   bf16 *__restrict__ out, float *__restrict__ db, int keep)
{
    __shared__ float part[256][9];
    const int ng = N >> 3;
    float s[8];
#pragma unroll
    for (int i = 0; i < 8; i++)
        s[i] = 0.f;
    // the number of threads is a multiple of the channel groups
    for (long e = blockIdx.x * 256l + threadIdx.x; e < n8; e += gridDim.x * 256l) {
        float4 *p = reinterpret_cast<float4 *>(d) + 2 * e;
        const float4 a = p[0], c = p[1];
        const uint4 w = reinterpret_cast<const uint4 *>(act)[e];
        float v[8] = {a.x, a.y, a.z, a.w, c.x, c.y, c.z, c.w};
        float x[8];
        unpack8(w, x);
#pragma unroll
        for (int i = 0; i < 8; i++) {
            if (!(x[i] > 0.f))
                v[i] = 0.f;
            s[i] += v[i];
        }
        reinterpret_cast<uint4 *>(out)[e] =
            make_uint4(pack2(v[0], v[1]), pack2(v[2], v[3]), pack2(v[4], v[5]), pack2(v[6], v[7]));
        if (keep) {
            p[0] = make_float4(v[0], v[1], v[2], v[3]);
            p[1] = make_float4(v[4], v[5], v[6], v[7]);
        }
    }
#pragma unroll
    for (int i = 0; i < 8; i++)
        part[threadIdx.x][i] = s[i];
    __syncthreads();
    if (threadIdx.x < N) {
        float t = 0.f;
        for (int k = threadIdx.x >> 3; k < 256; k += ng)
            t += part[k][threadIdx.x & 7];
        atomicAdd(&db[threadIdx.x], t);
    }
}

// ---------------------------------------------------------------------------
// The same convolution from a halo in shared memory: a tile of 8 (x) x 16 (y)
// voxels of one plane of one sample with the 10 x 18 x 3 voxels around it (zero
// outside the grid), per 8 input channels a chunk of 16-byte rows, x fastest.
// Tap (dz, dy, dx) is then the 128 x CK operand whose row (x, y) is halo row
// ((dz+1) 18 + y + dy + 1) 10 + x + dx + 1: a descriptor at that start with
// 8-row groups one halo row (160 B) apart (SBO) and the channel chunks one
// chunk apart (LBO) -- no copy per tap.  One thread issues every MMA.
// k_conv3_halo takes up to four planes per block and copies halo and weights by
// cp.async; k_conv3_halo_p, the persistent form, loads its halos with one TMA
// box per 8 channels.
// ---------------------------------------------------------------------------
constexpr int kHaloRows = 10 * 18 * 3;                 // 540 rows of one channel chunk
constexpr int kHaloChunk = (kHaloRows * 16 + 127) / 128 * 128;   // 8704 B, 128-byte aligned chunks

__device__ __forceinline__ void mbar_expect_tx(uint32_t mbar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void tma_load5(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, int c3, int c4,
                                          uint32_t mbar)
{
    asm volatile("cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, "
                 "%3, %4, %5, %6}], [%7];" ::"r"(dst),
                 "l"((unsigned long long)map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(mbar)
                 : "memory");
}
// This kernel: tz planes per block (tz accumulators), the halo by cp.async.  A
// warp copies a line of 10 voxels, 16 bytes per lane, channels fastest, so the
// reads are whole sectors; the channel chunks in shared memory start in
// different banks (halo_chunk, and N + 1 rows per weight chunk).  What bounded
// the one-plane form with one TMA box per chunk was the thread that issues the
// MMAs, which built two descriptors from run-time sizes for each (100 cycles an
// MMA; with constant steps 55 to 65, near the 32 its 4 KB of A take), then
// loading three planes and all weights for one.  4 x 64^3, 16 -> 16 channels 63
// -> 43 us, 32 -> 16 145 -> 98 us, data gradient 32 <- 16 122 -> 74 us.
// Layers whose weights do not fit beside the halo stream them, three taps a
// stage; per tap, the gather of k_conv3_tc took an L1 line per lane: 4 x 16^3,
// 128 -> 32 channels 54 -> 19 us, 4 x 8^3, 64 -> 64 36 -> 16 us.
// Every accumulator takes its products in the same order in all these forms.
__host__ __device__ constexpr int halo_chunk(int tz) { return (180 * (tz + 2) + 1) * 16; }
// all 27 taps' weights stay beside the halo, else they stream through it three taps at a time
__host__ __device__ constexpr bool halo_resident(int CK, int N) { return 27 * N * CK * 2 <= 64 * 1024 && CK <= 64; }

template <int N, bool FLIP, int CK>
__global__ void __launch_bounds__(256) k_conv3_halo(const bf16 *__restrict__ in, const bf16 *__restrict__ W,
                                                    const float *__restrict__ bias, void *__restrict__ out,
                                                    int out_bf16, int relu, int lg, int tz, int ncol, int fault,
                                                    int *__restrict__ err)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t mbar[4];   // accumulator of a plane complete; streamed weights: a stage read
    __shared__ uint32_t tslot;
    constexpr uint32_t IDESC = tc_idesc_bf16(128, N);
    constexpr bool kStream = !halo_resident(CK, N);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr int nk8 = CK / 8;
    const int chunk = halo_chunk(tz);
    const uint32_t halo = smem_u32(smem), wts = halo + nk8 * chunk;
    const uint32_t mb0 = smem_u32(&mbar[0]);
    const int n = 1 << lg;
    const int tx = n >> 3, ty = (n + 15) >> 4;          // tiles per row and per column of a plane
    int t = blockIdx.x;
    const int x0 = (t % tx) * 8;
    t /= tx;
    const int y0 = (t % ty) * 16;
    t /= ty;
    const int z0 = (t % (n / tz)) * tz, b = t / (n / tz);
    if (warp == 0) {
        tc_alloc(smem_u32(&tslot), ncol);
        tc_relinquish();
    }
    if (tid == 0) {
        for (int q = 0; q < 4; q++)
            mbar_init1(mb0 + 8 * q);
        fence_mbar_init();
    }
    // the halo, zero outside the grid
    for (int line = warp; line < 18 * (tz + 2); line += 8) {
        const int hz = line / 18, hy = line - hz * 18, gz = z0 - 1 + hz, gy = y0 - 1 + hy;
        const bool inside = (unsigned)gy < (unsigned)n && (unsigned)gz < (unsigned)n;
        const bf16 *src = in + (((((size_t)b << lg) + gz) << lg) + gy << lg) * CK;
        for (int c = lane; c < 10 * nk8; c += 32) {
            const int hx = c / nk8, k8 = c % nk8, gx = x0 - 1 + hx;
            const bool ok = inside && (unsigned)gx < (unsigned)n;
            cp16(halo + k8 * chunk + (line * 10 + hx) * 16, ok ? src + (size_t)gx * CK + 8 * k8 : in, ok);
        }
    }
    // the weights of taps t0 .. t0 + nt - 1, N rows of 16 B per (tap, chunk)
    auto weights = [&](int t0, int nt, uint32_t dst) {
        for (int e = tid; e < nt * N * nk8; e += 256) {
            const int k8 = e % nk8, row = e / nk8;   // row = tap * N + output channel
            const int tap = row / N, nn = row - tap * N;
            cp16(dst + ((tap * nk8 + k8) * (N + 1) + nn) * 16, W + ((size_t)t0 * N + row) * CK + 8 * k8, true);
        }
    };
    // the MMAs of a tap: one thread issues them; with the descriptors' steps as
    // constants an MMA costs it few instructions
    auto tap_mmas = [&](int tap, uint32_t d, uint64_t da, uint64_t db) {
        const int p = FLIP ? 26 - tap : tap;   // position of the tap in the 3 x 3 x 3 box
        const int off = ((p / 9) * 18 + (p / 3) % 3) * 10 + p % 3;
#pragma unroll
        for (int k = 0; k < CK / 16; k++)
            tc_mma(d, da + off + k * (2 * chunk / 16), db + 2 * k * (N + 1), IDESC, (tap > 0 || k > 0) ? 1u : 0u);
    };
    // fault (test of the timeout path): no MMA is issued, the waits for them run out
    const long long budget = fault ? (1ll << 21) : kTcBudget;
    bool bad = false;
    if constexpr (kStream) {
        // three taps a stage, three stages in a ring; one plane
        constexpr int SB = 3 * nk8 * (N + 1) * 16;
        weights(0, 3, wts);
        cp_commit();
        weights(3, 3, wts + SB);
        cp_commit();
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        const uint32_t tmem = tslot;
        for (int st = 0; st < 9; st++) {
            cp_wait<1>();
            fence_async_smem();
            tc_fence_before();
            __syncthreads();
            tc_fence_after();
            if (tid == 0 && !fault) {
                const uint64_t da = tc_sdesc(halo, chunk, 160), db = tc_sdesc(wts + (st % 3) * SB, (N + 1) * 16, 128);
                for (int q = 0; q < 3; q++)
                    tap_mmas(3 * st + q, tmem, da, db + q * nk8 * (N + 1));
                tc_commit(mb0 + 8 * (st % 3));
                if (st == 8)
                    tc_commit(mb0 + 24);
            }
            if (st + 2 < 9) {
                if (st > 0) {   // the MMAs of stage st - 1 have read the ring's third stage
                    const bool done = mbar_wait_for(mb0 + 8 * ((st - 1) % 3), ((st - 1) / 3) & 1, budget);
                    if (__syncthreads_or(!done)) {
                        bad = true;
                        break;
                    }
                }
                weights(3 * (st + 2), 3, wts + ((st + 2) % 3) * SB);
            }
            cp_commit();
        }
        cp_wait<0>();
    } else {
        weights(0, 27, wts);
        cp_commit();
        cp_wait<0>();
        fence_async_smem();
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (tid == 0 && !fault)
            for (int zi = 0; zi < tz; zi++) {
                const uint64_t da = tc_sdesc(halo + zi * 180 * 16, chunk, 160), db = tc_sdesc(wts, (N + 1) * 16, 128);
#pragma unroll
                for (int tap = 0; tap < 27; tap++)
                    tap_mmas(tap, tslot + zi * N, da, db + tap * nk8 * (N + 1));
                tc_commit(mb0 + 8 * zi);
            }
    }
    const uint32_t tmem = tslot;
    const auto acc_bar = [&](int zi) { return mb0 + 8 * (kStream ? 3 : zi); };
    // four warps cover an accumulator's 128 rows: planes alternate between the two halves of the block
    for (int zi = warp >> 2; zi < tz && !bad; zi += 2) {
        bad = !mbar_wait_for(acc_bar(zi), 0, budget);
        bad = __any_sync(0xffffffffu, bad);
        if (bad)
            break;
        tc_fence_after();
        const int row = (warp & 3) * 32 + lane, x = x0 + (row & 7), y = y0 + (row >> 3);
        const bool mine = y < n;
        const size_t r = ((((size_t)b * n + z0 + zi) * n + y) * n + x);
        const uint32_t lane_base = tmem + zi * N + ((uint32_t)((warp & 3) * 32) << 16);
        for (int c0 = 0; c0 < N; c0 += 16) {
            float v[16];
            tc_ld16(lane_base + c0, v);
            if (bias)
#pragma unroll
                for (int i = 0; i < 16; i++)
                    v[i] += bias[c0 + i];
            if (relu)
#pragma unroll
                for (int i = 0; i < 16; i++)
                    v[i] = fmaxf(v[i], 0.f);
            if (!mine)
                continue;
            if (out_bf16) {
                uint4 *o = reinterpret_cast<uint4 *>(reinterpret_cast<bf16 *>(out) + r * N + c0);
                o[0] = make_uint4(pack2(v[0], v[1]), pack2(v[2], v[3]), pack2(v[4], v[5]), pack2(v[6], v[7]));
                o[1] = make_uint4(pack2(v[8], v[9]), pack2(v[10], v[11]), pack2(v[12], v[13]), pack2(v[14], v[15]));
            } else {
                float4 *o = reinterpret_cast<float4 *>(reinterpret_cast<float *>(out) + r * N + c0);
#pragma unroll
                for (int i = 0; i < 4; i++)
                    o[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
            }
        }
    }
    // every MMA has completed (or the wait for one ran out) before the block leaves
    if (!bad)
        bad = !mbar_wait_for(acc_bar(tz - 1), 0, budget);
    tc_fence_before();
    bad = __syncthreads_or(bad);
    if (warp == 0)
        tc_dealloc(tmem, ncol);
    if (bad && tid == 0)
        atomicExch(err, 1);
}

// The halo convolution as a persistent kernel: each block loads all 27 taps'
// weights once and then walks tiles blockIdx.x, blockIdx.x + gridDim.x, ...
// with two halo buffers and two TMEM accumulators, so that the TMA of tile
// i + 2 and the MMAs of tile i + 1 run while the block stores tile i.  Thread
// 0 issues every copy and product; the mbarriers of buffer s (halo arrived,
// accumulator complete) complete once per tile on that buffer, the k-th time
// with parity k & 1, and a phase is always waited for before the next copy or
// product on that buffer is issued.  Every wait is bounded; on a timeout the
// block stops issuing, waits (bounded) for what it has in flight, frees its
// TMEM and raises *err.
template <int N, bool FLIP>
__global__ void __launch_bounds__(128) k_conv3_halo_p(const __grid_constant__ CUtensorMap tm_in,
                                                      const bf16 *__restrict__ W, int CK,
                                                      const float *__restrict__ bias, void *__restrict__ out,
                                                      int out_bf16, int relu, int lg, int ntiles, int fault,
                                                      int *__restrict__ err)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t mbar[4];   // 0, 1: halo of buffer s arrived; 2, 3: accumulator s complete
    __shared__ uint32_t tslot;
    constexpr int NCOL = N < 32 ? 32 : N;
    constexpr uint32_t IDESC = tc_idesc_bf16(128, N);
    const int tid = threadIdx.x, warp = tid >> 5;
    const int nk8 = CK >> 3;
    const uint32_t hbytes = (uint32_t)(nk8 * kHaloChunk);
    const uint32_t halo0 = smem_u32(smem), wts = halo0 + 2 * hbytes;
    const int n = 1 << lg;
    const int tx = n >> 3, ty = (n + 15) >> 4;
    if (warp == 0) {
        tc_alloc(smem_u32(&tslot), 2 * NCOL);
        tc_relinquish();
    }
    if (tid == 0) {
        for (int q = 0; q < 4; q++)
            mbar_init1(smem_u32(&mbar[q]));
        fence_mbar_init();
    }
    for (int e = tid; e < 27 * N * nk8; e += 128) {
        const int k8 = e % nk8, row = e / nk8;   // row = tap * N + output channel
        const int tap = row / N, nn = row - tap * N;
        cp16(wts + ((tap * nk8 + k8) * N + nn) * 16, W + (size_t)row * CK + 8 * k8, true);
    }
    cp_commit();
    cp_wait<0>();
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tslot;
    const int first = blockIdx.x, stride = gridDim.x;
    const int nt = first < ntiles ? (ntiles - 1 - first) / stride + 1 : 0;
    auto coords = [&](int i, int &x0, int &y0, int &z0, int &b) {
        int t = first + i * stride;
        x0 = (t % tx) * 8;
        t /= tx;
        y0 = (t % ty) * 16;
        t /= ty;
        z0 = t % n;
        b = t / n;
    };
    auto load = [&](int i) {   // thread 0: the halo of tile i into buffer i & 1
        int x0, y0, z0, b;
        coords(i, x0, y0, z0, b);
        const uint32_t mb = smem_u32(&mbar[i & 1]), dst = halo0 + (uint32_t)(i & 1) * hbytes;
        mbar_expect_tx(mb, (uint32_t)(nk8 * kHaloRows * 16));
        for (int k8 = 0; k8 < nk8; k8++)
            tma_load5(dst + k8 * kHaloChunk, &tm_in, 8 * k8, x0 - 1, y0 - 1, z0 - 1, b, mb);
    };
    auto issue = [&](int i) {   // thread 0: the 27 taps' products of tile i into accumulator i & 1
        const uint32_t hb = halo0 + (uint32_t)(i & 1) * hbytes, d = tmem + (uint32_t)((i & 1) * NCOL);
        tc_fence_after();
        for (int tap = 0; tap < 27; tap++) {
            int dz = tap / 9 - 1, dy = (tap / 3) % 3 - 1, dx = tap % 3 - 1;
            if (FLIP) {
                dz = -dz;
                dy = -dy;
                dx = -dx;
            }
            const uint32_t a0 = hb + (uint32_t)((((dz + 1) * 18 + dy + 1) * 10 + dx + 1) * 16);
            for (int k = 0; k < CK / 16; k++)
                tc_mma(d, tc_sdesc(a0 + 2 * k * kHaloChunk, kHaloChunk, 160),
                       tc_sdesc(wts + (tap * nk8 + 2 * k) * N * 16, N * 16, 128), IDESC,
                       (tap > 0 || k > 0) ? 1u : 0u);
        }
        tc_commit(smem_u32(&mbar[2 + (i & 1)]));
    };
    // thread 0's count of tiles whose copies were issued / waited for and
    // whose products were issued (for the exit after a timeout)
    int tma_issued = 0, tma_waited = 0, mma_issued = 0;
    bool ok = true;
    if (tid == 0 && nt > 0) {
        load(0);
        tma_issued = 1;
        if (nt > 1) {
            load(1);
            tma_issued = 2;
        }
        ok = mbar_wait_for(smem_u32(&mbar[0]), 0, kTcBudget);
        if (ok) {
            tma_waited = 1;
            if (!fault) {   // fault (test of the timeout path): nothing is issued, the accumulator wait runs out
                issue(0);
                mma_issued = 1;
            }
        }
    }
    ok = !__syncthreads_or(!ok);
    int i = 0;
    for (; ok && i < nt; i++) {
        const int s = i & 1;
        bool good = true;
        if (tid == 0 && i + 1 < nt) {
            good = mbar_wait_for(smem_u32(&mbar[(i + 1) & 1]), ((i + 1) >> 1) & 1, kTcBudget);
            if (good) {
                tma_waited = i + 2;
                if (!fault) {
                    issue(i + 1);
                    mma_issued = i + 2;
                }
            }
        }
        good = good && mbar_wait_for(smem_u32(&mbar[2 + s]), (i >> 1) & 1, fault ? (1ll << 21) : kTcBudget);
        if (__syncthreads_or(!good)) {
            ok = false;
            break;
        }
        if (tid == 0 && i + 2 < nt) {   // buffer s is free: the products of tile i have completed
            load(i + 2);
            tma_issued = i + 3;
        }
        tc_fence_after();
        int x0, y0, z0, b;
        coords(i, x0, y0, z0, b);
        const int x = x0 + (tid & 7), y = y0 + (tid >> 3);
        const bool mine = y < n;
        const size_t r = ((((size_t)b * n + z0) * n + y) * n + x);
        const uint32_t lane_base = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(s * NCOL);
        for (int c0 = 0; c0 < N; c0 += 16) {
            float v[16];
            tc_ld16(lane_base + c0, v);
            if (bias)
#pragma unroll
                for (int q = 0; q < 16; q++)
                    v[q] += bias[c0 + q];
            if (relu)
#pragma unroll
                for (int q = 0; q < 16; q++)
                    v[q] = fmaxf(v[q], 0.f);
            if (!mine)
                continue;
            if (out_bf16) {
                uint4 *o = reinterpret_cast<uint4 *>(reinterpret_cast<bf16 *>(out) + r * N + c0);
                o[0] = make_uint4(pack2(v[0], v[1]), pack2(v[2], v[3]), pack2(v[4], v[5]), pack2(v[6], v[7]));
                o[1] = make_uint4(pack2(v[8], v[9]), pack2(v[10], v[11]), pack2(v[12], v[13]), pack2(v[14], v[15]));
            } else {
                float4 *o = reinterpret_cast<float4 *>(reinterpret_cast<float *>(out) + r * N + c0);
#pragma unroll
                for (int q = 0; q < 4; q++)
                    o[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            }
        }
        tc_fence_before();
        __syncthreads();   // accumulator s read by every thread before tile i + 2's products
    }
    if (!ok && tid == 0) {   // what is still in flight lands before the block leaves
        for (int j = tma_waited; j < tma_issued; j++)
            mbar_wait_for(smem_u32(&mbar[j & 1]), (j >> 1) & 1, kTcBudget);
        for (int j = i; j < mma_issued; j++)
            mbar_wait_for(smem_u32(&mbar[2 + (j & 1)]), (j >> 1) & 1, kTcBudget);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0)
        tc_dealloc(tmem, 2 * NCOL);
    if (!ok && tid == 0)
        atomicExch(err, 1);
}

// Weight and bias gradients of a 3x3x3 convolution (FP32 on the CUDA cores):
//   dW[tap][ci][co] += sum_v in[v + off(tap)][ci] * d[v][co],  db[co] += sum_v d[v][co]
// Each block takes one tap and a run of voxels, stages 32 voxels at a time
// in shared memory and accumulates 4x4 (ci, co) tiles per thread.
__global__ void __launch_bounds__(kT) k_wgrad(const bf16 *__restrict__ in, int CKin, int Cin, const float *__restrict__ d,
                                              int N, float *__restrict__ dW, float *__restrict__ db, int lg, int V,
                                              int vox_per_block)
{
    constexpr int VS = 32;
    __shared__ float sIn[VS][128 + 1];
    __shared__ float sD[VS][64 + 1];
    const int tap = blockIdx.y;
    const int dz = tap / 9 - 1, dy = (tap / 3) % 3 - 1, dx = tap % 3 - 1;
    const int n = 1 << lg, msk = n - 1;
    const int ntc = Cin / 4 > 0 ? (Cin + 3) / 4 : 1, nto = N / 4;
    const int ntiles = ntc * nto;
    float acc[2][16];
    for (int u = 0; u < 2; u++)
        for (int e = 0; e < 16; e++)
            acc[u][e] = 0.f;
    float bacc = 0.f;
    const int vbeg = blockIdx.x * vox_per_block, vend = min(vbeg + vox_per_block, V);
    for (int v0 = vbeg; v0 < vend; v0 += VS) {
        __syncthreads();
        for (int e = threadIdx.x; e < VS * Cin; e += kT) {
            const int vv = e / Cin, ci = e - vv * Cin;
            const int v = v0 + vv;
            float val = 0.f;
            if (v < vend) {
                const int x = v & msk, y = (v >> lg) & msk, z = (v >> (2 * lg)) & msk, b = v >> (3 * lg);
                const int zz = z + dz, yy = y + dy, xx = x + dx;
                if ((unsigned)zz < (unsigned)n && (unsigned)yy < (unsigned)n && (unsigned)xx < (unsigned)n)
                    val = __bfloat162float(in[(size_t)((((b << lg | zz) << lg | yy) << lg) | xx) * CKin + ci]);
            }
            sIn[vv][ci] = val;
        }
        for (int e = threadIdx.x; e < VS * N; e += kT) {
            const int vv = e / N, co = e - vv * N;
            const int v = v0 + vv;
            sD[vv][co] = v < vend ? d[(size_t)v * N + co] : 0.f;
        }
        __syncthreads();
        for (int u = 0; u < 2; u++) {
            const int tile = threadIdx.x + u * kT;
            if (tile >= ntiles)
                break;
            const int tc = tile / nto, to = tile - tc * nto;
            for (int vv = 0; vv < VS; vv++) {
                float a[4], bb[4];
                for (int e = 0; e < 4; e++) {
                    const int ci = tc * 4 + e;
                    a[e] = ci < Cin ? sIn[vv][ci] : 0.f;
                    bb[e] = sD[vv][to * 4 + e];
                }
                for (int i = 0; i < 4; i++)
                    for (int j = 0; j < 4; j++)
                        acc[u][i * 4 + j] = fmaf(a[i], bb[j], acc[u][i * 4 + j]);
            }
        }
        if (tap == 13 && threadIdx.x < N)
            for (int vv = 0; vv < VS; vv++)
                bacc += sD[vv][threadIdx.x];
    }
    for (int u = 0; u < 2; u++) {
        const int tile = threadIdx.x + u * kT;
        if (tile >= ntiles)
            break;
        const int tc = tile / nto, to = tile - tc * nto;
        for (int i = 0; i < 4; i++) {
            const int ci = tc * 4 + i;
            if (ci >= Cin)
                continue;
            for (int j = 0; j < 4; j++)
                atomicAdd(&dW[((size_t)tap * Cin + ci) * N + to * 4 + j], acc[u][i * 4 + j]);
        }
    }
    if (tap == 13 && threadIdx.x < N && db)
        atomicAdd(&db[threadIdx.x], bacc);
}

// master FP32 weights [27][Cin][Cout] -> forward layout [27][Cout][CKin] and
// backward-data layout [27][Cin_p16][Cout] (BF16, zero padded)
__global__ void k_pack_weights(const float *__restrict__ w, int Cin, int CKin, int Cout, bf16 *__restrict__ wf,
                               bf16 *__restrict__ wd)
{
    const int total = 27 * CKin * Cout;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const int co = e % Cout, ci = (e / Cout) % CKin, tap = e / (Cout * CKin);
        const float v = ci < Cin ? w[((size_t)tap * Cin + ci) * Cout + co] : 0.f;
        wf[((size_t)tap * Cout + co) * CKin + ci] = __float2bfloat16_rn(v);
        if (wd)
            wd[((size_t)tap * CKin + ci) * Cout + co] = __float2bfloat16_rn(v);
    }
}

// 2x2x2 mean pool (BF16, C channels): fine n = 2^lg -> coarse
__global__ void k_pool(const bf16 *__restrict__ in, bf16 *__restrict__ out, int C, int lgc, int Vc)
{
    const int nc = 1 << lgc, m = nc - 1, lgf = lgc + 1, C8 = C >> 3;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < Vc * C8; e += gridDim.x * blockDim.x) {
        const int c = 8 * (e % C8), v = e / C8;
        const int x = v & m, y = (v >> lgc) & m, z = (v >> (2 * lgc)) & m, b = v >> (3 * lgc);
        uint4 q[8];
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const int fz = 2 * z + (k >> 2), fy = 2 * y + ((k >> 1) & 1), fx = 2 * x + (k & 1);
            q[k] = *reinterpret_cast<const uint4 *>(
                in + (size_t)((((b << lgf | fz) << lgf | fy) << lgf) | fx) * C + c);
        }
        float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int k = 0; k < 8; k++) {
            float f[8];
            unpack8(q[k], f);
#pragma unroll
            for (int i = 0; i < 8; i++)
                s[i] += f[i];
        }
#pragma unroll
        for (int i = 0; i < 8; i++)
            s[i] *= 0.125f;
        reinterpret_cast<uint4 *>(out)[e] =
            make_uint4(pack2(s[0], s[1]), pack2(s[2], s[3]), pack2(s[4], s[5]), pack2(s[6], s[7]));
    }
}

// pool backward, added: dIn[fine] += dOut[coarse] / 8
__global__ void k_pool_bwd_add(const float *__restrict__ dout, float *__restrict__ din, int C, int lgf, int Vf)
{
    const int nf = 1 << lgf, m = nf - 1, lgc = lgf - 1, C4 = C >> 2;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < Vf * C4; e += gridDim.x * blockDim.x) {
        const int c = 4 * (e % C4), v = e / C4;
        const int x = v & m, y = (v >> lgf) & m, z = (v >> (2 * lgf)) & m, b = v >> (3 * lgf);
        const float4 d = *reinterpret_cast<const float4 *>(
            dout + (size_t)((((b << lgc | (z >> 1)) << lgc | (y >> 1)) << lgc) | (x >> 1)) * C + c);
        float4 o = reinterpret_cast<float4 *>(din)[e];
        o.x += 0.125f * d.x;
        o.y += 0.125f * d.y;
        o.z += 0.125f * d.z;
        o.w += 0.125f * d.w;
        reinterpret_cast<float4 *>(din)[e] = o;
    }
}

// [up(low), skip] at the fine level: channels 0..Cu-1 from the parent, Cu..Cu+Cs-1 from skip
__global__ void k_upcat(const bf16 *__restrict__ low, int Cu, const bf16 *__restrict__ skip, int Cs,
                        bf16 *__restrict__ out, int lgf, int Vf)
{
    const int nf = 1 << lgf, m = nf - 1, lgc = lgf - 1, C8 = (Cu + Cs) >> 3;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < Vf * C8; e += gridDim.x * blockDim.x) {
        const int c = 8 * (e % C8), v = e / C8;
        const bf16 *src;
        if (c < Cu) {
            const int x = v & m, y = (v >> lgf) & m, z = (v >> (2 * lgf)) & m, b = v >> (3 * lgf);
            src = low + (size_t)((((b << lgc | (z >> 1)) << lgc | (y >> 1)) << lgc) | (x >> 1)) * Cu + c;
        } else {
            src = skip + (size_t)v * Cs + c - Cu;
        }
        reinterpret_cast<uint4 *>(out)[e] = *reinterpret_cast<const uint4 *>(src);
    }
}

// backward of k_upcat: dLow[coarse] = sum of the 8 children's channels 0..Cu-1; dSkip = channels Cu.. (written)
__global__ void k_upcat_bwd(const float *__restrict__ dout, int Cu, int Cs, float *__restrict__ dlow,
                            float *__restrict__ dskip, int lgc, int Vc)
{
    const int nc = 1 << lgc, m = nc - 1, lgf = lgc + 1, C = Cu + Cs, U4 = Cu >> 2, S4 = Cs >> 2;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < Vc * U4; e += gridDim.x * blockDim.x) {
        const int c = 4 * (e % U4), v = e / U4;
        const int x = v & m, y = (v >> lgc) & m, z = (v >> (2 * lgc)) & m, b = v >> (3 * lgc);
        float4 d[8];
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const int fz = 2 * z + (k >> 2), fy = 2 * y + ((k >> 1) & 1), fx = 2 * x + (k & 1);
            d[k] = *reinterpret_cast<const float4 *>(
                dout + (size_t)((((b << lgf | fz) << lgf | fy) << lgf) | fx) * C + c);
        }
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int k = 0; k < 8; k++) {
            s.x += d[k].x;
            s.y += d[k].y;
            s.z += d[k].z;
            s.w += d[k].w;
        }
        reinterpret_cast<float4 *>(dlow)[e] = s;
    }
    const int Vf = Vc * 8;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < Vf * S4; e += gridDim.x * blockDim.x) {
        const int c = 4 * (e % S4), v = e / S4;
        reinterpret_cast<float4 *>(dskip)[e] = *reinterpret_cast<const float4 *>(dout + (size_t)v * C + Cu + c);
    }
}

// d *= (act > 0)
__global__ void k_relu_mask(float *__restrict__ d, const bf16 *__restrict__ act, long n)
{
    for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < n; e += (long)gridDim.x * blockDim.x)
        if (!(__bfloat162float(act[e]) > 0.f))
            d[e] = 0.f;
}

// y[v] = sum_c d0[v][c] w[c] + b
__global__ void k_out1(const bf16 *__restrict__ d0, const float *__restrict__ w, const float *__restrict__ b,
                       float *__restrict__ y, int V)
{
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < V; v += gridDim.x * blockDim.x) {
        const uint4 *q = reinterpret_cast<const uint4 *>(d0) + 2 * (size_t)v;
        float f[16];
        unpack8(q[0], f);
        unpack8(q[1], f + 8);
        float s = b[0];
#pragma unroll
        for (int c = 0; c < 16; c++)
            s += f[c] * w[c];
        y[v] = s;
    }
}

// loss = mean (y - t)^2 per element; dy = 2 (y - t) / V; dd0 = dy w; dw, db of the 1x1 layer
__global__ void k_out1_bwd(const float *__restrict__ y, const float *__restrict__ tgt, const bf16 *__restrict__ d0,
                           const float *__restrict__ w, float *__restrict__ dd0, float *__restrict__ dw,
                           float *__restrict__ db, float *__restrict__ loss, int V)
{
    float accw[16], accb = 0.f, accl = 0.f;
    for (int c = 0; c < 16; c++)
        accw[c] = 0.f;
    const float inv = 1.f / (float)V;
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < V; v += gridDim.x * blockDim.x) {
        const float r = y[v] - tgt[v];
        const float dy = 2.f * r * inv;
        accl += r * r * inv;
        accb += dy;
        const uint4 *q = reinterpret_cast<const uint4 *>(d0) + 2 * (size_t)v;
        float f[16];
        unpack8(q[0], f);
        unpack8(q[1], f + 8);
#pragma unroll
        for (int c = 0; c < 16; c++)
            accw[c] += dy * f[c];
#pragma unroll
        for (int c = 0; c < 16; c += 4)
            *reinterpret_cast<float4 *>(dd0 + (size_t)v * 16 + c) =
                make_float4(dy * w[c], dy * w[c + 1], dy * w[c + 2], dy * w[c + 3]);
    }
    // block reductions of the 16 weight gradients, the bias gradient and the loss
    float vals[18];
    for (int c = 0; c < 16; c++)
        vals[c] = accw[c];
    vals[16] = accb;
    vals[17] = accl;
    for (int q = 0; q < 18; q++) {
        float v = vals[q];
        for (int o = 16; o > 0; o >>= 1)
            v += __shfl_down_sync(0xffffffffu, v, o);
        vals[q] = v;
    }
    __shared__ float red2[18][kT / 32];
    if ((threadIdx.x & 31) == 0)
        for (int q = 0; q < 18; q++)
            red2[q][threadIdx.x >> 5] = vals[q];
    __syncthreads();
    if (threadIdx.x < 18) {
        float s = 0.f;
        for (int wv = 0; wv < kT / 32; wv++)
            s += red2[threadIdx.x][wv];
        if (threadIdx.x < 16)
            atomicAdd(&dw[threadIdx.x], s);
        else if (threadIdx.x == 16)
            atomicAdd(db, s);
        else
            atomicAdd(loss, s);
    }
}

// AdamW on FP32 master weights
__global__ void k_adamw(float *__restrict__ p, const float *__restrict__ gr, float *__restrict__ m, float *__restrict__ v,
                        long n, float lr, float b1, float b2, float eps, float wd, float c1, float c2)
{
    for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < n; e += (long)gridDim.x * blockDim.x) {
        const float gg = gr[e];
        const float mm = b1 * m[e] + (1.f - b1) * gg;
        const float vv = b2 * v[e] + (1.f - b2) * gg * gg;
        m[e] = mm;
        v[e] = vv;
        p[e] -= lr * ((mm / c1) / (sqrtf(vv / c2) + eps) + wd * p[e]);
    }
}

// h^2 r = 4 pi G rho h^2 - (sum of the 6 neighbours - 6 Phi) on Omega, from
// (n+4)^3 level blocks (blk = 1) or copied from a dense array (blk = 0).
__global__ void k_resid_in(const double *__restrict__ rho, const double *__restrict__ phi,
                           const double *__restrict__ resid, int n, int blk, int lg, int B,
                           const double *__restrict__ frho, double *__restrict__ rh2)
{
    const int V = 1 << (3 * lg), m = (1 << lg) - 1, E = n + 4;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < B * V; e += gridDim.x * blockDim.x) {
        if (!blk) {
            rh2[e] = resid[e];
            continue;
        }
        const int b = e / V, v = e - b * V;
        const int x = v & m, y = (v >> lg) & m, z = v >> (2 * lg);
        const size_t q = (size_t)b * E * E * E + ((size_t)(z + 2) * E + y + 2) * E + x + 2;
        const size_t s1 = 1, s2 = E, s3 = (size_t)E * E;
        const double nb = phi[q - s1] + phi[q + s1] + phi[q - s2] + phi[q + s2] + phi[q - s3] + phi[q + s3];
        rh2[e] = frho[b] * rho[q] - (nb - 6.0 * phi[q]);
    }
}

// per sample b (blockIdx.y): the maxima of |Phi| on Omega and of |h^2 r| over
// this block's share of the cells, folded into bits[2b], bits[2b+1] by an
// atomic max on the float bit patterns (non-negative floats order as their
// bits: the result is the exact maximum, whatever the order)
__global__ void k_scales(const double *__restrict__ phi, const double *__restrict__ rh2, int n, int blk, int lg,
                         unsigned *__restrict__ bits)
{
    __shared__ float red[2][kT / 32];
    const int b = blockIdx.y;
    const int V = 1 << (3 * lg), m = (1 << lg) - 1, E = n + 4;
    float mx = 0.f, mr = 0.f;
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < V; v += gridDim.x * blockDim.x) {
        const int x = v & m, y = (v >> lg) & m, z = v >> (2 * lg);
        const size_t q = blk ? (size_t)b * E * E * E + ((size_t)(z + 2) * E + y + 2) * E + x + 2 : (size_t)b * V + v;
        mx = fmaxf(mx, fabsf((float)phi[q]));
        mr = fmaxf(mr, fabsf((float)rh2[(size_t)b * V + v]));
    }
    for (int o = 16; o > 0; o >>= 1) {
        mx = fmaxf(mx, __shfl_down_sync(0xffffffffu, mx, o));
        mr = fmaxf(mr, __shfl_down_sync(0xffffffffu, mr, o));
    }
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = mx;
        red[1][threadIdx.x >> 5] = mr;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        float s = 0.f, sr = 0.f;
        for (int w = 0; w < kT / 32; w++) {
            s = fmaxf(s, red[0][w]);
            sr = fmaxf(sr, red[1][w]);
        }
        atomicMax(&bits[2 * b], __float_as_uint(s));
        atomicMax(&bits[2 * b + 1], __float_as_uint(sr));
    }
}

// scale[2b] = max |Phi|, scale[2b+1] = max |h^2 r| (1 where the maximum is zero)
__global__ void k_scales_fin(const unsigned *__restrict__ bits, int B, float *__restrict__ scale)
{
    for (int e = threadIdx.x; e < 2 * B; e += blockDim.x) {
        const float v = __uint_as_float(bits[e]);
        scale[e] = v > 0.f ? v : 1.f;
    }
}

__global__ void k_make_input(const double *__restrict__ rho, const double *__restrict__ phi,
                             const double *__restrict__ rh2, int n, int blk, int lg, int B,
                             const double *__restrict__ frho, const float *__restrict__ scale, bf16 *__restrict__ x0)
{
    const int V = 1 << (3 * lg), m = (1 << lg) - 1, E = n + 4;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < B * V; e += gridDim.x * blockDim.x) {
        const int b = e / V, v = e - b * V;
        const int x = v & m, y = (v >> lg) & m, z = v >> (2 * lg);
        const size_t q = blk ? (size_t)b * E * E * E + ((size_t)(z + 2) * E + y + 2) * E + x + 2 : (size_t)e;
        const float s = scale[2 * b], sr = scale[2 * b + 1];
        uint4 *o = reinterpret_cast<uint4 *>(x0) + 2 * (size_t)e;
        o[0] = make_uint4(pack2((float)(frho[b] * rho[q]) / s, (float)phi[q] / s), pack2((float)rh2[e] / sr, 0.f), 0u, 0u);
        o[1] = make_uint4(0u, 0u, 0u, 0u);
    }
}

// output scale of sample b: s_r n^2 / 16
__device__ __forceinline__ double out_scale(const float *scale, int b, int n)
{
    return (double)scale[2 * b + 1] * (double)n * (double)n / 16.0;
}

// training target: (phi_true - phi_interp) / out_scale
__global__ void k_make_target(const double *__restrict__ phi_t, const double *__restrict__ phi_i,
                              const float *__restrict__ scale, int n, int V, int B, float *__restrict__ tgt)
{
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < B * V; e += gridDim.x * blockDim.x)
        tgt[e] = (float)((phi_t[e] - phi_i[e]) / out_scale(scale, e / V, n));
}

// Phi += out_scale * y on Omega (block or dense layout)
__global__ void k_apply(double *__restrict__ phi, int n, int blk, int lg, int B, const float *__restrict__ scale,
                        const float *__restrict__ y)
{
    const int V = 1 << (3 * lg), m = (1 << lg) - 1, E = n + 4;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < B * V; e += gridDim.x * blockDim.x) {
        const int b = e / V, v = e - b * V;
        const int x = v & m, yy = (v >> lg) & m, z = v >> (2 * lg);
        const size_t q = blk ? (size_t)b * E * E * E + ((size_t)(z + 2) * E + yy + 2) * E + x + 2 : (size_t)e;
        phi[q] += out_scale(scale, b, n) * (double)y[e];
    }
}

__global__ void k_fill(float *p, long n, float v)
{
    for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < n; e += (long)gridDim.x * blockDim.x)
        p[e] = v;
}

// ---------------------------------------------------------------------------
// layers
// ---------------------------------------------------------------------------
struct Conv {
    int cin, ckin, cout;     // real input channels, padded K channels, outputs
    long woff, boff;         // offsets into the parameter vector
};

// the nine 3x3x3 convolutions, then the 1x1 output (16 weights + bias)
const int kConvDims[9][2] = {{3, 16}, {16, 16}, {16, 32}, {32, 32}, {32, 64}, {64, 64}, {128, 32}, {64, 16}, {32, 16}};

int pad16(int c) { return (c + 15) / 16 * 16; }

}  // namespace

struct mg_unet {
    int nmax = 0, bmax = 0;
    Conv conv[9];
    long nparam = 0;
    float *p = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;   // FP32 master parameters and AdamW state
    bf16 *wf[9] = {}, *wd[9] = {};                                     // packed BF16 weights
    // activations (BF16) and gradients (FP32), sized for bmax * nmax^3
    bf16 *x0 = nullptr, *a0 = nullptr, *s0 = nullptr, *p0 = nullptr, *a1 = nullptr, *s1 = nullptr, *p1 = nullptr,
         *s2 = nullptr, *p2 = nullptr, *a3 = nullptr, *u2 = nullptr, *d2 = nullptr, *u1 = nullptr, *d1 = nullptr,
         *u0 = nullptr, *d0 = nullptr;
    float *y = nullptr, *tgt = nullptr, *scale = nullptr, *loss = nullptr, *gA = nullptr, *gB = nullptr, *gC = nullptr;
    double *frho = nullptr, *rh2 = nullptr;
    int *tcerr = nullptr;          // set when a tensor-core completion wait ran out
    bf16 *gbf = nullptr;           // BF16 copy of a data-gradient pass's input gradient
    unsigned *scale_bits = nullptr; // per-sample maxima as float bit patterns
    char *mem = nullptr;
    long step = 0;
    cudaStream_t stream = nullptr;
    bool packed = false;
};

namespace {

// The convolutions run on tcgen05 (k_conv3_tc); UNET_MMA_SYNC=1 selects the
// warp-level mma.sync kernel instead (for comparison).
bool use_mma_sync()
{
    static const bool on = [] {
        const char *v = std::getenv("UNET_MMA_SYNC");
        return v && v[0] == '1';
    }();
    return on;
}

int ilog2(int n)
{
    int l = 0;
    while ((1 << l) < n)
        l++;
    return l;
}

constexpr int kTcSmemMax = 200 * 1024;  // kTcStages stages of 128 x CK and N x CK BF16 tiles

template <int N, bool FLIP>
cudaError_t conv_launch_tc(const bf16 *in, int CK, const bf16 *W, const float *bias, void *out, int out_bf16,
                           int relu, int lg, int V, int *err, cudaStream_t s)
{
    static cudaError_t attr = cudaFuncSetAttribute(k_conv3_tc<N, FLIP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   kTcSmemMax);
    if (attr)
        return attr;
    const size_t smem = (size_t)kTcStages * ((size_t)128 * CK * 2 + (size_t)N * CK * 2);
    if (smem > (size_t)kTcSmemMax || CK % 16 || CK > 128)
        return cudaErrorInvalidValue;
    k_conv3_tc<N, FLIP><<<(V + 127) / 128, 128, smem, s>>>(in, CK, W, bias, out, out_bf16, relu, lg, V, err);
    return cudaGetLastError();
}

PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder()
{
    static const PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            p = nullptr;
        }
        return (PFN_cuTensorMapEncodeTiled_v12000)p;
    }();
    return fn;
}

// the persistent halo kernel with UNET_HALO_P=1 (as fast as the form of
// k_conv3_halo with one plane per block, slower than with several)
bool use_persistent_halo()
{
    static const bool on = [] {
        const char *v = std::getenv("UNET_HALO_P");
        return v && v[0] == '1';
    }();
    return on;
}

template <int N, bool FLIP, int CK>
cudaError_t conv_launch_halo(const bf16 *in, const bf16 *W, const float *bias, void *out, int out_bf16, int relu,
                             int lg, int V, int *err, cudaStream_t s)
{
    const int n = 1 << lg, B = V >> (3 * lg);
    static cudaError_t attr = cudaFuncSetAttribute(k_conv3_halo<N, FLIP, CK>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
    if (attr)
        return attr;
    const int tiles = B * n * ((n + 15) / 16) * (n / 8);   // of one plane
    static const int fault = [] {   // UNET_FAULT_WAIT=1: the accumulator waits run out (test of that path)
        const char *v = std::getenv("UNET_FAULT_WAIT");
        return v && v[0] == '1' ? 1 : 0;
    }();
    if (halo_resident(CK, N) && use_persistent_halo()) {
        const PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
        if (!enc)
            return cudaErrorNotSupported;
        CUtensorMap mi{};
        const cuuint64_t di[5] = {(cuuint64_t)CK, (cuuint64_t)n, (cuuint64_t)n, (cuuint64_t)n, (cuuint64_t)B};
        const cuuint64_t si[4] = {(cuuint64_t)CK * 2, (cuuint64_t)n * CK * 2, (cuuint64_t)n * n * CK * 2,
                                  (cuuint64_t)n * n * n * CK * 2};
        const cuuint32_t bi[5] = {8, 10, 18, 3, 1}, e5[5] = {1, 1, 1, 1, 1};
        if (enc(&mi, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<bf16 *>(in), di, si, bi, e5,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
        // persistent form: as many blocks as fit on the SMs at once, but never
        // more per SM than TMEM holds (each block keeps two accumulators of
        // NCOL columns allocated for its whole life; a block that could not
        // allocate would wait for one that never leaves)
        constexpr int NCOL = N < 32 ? 32 : N;
        constexpr int tmem_blocks = 512 / (2 * NCOL);
        size_t psmem = 2 * (size_t)(CK / 8) * kHaloChunk + (size_t)27 * (CK / 8) * N * 16;
        const size_t floor_smem = 233472 / (tmem_blocks + 1);   // more than 1/(t+1) of an SM's shared memory
        if (psmem < floor_smem)
            psmem = floor_smem;
        static cudaError_t pattr = [] {   // all of the SM's shared memory for several blocks
            cudaError_t e = cudaFuncSetAttribute(k_conv3_halo_p<N, FLIP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 200 * 1024);
            if (!e)
                e = cudaFuncSetAttribute(k_conv3_halo_p<N, FLIP>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                         (int)cudaSharedmemCarveoutMaxShared);
            return e;
        }();
        if (pattr)
            return pattr;
        int per_sm = 0, dev = 0, nsm = 0;
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_conv3_halo_p<N, FLIP>, 128, psmem);
        if (!e)
            e = cudaGetDevice(&dev);
        if (!e)
            e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        if (e)
            return e;
        // with one block per SM a block's tiles run one after another with
        // little to overlap: the one-tile-per-block kernel is faster there
        if (psmem <= 200 * 1024 && per_sm >= 2 && per_sm <= tmem_blocks) {
            const int grid = std::min(tiles, per_sm * nsm);
            k_conv3_halo_p<N, FLIP><<<grid, 128, psmem, s>>>(mi, W, CK, bias, out, out_bf16, relu, lg, tiles, fault,
                                                             err);
            return cudaGetLastError();
        }
    }
    // planes per block: fewer loads per voxel against fewer blocks.  Time of a
    // wave of blocks on an SM in cycles: copies at 64 bytes and MMAs at 32
    // cycles (each reads 4 KB of shared memory) overlap between the blocks of an
    // SM; a block alone does one after the other.
    int tz = 1, ncol = 32;
    size_t smem = 0;
    double best = 0.0;
    for (int z = 1; z <= (halo_resident(CK, N) ? 4 : 1); z *= 2) {
        const int cols = std::max(32, z * N);
        const size_t sm =
            (size_t)(CK / 8) * halo_chunk(z) + (size_t)(halo_resident(CK, N) ? 27 : 9) * (CK / 8) * (N + 1) * 16;
        if (sm > 226 * 1024 || cols > 512)
            continue;
        const int per_sm = std::min((int)(227 * 1024 / (sm + 2048)), 512 / cols);
        const double copy = sm / 64.0, mma = z * 27.0 * (CK / 16) * 32.0;
        const int blocks = tiles / z, waves = (blocks + 152 * per_sm - 1) / (152 * per_sm);
        const int co = std::min(per_sm, (blocks + 151) / 152);   // blocks at once on an SM
        const double time = waves * (co * std::max(copy, mma) + std::min(copy, mma) + 3000.0);
        if (best == 0.0 || time < best) {
            best = time;
            tz = z;
            ncol = cols;
            smem = sm;
        }
    }
    if (!smem)
        return cudaErrorInvalidValue;
    k_conv3_halo<N, FLIP, CK><<<tiles / tz, 256, smem, s>>>(in, W, bias, out, out_bf16, relu, lg, tz, ncol, fault, err);
    return cudaGetLastError();
}

// the halo kernel unless UNET_HALO=0
bool use_halo()
{
    static const bool on = [] {
        const char *v = std::getenv("UNET_HALO");
        return !(v && v[0] == '0');
    }();
    return on;
}

// tcgen05 path: BF16 input; the mma.sync kernel also takes FP32 (the
// data-gradient pass) and rounds it when it loads it
template <int NT, bool FLIP, typename TIn>
cudaError_t conv_launch(const TIn *in, int CK, const bf16 *W, const float *bias, void *out, int out_bf16, int relu,
                        int lg, int V, int *err, cudaStream_t s)
{
    if (!use_mma_sync()) {
        if constexpr (sizeof(TIn) == 2) {
            if (use_halo() && lg >= 3) {
#define HALO(ck)      \
    if (CK == ck)     \
        return conv_launch_halo<NT * 8, FLIP, ck>(in, W, bias, out, out_bf16, relu, lg, V, err, s);
                HALO(16) HALO(32) HALO(64)
                if constexpr (NT * 8 <= 32)
                    HALO(128)
#undef HALO
            }
            return conv_launch_tc<NT * 8, FLIP>(in, CK, W, bias, out, out_bf16, relu, lg, V, err, s);
        }
        return cudaErrorInvalidValue;
    }
    k_conv3<NT, FLIP, TIn><<<(V + 63) / 64, 128, 0, s>>>(in, CK, W, bias, out, out_bf16, relu, lg, V);
    return cudaGetLastError();
}

template <bool FLIP, typename TIn>
cudaError_t conv_any(const TIn *in, int CK, const bf16 *W, const float *bias, int N, void *out, int out_bf16, int relu,
                     int lg, int V, int *err, cudaStream_t s)
{
    switch (N) {
    case 16: return conv_launch<2, FLIP, TIn>(in, CK, W, bias, out, out_bf16, relu, lg, V, err, s);
    case 32: return conv_launch<4, FLIP, TIn>(in, CK, W, bias, out, out_bf16, relu, lg, V, err, s);
    case 64: return conv_launch<8, FLIP, TIn>(in, CK, W, bias, out, out_bf16, relu, lg, V, err, s);
    case 128: return conv_launch<16, FLIP, TIn>(in, CK, W, bias, out, out_bf16, relu, lg, V, err, s);
    }
    return cudaErrorInvalidValue;
}

cudaError_t pack_all(mg_unet *u)
{
    for (int i = 0; i < 9; i++) {
        const Conv &c = u->conv[i];
        k_pack_weights<<<blocks_for(27L * c.ckin * c.cout), kT, 0, u->stream>>>(u->p + c.woff, c.cin, c.ckin, c.cout,
                                                                              u->wf[i], u->wd[i]);
    }
    u->packed = true;
    return cudaGetLastError();
}

// forward through the network for B samples of edge n = 2^lg (x0 ready)
cudaError_t forward(mg_unet *u, int B, int lg)
{
    cudaStream_t s = u->stream;
    const int V0 = B << (3 * lg), V1 = V0 >> 3, V2 = V1 >> 3, V3 = V2 >> 3;
    cudaError_t e;
    auto C = [&](int i) -> const Conv & { return u->conv[i]; };
    float *P = u->p;
#define FWD(i, in, out, lgv, V)                                                                                   \
    if ((e = conv_any<false, bf16>(in, C(i).ckin, u->wf[i], P + C(i).boff, C(i).cout, out, 1, 1, lgv, V, u->tcerr, \
                                   s)))                                                                \
        return e;
    FWD(0, u->x0, u->a0, lg, V0);
    FWD(1, u->a0, u->s0, lg, V0);
    k_pool<<<blocks_for((long)V1 * 2), kT, 0, s>>>(u->s0, u->p0, 16, lg - 1, V1);
    FWD(2, u->p0, u->a1, lg - 1, V1);
    FWD(3, u->a1, u->s1, lg - 1, V1);
    k_pool<<<blocks_for((long)V2 * 4), kT, 0, s>>>(u->s1, u->p1, 32, lg - 2, V2);
    FWD(4, u->p1, u->s2, lg - 2, V2);
    k_pool<<<blocks_for((long)V3 * 8), kT, 0, s>>>(u->s2, u->p2, 64, lg - 3, V3);
    FWD(5, u->p2, u->a3, lg - 3, V3);
    k_upcat<<<blocks_for((long)V2 * 16), kT, 0, s>>>(u->a3, 64, u->s2, 64, u->u2, lg - 2, V2);
    FWD(6, u->u2, u->d2, lg - 2, V2);
    k_upcat<<<blocks_for((long)V1 * 8), kT, 0, s>>>(u->d2, 32, u->s1, 32, u->u1, lg - 1, V1);
    FWD(7, u->u1, u->d1, lg - 1, V1);
    k_upcat<<<blocks_for((long)V0 * 4), kT, 0, s>>>(u->d1, 16, u->s0, 16, u->u0, lg, V0);
    FWD(8, u->u0, u->d0, lg, V0);
#undef FWD
    k_out1<<<blocks_for(V0), kT, 0, s>>>(u->d0, P + u->nparam - 17, P + u->nparam - 1, u->y, V0);
    return cudaGetLastError();
}

template <int CK, int N, int NZ>
cudaError_t wgrad_rows(const bf16 *in, int Cin, const bf16 *gbf, float *dW, int lg, int V, int *err, cudaStream_t s)
{
    typedef WgradTile<CK, N, NZ> W;
    static cudaError_t attr = cudaFuncSetAttribute(k_wgrad_rows<CK, N, NZ>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   W::kSmemMax);
    if (attr)
        return attr;
    // no more blocks per SM than tensor memory has room for: a block never waits for its columns
    const int most = 512 / W::kAlloc, smem = std::max(2 * W::stage(1 << lg), W::kSmemMax / (most + 1) + 1024);
    // a block per chain (and dz with NZ = 1), and per dx where that leaves SMs without one
    const int chains = (V + kWgradChain - 1) / kWgradChain, nz = NZ == 3 ? 1 : 3, ndx = nz * chains < 152 ? 1 : 3;
    k_wgrad_rows<CK, N, NZ><<<dim3(chains, ndx == 1 ? 3 * nz : nz), 256, smem, s>>>(in, Cin, gbf, dW, lg,
                                                                                   V >> (3 * lg), ndx, err);
    return cudaGetLastError();
}

template <int CK, int N>
cudaError_t wgrad_tc(const bf16 *in, int Cin, const float *g, const bf16 *gbf, float *dW, int lg, int V, int *err,
                     cudaStream_t s)
{
    if constexpr (WgradTile<CK, N, 3>::kCols <= 512)
        if (WgradTile<CK, N, 3>::applies(lg))
            return wgrad_rows<CK, N, 3>(in, Cin, gbf, dW, lg, V, err, s);
    if (WgradTile<CK, N, 1>::applies(lg))
        return wgrad_rows<CK, N, 1>(in, Cin, gbf, dW, lg, V, err, s);
    constexpr size_t smem = 2 * ((size_t)128 * 64 * 2 + (size_t)N * 64 * 2);
    static cudaError_t attr = cudaFuncSetAttribute(k_wgrad_tc<CK, N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)smem);
    if (attr)
        return attr;
    const int vchunk = kWgradChain;
    dim3 grid((V + vchunk - 1) / vchunk, (27 + 128 / CK - 1) / (128 / CK));
    k_wgrad_tc<CK, N><<<grid, 128, smem, s>>>(in, Cin, g, dW, lg, V, vchunk, err);
    return cudaGetLastError();
}

// whether k_wgrad_rows takes the layer (else k_wgrad_tc, which reads the masked FP32 gradient)
bool wgrad_by_rows(int CK, int N, int lg)
{
#define WG(ck, nn)                   \
    if (CK == ck && N == nn)         \
        return WgradTile<ck, nn, 1>::applies(lg) || WgradTile<ck, nn, 3>::applies(lg);
    WG(16, 16) WG(16, 32) WG(32, 32) WG(32, 64) WG(64, 64) WG(128, 32) WG(64, 16) WG(32, 16)
#undef WG
    return false;
}

cudaError_t wgrad_tc_any(int CK, int N, const bf16 *in, int Cin, const float *g, const bf16 *gbf, float *dW, int lg,
                         int V, int *err, cudaStream_t s)
{
#define WG(ck, nn)                   \
    if (CK == ck && N == nn)         \
        return wgrad_tc<ck, nn>(in, Cin, g, gbf, dW, lg, V, err, s);
    WG(16, 16) WG(16, 32) WG(32, 32) WG(32, 64) WG(64, 64) WG(128, 32) WG(64, 16) WG(32, 16)
#undef WG
    return cudaErrorInvalidValue;
}

// weight and bias gradients of conv i from its input activation `in`, its
// output activation `act` and output gradient g (FP32, N channels); leaves what
// dgrad reads: the masked g, in BF16 in gbf on the tensor-core path
cudaError_t wgrad(mg_unet *u, int i, const bf16 *in, const bf16 *act, float *g, int lg, int V)
{
    const Conv &c = u->conv[i];
    const long n8 = (long)V * c.cout / 8;
    if (use_mma_sync()) {
        k_relu_mask<<<blocks_for(8 * n8), kT, 0, u->stream>>>(g, act, 8 * n8);
        const int vpb = 4096;
        dim3 grid((V + vpb - 1) / vpb, 27);
        k_wgrad<<<grid, kT, 0, u->stream>>>(in, c.ckin, c.cin, g, c.cout, u->grad + c.woff, u->grad + c.boff, lg, V,
                                            vpb);
        return cudaGetLastError();
    }
    k_grad_prep<<<blocks_for(n8, 152 * 8), 256, 0, u->stream>>>(g, act, c.cout, n8, u->gbf, u->grad + c.boff,
                                                                wgrad_by_rows(c.ckin, c.cout, lg) ? 0 : 1);
    return wgrad_tc_any(c.ckin, c.cout, in, c.cin, g, u->gbf, u->grad + c.woff, lg, V, u->tcerr, u->stream);
}

cudaError_t dgrad(mg_unet *u, int i, const float *g, float *out, int lg, int V)
{
    const Conv &c = u->conv[i];
    if (use_mma_sync())
        return conv_any<true, float>(g, c.cout, u->wd[i], nullptr, c.ckin, out, 0, 0, lg, V, u->tcerr, u->stream);
    return conv_any<true, bf16>(u->gbf, c.cout, u->wd[i], nullptr, c.ckin, out, 0, 0, lg, V, u->tcerr, u->stream);
}

// backward pass (loss gradient from y vs tgt), accumulating into u->grad
cudaError_t backward(mg_unet *u, int B, int lg)
{
    cudaStream_t s = u->stream;
    const int V0 = B << (3 * lg), V1 = V0 >> 3, V2 = V1 >> 3, V3 = V2 >> 3;
    float *gA = u->gA, *gB = u->gB, *gC = u->gC;
    cudaError_t e;
    k_out1_bwd<<<blocks_for(V0, 152 * 4), kT, 0, s>>>(u->y, u->tgt, u->d0, u->p + u->nparam - 17, gA,
                                                     u->grad + u->nparam - 17, u->grad + u->nparam - 1, u->loss, V0);
    // D0 (u0 -> d0), gA = dd0 [V0][16]
    if ((e = wgrad(u, 8, u->u0, u->d0, gA, lg, V0)) ||
        (e = dgrad(u, 8, gA, gB, lg, V0)))
        return e;                                                        // gB = du0 [V0][32]
    // split du0 -> dd1 (coarse) and ds0 (gC)
    k_upcat_bwd<<<blocks_for((long)V0 * 4), kT, 0, s>>>(gB, 16, 16, gA, gC, lg - 1, V1);   // gA = dd1 [V1][16], gC = ds0 [V0][16]
    if ((e = wgrad(u, 7, u->u1, u->d1, gA, lg - 1, V1)) ||
        (e = dgrad(u, 7, gA, gB, lg - 1, V1)))
        return e;                                                        // gB = du1 [V1][64]
    // ds1 lives behind ds0 in gC
    float *ds1 = gC + (size_t)V0 * 16;
    k_upcat_bwd<<<blocks_for((long)V1 * 8), kT, 0, s>>>(gB, 32, 32, gA, ds1, lg - 2, V2);  // gA = dd2 [V2][32]
    if ((e = wgrad(u, 6, u->u2, u->d2, gA, lg - 2, V2)) ||
        (e = dgrad(u, 6, gA, gB, lg - 2, V2)))
        return e;                                                        // gB = du2 [V2][128]
    float *ds2 = ds1 + (size_t)V1 * 32;
    k_upcat_bwd<<<blocks_for((long)V2 * 16), kT, 0, s>>>(gB, 64, 64, gA, ds2, lg - 3, V3);  // gA = da3 [V3][64]
    if ((e = wgrad(u, 5, u->p2, u->a3, gA, lg - 3, V3)) ||
        (e = dgrad(u, 5, gA, gB, lg - 3, V3)))
        return e;                                                        // gB = dp2 [V3][64]
    k_pool_bwd_add<<<blocks_for((long)V2 * 16), kT, 0, s>>>(gB, ds2, 64, lg - 2, V2);
    if ((e = wgrad(u, 4, u->p1, u->s2, ds2, lg - 2, V2)) ||
        (e = dgrad(u, 4, ds2, gB, lg - 2, V2)))
        return e;                                                        // gB = dp1 [V2][32]
    k_pool_bwd_add<<<blocks_for((long)V1 * 8), kT, 0, s>>>(gB, ds1, 32, lg - 1, V1);
    if ((e = wgrad(u, 3, u->a1, u->s1, ds1, lg - 1, V1)) ||
        (e = dgrad(u, 3, ds1, gB, lg - 1, V1)))
        return e;                                                        // gB = da1 [V1][32]
    if ((e = wgrad(u, 2, u->p0, u->a1, gB, lg - 1, V1)) ||
        (e = dgrad(u, 2, gB, gA, lg - 1, V1)))
        return e;                                                        // gA = dp0 [V1][16]
    float *ds0 = gC;
    k_pool_bwd_add<<<blocks_for((long)V0 * 4), kT, 0, s>>>(gA, ds0, 16, lg, V0);
    if ((e = wgrad(u, 1, u->a0, u->s0, ds0, lg, V0)) ||
        (e = dgrad(u, 1, ds0, gB, lg, V0)))
        return e;                                                        // gB = da0 [V0][16]
    if ((e = wgrad(u, 0, u->x0, u->a0, gB, lg, V0)))
        return e;
    return cudaGetLastError();
}

// He-style initialisation from a counter-based hash (deterministic per seed)
float hash_uniform(unsigned long long seed, unsigned long long i)
{
    unsigned long long z = seed + 0x9E3779B97F4A7C15ull * (i + 1);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    return (float)((z >> 11) * (1.0 / 9007199254740992.0));
}

}  // namespace

namespace {

// 4 once a tensor-core completion wait of a convolution ran out (the flag
// stays set), else 0; synchronises the stream
int tc_status(mg_unet *u)
{
    int f = 0;
    if (cudaMemcpyAsync(&f, u->tcerr, sizeof(int), cudaMemcpyDeviceToHost, u->stream) ||
        cudaStreamSynchronize(u->stream))
        return 3;
    return f ? 4 : 0;
}

}  // namespace

extern "C" {

long mg_unet_param_count(void)
{
    long n = 0;
    for (int i = 0; i < 9; i++)
        n += 27L * kConvDims[i][0] * kConvDims[i][1] + kConvDims[i][1];
    return n + 17;
}

int mg_unet_create(int nmax, int bmax, unsigned long long seed, void *stream, mg_unet **out)
{
    if (!out)
        return 1;
    *out = nullptr;
    if (nmax < 8 || (nmax & (nmax - 1)) || bmax < 1 || bmax > 1024)
        return 1;
    mg_unet *u = new (std::nothrow) mg_unet();
    if (!u)
        return 2;
    u->nmax = nmax;
    u->bmax = bmax;
    u->stream = (cudaStream_t)stream;
    long off = 0;
    for (int i = 0; i < 9; i++) {
        Conv &c = u->conv[i];
        c.cin = kConvDims[i][0];
        c.ckin = pad16(c.cin);
        c.cout = kConvDims[i][1];
        c.woff = off;
        off += 27L * c.cin * c.cout;
        c.boff = off;
        off += c.cout;
    }
    u->nparam = off + 17;
    const long V0 = (long)bmax * nmax * nmax * nmax;
    // arena
    std::vector<std::pair<void **, size_t>> sl;
    auto A = [&](void **p, size_t b) { sl.push_back({p, (b + 255) & ~(size_t)255}); };
    for (void **pp : {(void **)&u->p, (void **)&u->grad, (void **)&u->m, (void **)&u->v})
        A(pp, u->nparam * sizeof(float));
    for (int i = 0; i < 9; i++) {
        A((void **)&u->wf[i], 27L * u->conv[i].ckin * u->conv[i].cout * sizeof(bf16));
        A((void **)&u->wd[i], 27L * u->conv[i].ckin * u->conv[i].cout * sizeof(bf16));
    }
    const long V1 = V0 / 8, V2 = V1 / 8, V3 = V2 / 8;
    A((void **)&u->x0, V0 * 16 * sizeof(bf16));
    A((void **)&u->a0, V0 * 16 * sizeof(bf16));
    A((void **)&u->s0, V0 * 16 * sizeof(bf16));
    A((void **)&u->p0, V1 * 16 * sizeof(bf16));
    A((void **)&u->a1, V1 * 32 * sizeof(bf16));
    A((void **)&u->s1, V1 * 32 * sizeof(bf16));
    A((void **)&u->p1, V2 * 32 * sizeof(bf16));
    A((void **)&u->s2, V2 * 64 * sizeof(bf16));
    A((void **)&u->p2, V3 * 64 * sizeof(bf16));
    A((void **)&u->a3, V3 * 64 * sizeof(bf16));
    A((void **)&u->u2, V2 * 128 * sizeof(bf16));
    A((void **)&u->d2, V2 * 32 * sizeof(bf16));
    A((void **)&u->u1, V1 * 64 * sizeof(bf16));
    A((void **)&u->d1, V1 * 16 * sizeof(bf16));
    A((void **)&u->u0, V0 * 32 * sizeof(bf16));
    A((void **)&u->d0, V0 * 16 * sizeof(bf16));
    A((void **)&u->y, V0 * sizeof(float));
    A((void **)&u->tgt, V0 * sizeof(float));
    A((void **)&u->scale, 2048 * sizeof(float));
    A((void **)&u->scale_bits, 2048 * sizeof(unsigned));
    A((void **)&u->rh2, V0 * sizeof(double));
    A((void **)&u->loss, 256);
    A((void **)&u->tcerr, 256);
    A((void **)&u->gbf, V0 * 32 * sizeof(bf16));
    A((void **)&u->frho, bmax * sizeof(double));
    A((void **)&u->gA, V0 * 32 * sizeof(float));
    A((void **)&u->gB, V0 * 32 * sizeof(float));
    A((void **)&u->gC, (V0 * 16 + V1 * 32 + V2 * 64) * sizeof(float));
    size_t bytes = 0;
    for (auto &x : sl)
        bytes += x.second;
    if (cudaMalloc((void **)&u->mem, bytes) != cudaSuccess) {
        cudaGetLastError();
        delete u;
        return 2;
    }
    size_t pos = 0;
    for (auto &x : sl) {
        *x.first = u->mem + pos;
        pos += x.second;
    }
    cudaMemsetAsync(u->mem, 0, bytes, u->stream);
    // initial parameters: uniform(-a, a), a = sqrt(6 / fan_in); zero biases
    std::vector<float> h(u->nparam, 0.f);
    for (int i = 0; i < 9; i++) {
        const Conv &c = u->conv[i];
        const float a = std::sqrt(6.f / (27.f * c.cin));
        for (long k = 0; k < 27L * c.cin * c.cout; k++)
            h[c.woff + k] = a * (2.f * hash_uniform(seed, c.woff + k) - 1.f);
    }
    for (int c = 0; c < 16; c++)
        h[u->nparam - 17 + c] = 0.01f * (2.f * hash_uniform(seed, u->nparam + c) - 1.f);
    cudaMemcpyAsync(u->p, h.data(), u->nparam * sizeof(float), cudaMemcpyHostToDevice, u->stream);
    if (cudaStreamSynchronize(u->stream) != cudaSuccess) {
        cudaGetLastError();
        cudaFree(u->mem);
        delete u;
        return 3;
    }
    *out = u;
    return 0;
}

int mg_unet_destroy(mg_unet *u)
{
    if (!u)
        return 0;
    cudaStreamSynchronize(u->stream);
    cudaFree(u->mem);
    cudaGetLastError();
    delete u;
    return 0;
}

int mg_unet_get_params(mg_unet *u, float *out)
{
    if (!u || !out)
        return 1;
    if (cudaMemcpyAsync(out, u->p, u->nparam * sizeof(float), cudaMemcpyDeviceToHost, u->stream) ||
        cudaStreamSynchronize(u->stream))
        return 3;
    return 0;
}

int mg_unet_set_params(mg_unet *u, const float *in)
{
    if (!u || !in)
        return 1;
    if (cudaMemcpyAsync(u->p, in, u->nparam * sizeof(float), cudaMemcpyHostToDevice, u->stream) ||
        cudaStreamSynchronize(u->stream))
        return 3;
    u->packed = false;
    u->step = 0;
    return 0;
}

// Pack the BF16 weight copies now (before a solve graph captures inference).
int mg_unet_pack(mg_unet *u)
{
    if (!u)
        return 1;
    if (pack_all(u) || cudaStreamSynchronize(u->stream))
        return 3;
    return 0;
}

int mg_unet_get_grad(mg_unet *u, float *out)
{
    if (!u || !out)
        return 1;
    if (cudaMemcpyAsync(out, u->grad, u->nparam * sizeof(float), cudaMemcpyDeviceToHost, u->stream) ||
        cudaStreamSynchronize(u->stream))
        return 3;
    return 0;
}

// Internal entry used by the solver and by the public calls: from (n+4)^3
// blocks (blk = 1) or dense n^3 arrays (blk = 0) of B samples, predict y and
// (apply = 1) add scale * y to phi on Omega.
int mg_unet_predict_dev(mg_unet *u, int B, int n, int blk, const double *rho, double *phi, const double *resid,
                        const double *frho_dev, int apply, void *stream)
{
    if (!u || B < 1 || B > u->bmax || n < 8 || n > u->nmax || (n & (n - 1)) || (!blk && !resid))
        return 1;
    cudaStream_t s = stream ? (cudaStream_t)stream : u->stream;
    cudaStream_t keep = u->stream;
    u->stream = s;
    const int lg = ilog2(n);
    const int V0 = B << (3 * lg);
    if (!u->packed && pack_all(u)) {
        u->stream = keep;
        return 3;
    }
    k_resid_in<<<blocks_for(V0), kT, 0, s>>>(rho, phi, resid, n, blk, lg, B, frho_dev, u->rh2);
    cudaMemsetAsync(u->scale_bits, 0, 2 * B * sizeof(unsigned), s);
    k_scales<<<dim3(std::min(64, std::max(1, V0 / B / (kT * 16))), B), kT, 0, s>>>(phi, u->rh2, n, blk, lg,
                                                                                  u->scale_bits);
    k_scales_fin<<<1, 256, 0, s>>>(u->scale_bits, B, u->scale);
    k_make_input<<<blocks_for(V0), kT, 0, s>>>(rho, phi, u->rh2, n, blk, lg, B, frho_dev, u->scale, u->x0);
    cudaError_t e = forward(u, B, lg);
    if (!e && apply) {
        k_apply<<<blocks_for(V0), kT, 0, s>>>(phi, n, blk, lg, B, u->scale, u->y);
        e = cudaGetLastError();
    }
    u->stream = keep;
    return e ? 3 : 0;
}

int mg_unet_forward(mg_unet *u, int B, int n, const double *rho, const double *phi_interp, const double *resid,
                    const double *frho, float *y_out)
{
    if (!u || !frho || B > u->bmax)
        return 1;
    if (cudaMemcpyAsync(u->frho, frho, B * sizeof(double), cudaMemcpyHostToDevice, u->stream))
        return 3;
    int r = mg_unet_predict_dev(u, B, n, 0, rho, const_cast<double *>(phi_interp), resid, u->frho, 0, nullptr);
    if (r)
        return r;
    const long V0 = (long)B * n * n * n;
    if (y_out && (cudaMemcpyAsync(y_out, u->y, V0 * sizeof(float), cudaMemcpyDeviceToHost, u->stream) ||
                  cudaStreamSynchronize(u->stream)))
        return 3;
    return tc_status(u);
}

int mg_unet_train_step(mg_unet *u, int B, int n, const double *rho, const double *phi_interp,
                       const double *resid, const double *phi_true, const double *frho, float lr, float wd, int update,
                       float *loss_out)
{
    if (!u || !frho || B > u->bmax || n < 8 || n > u->nmax || (n & (n - 1)))
        return 1;
    cudaStream_t s = u->stream;
    const int lg = ilog2(n);
    const int V0 = B << (3 * lg);
    if (cudaMemcpyAsync(u->frho, frho, B * sizeof(double), cudaMemcpyHostToDevice, s))
        return 3;
    int r = mg_unet_predict_dev(u, B, n, 0, rho, const_cast<double *>(phi_interp), resid, u->frho, 0, nullptr);
    if (r)
        return r;
    k_make_target<<<blocks_for(V0), kT, 0, s>>>(phi_true, phi_interp, u->scale, n, 1 << (3 * lg), B, u->tgt);
    k_fill<<<blocks_for(u->nparam), kT, 0, s>>>(u->grad, u->nparam, 0.f);
    k_fill<<<1, 32, 0, s>>>(u->loss, 1, 0.f);
    if (backward(u, B, lg))
        return 3;
    if (update) {
        u->step++;
        const float b1 = 0.9f, b2 = 0.999f;
        const float c1 = 1.f - std::pow(b1, (float)u->step), c2 = 1.f - std::pow(b2, (float)u->step);
        k_adamw<<<blocks_for(u->nparam), kT, 0, s>>>(u->p, u->grad, u->m, u->v, u->nparam, lr, b1, b2, 1e-8f, wd, c1, c2);
        u->packed = false;
    }
    float l = 0.f;
    if (cudaMemcpyAsync(&l, u->loss, sizeof(float), cudaMemcpyDeviceToHost, s) || cudaStreamSynchronize(s))
        return 3;
    if (loss_out)
        *loss_out = l;
    if (cudaGetLastError())
        return 3;
    return tc_status(u);
}

}  // extern "C"
