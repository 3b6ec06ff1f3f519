// mlp.cu -- the closure network on the tensor cores: 9 (or 8) inputs -> 64 -> 64 -> 1, SiLU,
// bfloat16 weights and matrix inputs, FP32 accumulation.  Forward (inference) and one Adam
// training step over a batch (mean squared error).
//
// The paper's conclusion conjectures that the collisional friction on the return current can be
// expressed through the local plasma state; this network is the library's reading of that
// closure (inputs: the coarse moments of pic_record_moments rows 0..8; output: nu_eff).
//
// Tiles of 128 samples; in inference a sample (row) per thread.  The two hidden
// layers are tcgen05 matrix products with M = 128 rows, N = 64, K = 16 (layer 1, inputs zero
// padded) and K = 64 (layer 2): the operands are staged in shared memory as bfloat16 in the
// no-swizzle K-major layout (8-row x 16-byte core matrices; LBO = stride between core matrices
// along K, SBO = stride between 8-row groups), one thread issues the MMAs, the accumulator lives
// in 64 TMEM columns and each warp reads its 32 rows back with tcgen05.ld.  Bias, SiLU and the
// 64 -> 1 output layer run on the CUDA cores.  Training adds the backward product
// delta1 = (delta2 W2) * silu'(z1) on the tensor cores (W2 transposed in shared memory) and
// the weight gradients, summed per CTA; a second kernel sums the CTA
// partials in a fixed order and applies Adam, so a training step is deterministic.
//
// Every wait on the MMA completion barrier is bounded: on timeout the kernel records an error
// flag (read by pic_mlp_status), waits once more (bounded) so that a late MMA does not write into
// TMEM that has been freed, frees its TMEM and returns; that call's outputs are undefined.
#include <cuda_bf16.h>

#include "pic_internal.cuh"

namespace pic {

constexpr int MLP_IN = 9, MLP_H = 64, MLP_KIN = 16;
constexpr int MLP_NPARAM = MLP_H * MLP_IN + MLP_H + MLP_H * MLP_H + MLP_H + MLP_H + 1;   // 4865
constexpr int OFF_W1 = 0, OFF_B1 = MLP_H * MLP_IN, OFF_W2 = OFF_B1 + MLP_H, OFF_B2 = OFF_W2 + MLP_H * MLP_H,
              OFF_W3 = OFF_B2 + MLP_H, OFF_B3 = OFF_W3 + MLP_H;
static_assert(OFF_B3 + 1 == MLP_NPARAM, "parameter layout");

__device__ int g_mlp_err;     // sticky: 1 = an MMA completion wait timed out

namespace {

constexpr int ROWS = 128;
constexpr long long WAIT_LIMIT = 1ll << 26;   // polls of the completion barrier (~seconds)

// ------------------------------------------------------------------ PTX helpers
__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor, no swizzle, K-major: start address, LBO (next core matrix
// along K), SBO (next 8-row group), descriptor version 1.
__device__ __forceinline__ unsigned long long mdesc(const void* p, unsigned lbo, unsigned sbo) {
    const unsigned long long a = smem_u32(p);
    return ((a >> 4) & 0x3FFFull) | ((unsigned long long)((lbo >> 4) & 0x3FFF) << 16) |
           ((unsigned long long)((sbo >> 4) & 0x3FFF) << 32) | (1ull << 46);
}

// Instruction descriptor of kind::f16: D F32, A and B BF16, both K-major, N = 64, M = 128.
constexpr unsigned IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((64u >> 3) << 17) | ((128u >> 4) << 24);

__device__ __forceinline__ void mma_bf16(unsigned tmem, unsigned long long a, unsigned long long b, int acc,
                                         unsigned idesc = IDESC) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n"
        ::"r"(tmem), "l"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void mma_commit(unsigned long long* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n"
                 ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool bar_try_wait(unsigned long long* bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait for the phase `parity` of the barrier; false after `limit` polls.
__device__ __forceinline__ bool bar_wait(unsigned long long* bar, unsigned parity, long long limit = WAIT_LIMIT) {
    for (long long i = 0; i < limit; ++i)
        if (bar_try_wait(bar, parity)) return true;
    return false;
}
// After a wait gave up: flag it, then wait once more (bounded) so that no committed MMA is
// still writing when the kernel frees its TMEM; if that wait gives up too the flag says so (2).
__device__ __forceinline__ void timed_out(unsigned long long* bar, unsigned parity) {
    const bool late = bar_wait(bar, parity);
    atomicMax(&g_mlp_err, late ? 1 : 2);
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

// 16 consecutive FP32 accumulator columns of this thread's row (TMEM lane = row).
__device__ __forceinline__ void tmem_ld16(unsigned taddr, float* v) {
    unsigned r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr) : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_ld4(unsigned taddr, float* v) {
    unsigned r[4];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(taddr) : "memory");
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory"); }

// Byte offset of element (row, k) of a K-major tile with KB core matrices per 8-row group.
template <int KB>
__device__ __forceinline__ int kmaj(int row, int k) {
    return (((row >> 3) * KB + (k >> 3)) << 7) + ((row & 7) << 4) + ((k & 7) << 1);
}
// Logistic sigmoid through sigma(z) = (1 + tanh(z / 2)) / 2: one special-function operation
// (tanh.approx, relative error ~2^-11, below the bfloat16 rounding of the hidden activations)
// instead of an exponential and a reciprocal.  With h = z / 2 and t = tanh(h), silu(z) = z sigma(z) =
// h (1 + t): factors of two apart the same operations, so the same rounding of the bfloat16
// activations.  Both the forward and the training kernels use these, so training optimises the
// function inference evaluates.
__device__ __forceinline__ float tanh_approx(float x) {
    float y;
    asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// Two units at once in packed FP32 operations: h = acc / 2 + hb (hb: half the bias), t = tanh(h).
__device__ __forceinline__ float2 half_z2(float a0, float a1, float2 hb) {
    return __ffma2_rn(make_float2(a0, a1), make_float2(0.5f, 0.5f), hb);
}
__device__ __forceinline__ float2 tanh2(float2 h) { return make_float2(tanh_approx(h.x), tanh_approx(h.y)); }
__device__ __forceinline__ float2 silu2(float2 h, float2 t) { return __fmul2_rn(h, __fadd2_rn(t, make_float2(1.f, 1.f))); }
// silu'(z) = sigma (1 + z (1 - sigma)) = (1 + t) / 2 (1 + h (1 - t))
__device__ __forceinline__ float dsilu(float h, float t) {
    return fmaf(0.5f, t, 0.5f) * fmaf(h, 1.f - t, 1.f);
}

// Eight consecutive values of one row into a K-major tile as one 16-byte store (k0 % 8 == 0).
template <int KB>
__device__ __forceinline__ void put8_bf16(unsigned char* tile, int row, int k0, const float* v) {
    uint4 q;
    unsigned* w = reinterpret_cast<unsigned*>(&q);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __nv_bfloat162 b = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
        w[i] = *reinterpret_cast<const unsigned*>(&b);
    }
    *reinterpret_cast<uint4*>(tile + kmaj<KB>(row, k0)) = q;
}

struct MlpArgs {
    const float* params;   // [MLP_NPARAM] FP32 master parameters
    MlpNorm norm;
    const float* x;        // feature-major: x[j * ldx + i]
    long long ldx;
    long long n;
    const float* target;   // training: [n]
    float* y;              // inference: [n]
    float* part;           // training: [gridDim.x][MLP_NPARAM + 1] gradient and loss partials
};

// Parameters -> shared memory (bfloat16 operand tiles and FP32 vectors); zero the padding.
template <class S>
__device__ void load_params(S& s, const float* p, unsigned char* w2t) {
    const int NT = blockDim.x;
    // eight values of a row per thread and 16-byte store
    for (int i = threadIdx.x; i < MLP_H * MLP_KIN / 8; i += NT) {
        const int n = i >> 1, k0 = (i & 1) * 8;
        float v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = k0 + q < MLP_IN ? p[OFF_W1 + n * MLP_IN + k0 + q] : 0.f;
        put8_bf16<2>(s.W1, n, k0, v);
    }
    for (int i = threadIdx.x; i < MLP_H * MLP_H / 8; i += NT) {
        const int n = i >> 3, k0 = (i & 7) * 8;
        float v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = p[OFF_W2 + n * MLP_H + k0 + q];
        put8_bf16<8>(s.W2, n, k0, v);
    }
    for (int i = threadIdx.x; w2t && i < MLP_H * MLP_H / 8; i += NT) {
        const int k = i & (MLP_H - 1), n0 = (i / MLP_H) * 8;
        float v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = p[OFF_W2 + (n0 + q) * MLP_H + k];
        put8_bf16<8>(w2t, k, n0, v);
    }
    for (int i = threadIdx.x; i < MLP_H; i += NT) {
        s.hb1[i] = 0.5f * p[OFF_B1 + i];
        s.hb2[i] = 0.5f * p[OFF_B2 + i];
        s.w3[i] = p[OFF_W3 + i];
    }
    if (threadIdx.x == 0) s.b3 = p[OFF_B3];
}

// TMEM (NCOL columns) and the completion barrier; every thread gets the TMEM address.
template <int NCOL = 64, class S>
__device__ void setup(S& s) {
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n"
                     ::"r"(smem_u32(&s.tmem)), "r"(NCOL) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&s.bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
}

template <int NCOL = 64, class S>
__device__ void teardown(S& s) {
    fence_before();
    __syncthreads();
    fence_after();
    if (threadIdx.x < 32)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(s.tmem), "r"(NCOL) : "memory");
}

// ------------------------------------------------------------------ inference
// 256 threads: two groups of 4 warps, each with its own tiles of 128 samples (thread = sample row),
// accumulator (TMEM columns 64 h .. 64 h + 63 of 128), completion barrier and named barrier, so that
// one group's epilogue runs while the other (and the other 3 CTAs of the SM) waits for its products;
// the next tile's inputs are loaded meanwhile.  2^20 samples: 55.5 us with both groups in step and
// each unit's operations one by one, 47.2 with packed pairs of units and 64 registers, 45.9 so; it
// executes 24M warp instructions and is bound by the latency of a tile's two products and TMEM reads
// (the special-function unit, 128 operations per sample, is busy 30%).
constexpr int FWD_NT = 256, FWD_SUB = 2;

struct __align__(1024) MlpFwdSmem {
    unsigned char X[FWD_SUB][ROWS * MLP_KIN * 2];     // stride ROWS * 2 * 16 bytes (KB = 2)
    unsigned char H[FWD_SUB][ROWS * MLP_H * 2];       // stride ROWS * 8 * 16 bytes (KB = 8)
    unsigned char W1[MLP_H * MLP_KIN * 2];
    unsigned char W2[MLP_H * MLP_H * 2];
    alignas(16) float hb1[MLP_H], hb2[MLP_H], w3[MLP_H];   // half biases, output weights
    float b3;
    unsigned long long bar, bar1;                     // of group 0 and of group 1
    unsigned tmem;
};

// Barrier of group h (128 threads); the conjunction of ok over it.
__device__ __forceinline__ void group_sync(int h) { asm volatile("bar.sync %0, 128;\n" ::"r"(h + 1) : "memory"); }
__device__ __forceinline__ bool group_and(int h, bool ok) {
    unsigned all;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.and.pred q, %2, 128, p;\n\t"
                 "selp.u32 %0, 1, 0, q;\n\t}\n" : "=r"(all) : "r"((unsigned)ok), "r"(h + 1) : "memory");
    return all != 0;
}

// Group h's product (KB core matrices per row group) of the tile A with B; false (all its threads)
// on timeout.
template <int KB>
__device__ bool group_product(MlpFwdSmem& s, int h, const unsigned char* A, const unsigned char* B, unsigned& phase) {
    unsigned long long* bar = h ? &s.bar1 : &s.bar;
    fence_async_smem();
    fence_before();
    group_sync(h);
    fence_after();
    if ((threadIdx.x & (ROWS - 1)) == 0) {
        constexpr unsigned LBO = 128, SBO = 128 * KB;
#pragma unroll
        for (int ks = 0; ks < KB / 2; ++ks)
            mma_bf16(s.tmem + MLP_H * h, mdesc(A + ks * 256, LBO, SBO), mdesc(B + ks * 256, LBO, SBO), ks > 0);
        mma_commit(bar);
    }
    const bool ok = bar_wait(bar, phase);
    if (!ok) timed_out(bar, phase);
    phase ^= 1u;
    fence_after();
    return group_and(h, ok);
}

__device__ __forceinline__ void load_x(const MlpArgs& m, long long i, float x[MLP_IN]) {
#pragma unroll
    for (int j = 0; j < MLP_IN; ++j) x[j] = (i < m.n && j < m.norm.nin) ? __ldg(m.x + j * m.ldx + i) : 0.f;
}

__global__ void __launch_bounds__(FWD_NT, 4) mlp_forward_kernel(const MlpArgs m) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    MlpFwdSmem& s = *reinterpret_cast<MlpFwdSmem*>(smem_raw);
    load_params(s, m.params, nullptr);
    if (threadIdx.x == 0) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&s.bar1)) : "memory");
    setup<FWD_SUB * MLP_H>(s);
    const int h = threadIdx.x >> 7, r = threadIdx.x & (ROWS - 1);
    const unsigned taddr = s.tmem + ((unsigned)(r & ~31) << 16) + MLP_H * h;
    unsigned phase = 0;
    const long long ntiles = (m.n + ROWS - 1) / ROWS, step = (long long)gridDim.x * FWD_SUB;
    float xr[MLP_IN];
    load_x(m, ((long long)blockIdx.x * FWD_SUB + h) * ROWS + r, xr);
    for (long long t = (long long)blockIdx.x * FWD_SUB + h; t < ntiles; t += step) {
        const long long i = t * ROWS + r;
        float xs[16];
#pragma unroll
        for (int j = 0; j < 16; ++j)
            xs[j] = j < MLP_IN && j < m.norm.nin ? (xr[j] - m.norm.mu[j]) * m.norm.inv_sigma[j] : 0.f;
        put8_bf16<2>(s.X[h], r, 0, xs);
        put8_bf16<2>(s.X[h], r, 8, xs + 8);
        load_x(m, i + step * ROWS, xr);      // next tile, in flight meanwhile
        if (!group_product<2>(s, h, s.X[h], s.W1, phase)) break;
        // 16 units at a time, so that 4 CTAs fit an SM's registers
#pragma unroll
        for (int c = 0; c < MLP_H; c += 16) {
            float z[16];
            tmem_ld16(taddr + c, z);
            tmem_ld_wait();
#pragma unroll
            for (int q = 0; q < 16; q += 4) {
                const float4 hb = *reinterpret_cast<const float4*>(s.hb1 + c + q);
                const float2 h0 = half_z2(z[q], z[q + 1], make_float2(hb.x, hb.y));
                const float2 h1 = half_z2(z[q + 2], z[q + 3], make_float2(hb.z, hb.w));
                const float2 v0 = silu2(h0, tanh2(h0)), v1 = silu2(h1, tanh2(h1));
                z[q] = v0.x;
                z[q + 1] = v0.y;
                z[q + 2] = v1.x;
                z[q + 3] = v1.y;
            }
            put8_bf16<8>(s.H[h], r, c, z);
            put8_bf16<8>(s.H[h], r, c + 8, z + 8);
        }
        if (!group_product<8>(s, h, s.H[h], s.W2, phase)) break;
        float2 y2 = make_float2(0.f, 0.f);
#pragma unroll
        for (int c = 0; c < MLP_H; c += 16) {
            float z[16];
            tmem_ld16(taddr + c, z);
            tmem_ld_wait();
#pragma unroll
            for (int q = 0; q < 16; q += 4) {
                const float4 hb = *reinterpret_cast<const float4*>(s.hb2 + c + q);
                const float4 w = *reinterpret_cast<const float4*>(s.w3 + c + q);
                const float2 h0 = half_z2(z[q], z[q + 1], make_float2(hb.x, hb.y));
                const float2 h1 = half_z2(z[q + 2], z[q + 3], make_float2(hb.z, hb.w));
                y2 = __ffma2_rn(make_float2(w.x, w.y), silu2(h0, tanh2(h0)), y2);
                y2 = __ffma2_rn(make_float2(w.z, w.w), silu2(h1, tanh2(h1)), y2);
            }
        }
        const float y = s.b3 + (y2.x + y2.y);
        if (i < m.n) m.y[i] = y;
    }
    teardown<FWD_SUB * MLP_H>(s);
}

// ------------------------------------------------------------------ training
// One CTA of 512 threads per SM, tiles of 128 samples, four threads per sample (16 of the 64 units
// each).  Per tile the two hidden products and the backward product run on the tensor cores as in
// inference, and so do the weight gradients: with Q the matrix of the rows [delta2 | delta1] (128
// samples x 128 units) and Z that of [h1 | xn, 1] (128 samples x 80),
//   G = Q^T Z   (M = 128, N = 80, K = 128 samples, FP32 in TMEM)
// holds dW2 = delta2^T h1 and db2 = delta2^T 1 in its upper 64 rows and dW1, db1 in the lower ones (the
// remaining products, delta1^T h1 and delta2^T xn, are not used).  Z is bfloat16 already (the operands
// of the forward products, plus a column of ones); Q keeps its FP32 values as the sum of three
// bfloat16 parts (8 + 8 + 8 bits of mantissa), so G is three products, the smallest part first.  The
// tensor cores round their sums towards zero, a shrinkage that does not average out: so the tile's
// samples are summed in four groups of 32 (two products of K = 16 per part) in TMEM columns of their
// own, and the groups' sums are added, rounded to nearest, to an FP32 copy in shared memory.  Error
// against FP64 sums of the same factors, 1000 / 403938 samples: FP32 sums on the CUDA cores 8.3e-8 /
// 1.9e-7, one group per tile 1.5e-7 / 2.3e-7, four 7e-8 / 7e-8 (left in TMEM over a call's tiles, 4e-6).
// Both operands are the tiles
// as they were written row by row for the K-major products: read as MN-major, their 8 x 16-byte
// core matrices are the same bytes with the roles of the strides exchanged.  G's products run while
// the next tile's inputs are staged: the wait for that tile's first product, whose commit comes after
// them from the same thread, covers them.  The output layer's gradient (dy h2, FP32) is summed over a
// warp's 32 samples by exchanges that halve the columns a lane carries.
// 403938 samples: 656 -> 114 us (109 with one group per tile); the gradient sums on the CUDA cores had taken most of it.
constexpr int TR_NT = 512, TPR = 4, CPT = MLP_H / TPR;      // threads, threads per sample, units of one
constexpr int QB = 16, ZB = 10;                             // 8-column groups of the Q and Z tiles
constexpr int ZN = 8 * ZB, ONE = MLP_H + MLP_IN;            // Z's columns; the column of ones
constexpr int GG = 4;                                       // groups of samples of G
constexpr int TR_TMEM = 512, TR_G = MLP_H;                  // allocated columns; first column of G
static_assert(TR_G + GG * ZN <= TR_TMEM && (ROWS / 16) % GG == 0, "TMEM columns of G");

struct __align__(1024) MlpTrainSmem {
    unsigned char Q[3][ROWS * QB * 16];       // parts of [delta2 | delta1]; Q[0] is also the backward A
    unsigned char Z[2][ROWS * ZB * 16];       // [h1 | xn, 1, 0]: layer-2 A and layer-1 A; two tiles in turn
    unsigned char W1[MLP_H * MLP_KIN * 2];
    unsigned char W2[MLP_H * MLP_H * 2];
    unsigned char W2T[MLP_H * MLP_H * 2];     // backward B: W2T[k][n] = W2[n][k]
    alignas(16) float hb1[MLP_H], hb2[MLP_H], w3[MLP_H];   // half biases, output weights
    float b3;
    float G[ROWS][ZN + 1];                    // sum of the tiles' G (row = unit of Q)
    float yp[TPR][ROWS];                      // parts of the output layer's sum
    float red[TR_NT / 32][CPT + 2];           // closing sums of the output layer's gradient
    unsigned long long bar, gbar;             // forward and backward products; G
    unsigned tmem;
};

// Descriptor of kind::f16 for G: A and B MN-major (bits 15, 16), N = 80, M = 128.
constexpr unsigned IDESC_G = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((ZN >> 3) << 17) | ((128u >> 4) << 24);

// One hidden product (KS steps of K = 16) of the tile A (8-row groups sboA bytes apart) with the
// weight tile B (KB core matrices per group); false (all threads) if it did not complete in time.
template <int KS, int KB>
__device__ bool train_product(MlpTrainSmem& s, const unsigned char* A, unsigned sboA, const unsigned char* B,
                              unsigned& phase) {
    fence_async_smem();
    fence_before();
    __syncthreads();
    fence_after();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int ks = 0; ks < KS; ++ks)
            mma_bf16(s.tmem, mdesc(A + ks * 256, 128, sboA), mdesc(B + ks * 256, 128, 128 * KB), ks > 0);
        mma_commit(&s.bar);
    }
    const bool ok = bar_wait(&s.bar, phase);
    if (!ok) timed_out(&s.bar, phase);
    phase ^= 1u;
    fence_after();
    return __syncthreads_and(ok);
}

// v as hi + mid + lo, each bfloat16 (the remainders are exact), 8 columns at k0 of row r of the
// three Q tiles.
__device__ __forceinline__ void put8_parts(MlpTrainSmem& s, int r, int k0, const float* v) {
    float hi[8], mid[8], lo[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        hi[i] = __bfloat162float(__float2bfloat16_rn(v[i]));
        const float a = __fsub_rn(v[i], hi[i]);
        mid[i] = __bfloat162float(__float2bfloat16_rn(a));
        lo[i] = __fsub_rn(a, mid[i]);
    }
    put8_bf16<QB>(s.Q[0], r, k0, hi);
    put8_bf16<QB>(s.Q[1], r, k0, mid);
    put8_bf16<QB>(s.Q[2], r, k0, lo);
}

__global__ void __launch_bounds__(TR_NT) mlp_train_kernel(const MlpArgs m) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    MlpTrainSmem& s = *reinterpret_cast<MlpTrainSmem*>(smem_raw);
    load_params(s, m.params, s.W2T);
    if (threadIdx.x == 0) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&s.gbar)) : "memory");
    setup<TR_TMEM>(s);
    const int q = threadIdx.x >> 7, r = threadIdx.x & (ROWS - 1), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c0 = q * CPT;
    const unsigned taddr = s.tmem + ((unsigned)(r & ~31) << 16);
    const long long ntiles = (m.n + ROWS - 1) / ROWS;
    const float inv_n = 1.f / (float)m.n;
    unsigned phase = 0, gphase = 0;
    bool ok = true, pending = false;     // pending: G products of the last tile not waited for
    float gw3 = 0.f, gb3 = 0.f, loss = 0.f;
    float xr[MLP_IN], tr = 0.f;
    auto load = [&](long long i) {
        if (q == 0) load_x(m, i, xr);
        tr = i < m.n ? __ldg(m.target + i) : 0.f;
    };
    auto wait_g = [&]() {
        if (!pending) return;
        const bool w = bar_wait(&s.gbar, gphase);
        if (!w) timed_out(&s.gbar, gphase);
        gphase ^= 1u;
        pending = false;
        fence_after();
        ok = __syncthreads_and(w);
        if (!ok) return;
        // this thread's 20 columns of G, over the groups
        float g[20];
#pragma unroll
        for (int c = 0; c < GG; ++c) {
            float gc[20];
            tmem_ld16(taddr + TR_G + c * ZN + q * 16, gc);
            tmem_ld4(taddr + TR_G + c * ZN + MLP_H + q * 4, gc + 16);
            tmem_ld_wait();
#pragma unroll
            for (int k = 0; k < 20; ++k) g[k] = c == 0 ? gc[k] : g[k] + gc[k];
        }
#pragma unroll
        for (int k = 0; k < 20; ++k) s.G[r][k < 16 ? q * 16 + k : MLP_H + q * 4 + k - 16] += g[k];
    };
    for (int i = threadIdx.x; i < ROWS * (ZN + 1); i += TR_NT) (&s.G[0][0])[i] = 0.f;
    load((long long)blockIdx.x * ROWS + r);
    int tile = 0;
    for (long long t = blockIdx.x; t < ntiles; t += gridDim.x, ++tile) {
        const bool live = t * ROWS + r < m.n;
        const float target = tr;
        unsigned char* Z = s.Z[tile & 1];
        if (q == 0) {
            float xs[16];
#pragma unroll
            for (int j = 0; j < 16; ++j)
                xs[j] = j == MLP_IN ? 1.f
                                    : (live && j < MLP_IN && j < m.norm.nin ? (xr[j] - m.norm.mu[j]) * m.norm.inv_sigma[j] : 0.f);
            put8_bf16<ZB>(Z, r, MLP_H, xs);
            put8_bf16<ZB>(Z, r, MLP_H + 8, xs + 8);
        }
        load((t + gridDim.x) * ROWS + r);       // the next tile's, in flight meanwhile
        if (!(ok = train_product<1, 2>(s, Z + 128 * (MLP_H / 8), 128 * ZB, s.W1, phase))) break;
        float z1[CPT], v[CPT];
        tmem_ld16(taddr + c0, z1);
        tmem_ld_wait();
#pragma unroll
        for (int k = 0; k < CPT; k += 2) {
            const float2 h = half_z2(z1[k], z1[k + 1], *reinterpret_cast<const float2*>(s.hb1 + c0 + k));
            const float2 t = tanh2(h), f = silu2(h, t);
            v[k] = f.x;
            v[k + 1] = f.y;
            z1[k] = dsilu(h.x, t.x);                      // silu'(z1)
            z1[k + 1] = dsilu(h.y, t.y);
        }
        put8_bf16<ZB>(Z, r, c0, v);
        put8_bf16<ZB>(Z, r, c0 + 8, v + 8);
        if (!(ok = train_product<4, 8>(s, Z, 128 * ZB, s.W2, phase))) break;
        float z2[CPT];
        tmem_ld16(taddr + c0, z2);
        tmem_ld_wait();
        float y = 0.f;
#pragma unroll
        for (int k = 0; k < CPT; k += 2) {
            const float2 h = half_z2(z2[k], z2[k + 1], *reinterpret_cast<const float2*>(s.hb2 + c0 + k));
            const float2 t = tanh2(h), f = silu2(h, t);
            v[k] = f.x;                                   // h2
            v[k + 1] = f.y;
            y = fmaf(s.w3[c0 + k], f.x, y);
            y = fmaf(s.w3[c0 + k + 1], f.y, y);
            z2[k] = dsilu(h.x, t.x);                      // silu'(z2)
            z2[k + 1] = dsilu(h.y, t.y);
        }
        s.yp[q][r] = y;
        __syncthreads();
        y = s.b3 + ((s.yp[0][r] + s.yp[1][r]) + (s.yp[2][r] + s.yp[3][r]));
        const float res = live ? y - target : 0.f;
        const float dy = 2.f * res * inv_n;
        if (q == 0) {
            gb3 += dy;
            loss = fmaf(res, res, loss);
        }
        // delta2, and the output layer's gradient dy h2 summed over the warp's samples
#pragma unroll
        for (int k = 0; k < CPT; ++k) {
            z2[k] *= dy * s.w3[c0 + k];
            v[k] *= dy;
        }
#pragma unroll
        for (int n = CPT / 2; n > 0; n >>= 1) {
            const bool up = lane & (2 * n);
#pragma unroll
            for (int k = 0; k < n; ++k) {
                const float mine = up ? v[k + n] : v[k], other = up ? v[k] : v[k + n];
                v[k] = mine + __shfl_xor_sync(0xffffffffu, other, 2 * n);
            }
        }
        gw3 += v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);   // column c0 + lane / 2
        wait_g();                                // the previous tile's Q is free
        if (!ok) break;
        put8_parts(s, r, c0, z2);
        put8_parts(s, r, c0 + 8, z2 + 8);
        if (!(ok = train_product<4, 8>(s, s.Q[0], 128 * QB, s.W2T, phase))) break;
        tmem_ld16(taddr + c0, v);
        tmem_ld_wait();
#pragma unroll
        for (int k = 0; k < CPT; ++k) v[k] *= z1[k];          // delta1
        put8_parts(s, r, MLP_H + c0, v);
        put8_parts(s, r, MLP_H + c0 + 8, v + 8);
        fence_async_smem();
        fence_before();
        __syncthreads();
        fence_after();
        if (threadIdx.x == 0) {
#pragma unroll 1
            for (int p = 2; p >= 0; --p)
#pragma unroll
                for (int ks = 0; ks < ROWS / 16; ++ks)
                    mma_bf16(s.tmem + TR_G + ks / (ROWS / 16 / GG) * ZN, mdesc(s.Q[p] + ks * 2 * 128 * QB, 128 * QB, 128),
                             mdesc(Z + ks * 2 * 128 * ZB, 128 * ZB, 128), p < 2 || ks % (ROWS / 16 / GG) > 0, IDESC_G);
            mma_commit(&s.gbar);
        }
        pending = true;
    }
    wait_g();
    float* out = m.part + (size_t)blockIdx.x * (MLP_NPARAM + 1);
    teardown<TR_TMEM>(s);
    for (int i = threadIdx.x; i < MLP_H * MLP_H; i += TR_NT) out[OFF_W2 + i] = s.G[i / MLP_H][i % MLP_H];
    for (int i = threadIdx.x; i < MLP_H * MLP_IN; i += TR_NT)
        out[OFF_W1 + i] = s.G[MLP_H + i / MLP_IN][MLP_H + i % MLP_IN];
    for (int i = threadIdx.x; i < MLP_H; i += TR_NT) {
        out[OFF_B2 + i] = s.G[i][ONE];
        out[OFF_B1 + i] = s.G[MLP_H + i][ONE];
    }
    // output layer: sums over the warps of a unit group (32 samples each), in a fixed order
    for (int o = 16; o > 0; o >>= 1) {
        gb3 += __shfl_xor_sync(0xffffffffu, gb3, o);
        loss += __shfl_xor_sync(0xffffffffu, loss, o);
    }
    if ((lane & 1) == 0) s.red[warp][lane >> 1] = gw3;
    if (lane == 0) {
        s.red[warp][CPT] = gb3;
        s.red[warp][CPT + 1] = loss;
    }
    __syncthreads();
    if (threadIdx.x < MLP_H) {
        const int w0 = (threadIdx.x / CPT) * (ROWS / 32), k = threadIdx.x % CPT;
        out[OFF_W3 + threadIdx.x] = (s.red[w0][k] + s.red[w0 + 1][k]) + (s.red[w0 + 2][k] + s.red[w0 + 3][k]);
    }
    if (threadIdx.x < 2)
        out[threadIdx.x ? MLP_NPARAM : OFF_B3] = (s.red[0][CPT + threadIdx.x] + s.red[1][CPT + threadIdx.x]) +
                                                 (s.red[2][CPT + threadIdx.x] + s.red[3][CPT + threadIdx.x]);
}

// Sum the CTA partials and take one Adam step (Kingma & Ba 2015, Algorithm 1).  Eight sums in turn, then
// a tree, in a fixed order: 152 partials added one after the other were most of the gradient's rounding
// error (403938 samples: 1.9e-7 -> 7e-8).
constexpr int MLP_TRAIN_GRID = 152;
static_assert(MLP_TRAIN_GRID % 8 == 0, "sums of mlp_adam_kernel");
__global__ void mlp_adam_kernel(float* params, float* am, float* av, const float* part, int t,
                                float lr, float beta1, float beta2, float eps, long long n, float* loss) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i <= MLP_NPARAM; i += gridDim.x * blockDim.x) {
        float p[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int c = 0; c < MLP_TRAIN_GRID; c += 8)
#pragma unroll
            for (int k = 0; k < 8; ++k) p[k] += part[(size_t)(c + k) * (MLP_NPARAM + 1) + i];
        const float g = ((p[0] + p[1]) + (p[2] + p[3])) + ((p[4] + p[5]) + (p[6] + p[7]));
        if (i == MLP_NPARAM) {
            if (loss) *loss = g / (float)n;
            continue;
        }
        const float mi = beta1 * am[i] + (1.f - beta1) * g;
        const float vi = beta2 * av[i] + (1.f - beta2) * g * g;
        am[i] = mi;
        av[i] = vi;
        const float mh = mi / (1.f - powf(beta1, (float)t));
        const float vh = vi / (1.f - powf(beta2, (float)t));
        params[i] -= lr * mh / (sqrtf(vh) + eps);
    }
}


}  // namespace

size_t mlp_train_scratch_bytes() { return (size_t)MLP_TRAIN_GRID * (MLP_NPARAM + 1) * sizeof(float); }

cudaError_t launch_mlp_forward(const float* params, const MlpNorm& norm, const float* x, long long ldx, long long n,
                               float* y, cudaStream_t s) {
    cudaError_t e = smem_attr_once((const void*)mlp_forward_kernel, (int)sizeof(MlpFwdSmem));
    if (e != cudaSuccess) return e;
    if (n <= 0) return cudaSuccess;
    MlpArgs m{params, norm, x, ldx, n, nullptr, y, nullptr};
    const long long tiles = (n + FWD_SUB * ROWS - 1) / (FWD_SUB * ROWS);
    const int grid = (int)(tiles < 152LL * 4 ? tiles : 152LL * 4);
    mlp_forward_kernel<<<grid, FWD_NT, sizeof(MlpFwdSmem), s>>>(m);
    return cudaGetLastError();
}

cudaError_t launch_mlp_train(float* params, float* am, float* av, int t, float lr, const MlpNorm& norm,
                             const float* x, long long ldx, const float* target, long long n, float* loss,
                             void* scratch, cudaStream_t s) {
    cudaError_t e = smem_attr_once((const void*)mlp_train_kernel, (int)sizeof(MlpTrainSmem));
    if (e != cudaSuccess) return e;
    float* part = static_cast<float*>(scratch);
    MlpArgs m{params, norm, x, ldx, n, target, nullptr, part};
    // a fixed grid: CTA c takes tiles c, c + grid, ... so the partials and their sum are fixed
    mlp_train_kernel<<<MLP_TRAIN_GRID, TR_NT, sizeof(MlpTrainSmem), s>>>(m);
    mlp_adam_kernel<<<20, 256, 0, s>>>(params, am, av, part, t, lr, 0.9f, 0.999f, 1e-8f, n, loss);
    return cudaGetLastError();
}

// Test hook: one CTA waits on a barrier that nothing arrives on (no MMA is issued), gives up
// after `polls` polls and sets the flag as a timed-out network kernel does.
__global__ void mlp_wait_test_kernel(long long polls) {
    __shared__ unsigned long long bar;
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0 && !bar_wait(&bar, 0, polls)) atomicMax(&g_mlp_err, 1);
}

cudaError_t launch_mlp_wait_test(long long polls, cudaStream_t s) {
    mlp_wait_test_kernel<<<1, 32, 0, s>>>(polls);
    return cudaGetLastError();
}

cudaError_t mlp_status(int* err, bool clear) {
    cudaError_t e = cudaMemcpyFromSymbol(err, g_mlp_err, sizeof(int));
    if (e == cudaSuccess && clear && *err) {
        const int z = 0;
        e = cudaMemcpyToSymbol(g_mlp_err, &z, sizeof(int));
    }
    return e;
}

cudaError_t preload_mlp() {
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, mlp_forward_kernel);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, mlp_train_kernel);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, mlp_adam_kernel);
    return e;
}

}  // namespace pic
