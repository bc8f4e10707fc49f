// gemm_tc.cu -- BF16 x BF16 -> FP32 GEMM on the fifth-generation tensor cores
// (tcgen05.mma, accumulators in tensor memory), fed by TMA.  It computes the
// products of the learned initialiser's network (mlp.cu) where the shapes
// allow (at least 128 x 128 x 64, 16-byte aligned rows).
//
//   C[M][N] (FP32, row stride ldc) = sum_k A(m, k) B(n, k).  Each operand is
//   stored either K-contiguous (A [M][K], B [N][K]) or K-strided (A [K][M],
//   B [K][N]); both forms feed the tensor cores straight from memory (K-major
//   or MN-major shared-memory tiles), so no operand is transposed first.  (A
//   K-strided with B K-contiguous, which no product of the network has, is left out.)
//
// One CTA computes one 128 x BN tile of C with 4 warps:
//   warp 0, one lane: TMA producer.  Each k-step of 64 elements loads a
//     128 x 64 tile of A and a BN x 64 tile of B (128-byte rows, 128-byte
//     swizzle) into one of `stages` shared-memory stages, arriving on the
//     stage's "full" mbarrier with the transferred byte count;
//   warp 1, one lane: MMA issuer.  Per k-step, four tcgen05.mma of
//     M = 128, N = BN, K = 16 (kind::f16, BF16 operands, FP32 accumulator in
//     BN tensor-memory columns), then tcgen05.commit onto the stage's
//     "empty" mbarrier, which hands the stage back to the producer when the
//     MMAs that read it are done; after the last k-step a commit onto the
//     "done" mbarrier;
//   all 4 warps: epilogue.  Warp w reads tensor-memory lanes 32w .. 32w + 31
//     (rows of the tile) with tcgen05.ld, 32 columns at a time, turns the
//     block around in shared memory (the stages are free by then) and runs
//     the network's elementwise step on whole 128-byte row segments: bias and
//     GELU, GELU's derivative, or Adam's update of the weights whose gradient
//     the tile is (gemm_epilogue in internal.h).  As separate kernels these
//     steps read and wrote every product once more.
// BN and the number of stages follow the shape (plan() below).  Tensor memory
// (BN columns, at least 32) is allocated and freed by warp 0.  Out-of-range
// rows and the K tail are zero-filled by TMA.  Every mbarrier wait is
// bounded: after kSpinLimit polls the waiting thread raises *err and stops
// issuing work (the other role's next wait then runs out too), and the CTA
// waits (bounded again) for the MMAs and loads it issued, frees its tensor
// memory and returns; the caller reads the flag.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <mutex>

#include "internal.h"
#include "mlp_math.cuh"
#include "tmr.h"

namespace tmr {

namespace {

constexpr int kBM = 128, kBK = 64, kMaxStages = 10;
constexpr int kTileA = kBM * kBK * 2;  // bytes per stage
__host__ __device__ constexpr int tile_b(int bn) { return bn * kBK * 2; }
constexpr long long kSpinLimit = 1LL << 22;  // polls of a barrier wait (about 0.1 - 1 s)
constexpr int kStageBytes = 200 * 1024;      // of all stages together, at most
constexpr size_t smem_bytes(int bn, int stages)
{
    return 1024 /*alignment slack*/ + (size_t)stages * (kTileA + tile_b(bn)) + 256;
}
// the most a plan of this tile width asks for
constexpr size_t smem_most(int bn)
{
    const int st = kStageBytes / (kTileA + tile_b(bn));
    return smem_bytes(bn, st < kMaxStages ? st : kMaxStages);
}

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// One lane of a converged warp (the same one each time).  The compiler knows
// that a branch on it is taken by a single thread, which tcgen05 and TMA
// instructions, whose operands are warp-uniform, need; behind lane == 0 it
// emits code for any set of lanes.
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile(
        "{\n\t.reg .pred e;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, e;\n\t}"
        : "=r"(p));
    return p != 0;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// Wait until the phase with parity `parity` of the barrier has completed, at
// most kSpinLimit polls (test_wait does not block; after the first 1024 polls
// each one is followed by a 64 ns sleep); false on timeout.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity)
{
    for (long long i = 0; i < kSpinLimit; i++) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
        if (i >= 1024) __nanosleep(64);
    }
    return false;
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

// Shared-memory matrix descriptor of a K-major tile with 128-byte rows in the
// 128-byte swizzle layout: 8-row groups 1024 bytes apart (stride byte offset),
// descriptor version 1, swizzle mode 2 (128 B).  The leading byte offset is
// not used by this layout (set to 16 bytes).
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFF);
    d |= (uint64_t)1 << 16;              // leading byte offset >> 4
    d |= (uint64_t)(1024 >> 4) << 32;    // stride byte offset >> 4
    d |= (uint64_t)1 << 46;              // version
    d |= (uint64_t)2 << 61;              // 128-byte swizzle
    return d;
}

// The same for an MN-major tile (K-strided operand): TMA boxes of 64 k-rows x
// 64 elements (128 bytes, 128-byte swizzle), one after the other along M or
// N.  8-row groups along K are 1024 bytes apart (stride byte offset), boxes
// 8192 bytes (leading byte offset).
__device__ __forceinline__ uint64_t sw128_desc_mn(uint32_t saddr)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFF);
    d |= (uint64_t)(8192 >> 4) << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// Instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, each
// K-major (0) or MN-major (1), N = bn, M = kBM.
__host__ __device__ constexpr uint32_t idesc(int bn, bool mn_a, bool mn_b)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((mn_a ? 1u : 0u) << 15) | ((mn_b ? 1u : 0u) << 16) |
           ((uint32_t)(bn >> 3) << 17) | ((uint32_t)(kBM >> 4) << 24);
}

__device__ __forceinline__ void umma_f16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}

__device__ __forceinline__ void umma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}

// Four consecutive columns of a row as one 16-byte access where the matrices
// allow it (V), else one by one up to n.
template <bool V>
__device__ __forceinline__ float4 ld4(const float *p, int n)
{
    if constexpr (V) return *reinterpret_cast<const float4 *>(p);
    else return make_float4(n > 0 ? p[0] : 0.f, n > 1 ? p[1] : 0.f, n > 2 ? p[2] : 0.f, n > 3 ? p[3] : 0.f);
}
template <bool V>
__device__ __forceinline__ void st4(float *p, float4 x, int n)
{
    if constexpr (V) {
        *reinterpret_cast<float4 *>(p) = x;
    } else {
        if (n > 0) p[0] = x.x;
        if (n > 1) p[1] = x.y;
        if (n > 2) p[2] = x.z;
        if (n > 3) p[3] = x.w;
    }
}
template <bool V>
__device__ __forceinline__ void st4(__nv_bfloat16 *p, float4 x, int n)
{
    if constexpr (V) {
        const __nv_bfloat162 lo = __floats2bfloat162_rn(x.x, x.y), hi = __floats2bfloat162_rn(x.z, x.w);
        *reinterpret_cast<uint2 *>(p) =
            make_uint2(*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi));
    } else {
        if (n > 0) p[0] = __float2bfloat16(x.x);
        if (n > 1) p[1] = __float2bfloat16(x.y);
        if (n > 2) p[2] = __float2bfloat16(x.z);
        if (n > 3) p[3] = __float2bfloat16(x.w);
    }
}

// The elementwise step on a warp's 32 x 32 block of products: lane (r, c) takes
// the four columns from 4 c of rows r, r + 4, ...  Four rows' loads (12 of 16
// bytes for Adam) are in flight together.  blk: the block in shared memory;
// row0, col: the block's first row and this lane's first column.
template <bool V>
__device__ __forceinline__ void epilogue_block(const GemmEpilogue &E, const float (*blk)[33], int row0, int col, int M,
                                               int N, int ldc)
{
    const int lane = threadIdx.x & 31, c = 4 * (lane & 7);
    const int n = N - col;  // columns left (V: at least 4 or none)
    if (n <= 0) return;
    float4 bias = make_float4(0.f, 0.f, 0.f, 0.f);
    if (E.kind == GEMM_BIAS || E.kind == GEMM_BIAS_GELU) bias = ld4<V>(E.bias + col, n);
#pragma unroll 1
    for (int r0 = lane >> 3; r0 < 32; r0 += 16) {
        float4 x[4];
        size_t o[4];
        __nv_bfloat16 *h[4];
        bool in[4];
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const float *p = &blk[r0 + 4 * i][c];
            x[i] = make_float4(p[0], p[1], p[2], p[3]);
            in[i] = row0 + r0 + 4 * i < M;
            o[i] = (size_t)(row0 + r0 + 4 * i) * ldc + col;
            h[i] = E.H + (size_t)(row0 + r0 + 4 * i) * E.ldh + col;
        }
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        switch (E.kind) {
        case GEMM_BIAS:
        case GEMM_BIAS_GELU:
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const float4 z = make_float4(x[i].x + bias.x, x[i].y + bias.y, x[i].z + bias.z, x[i].w + bias.w);
                if (!in[i]) continue;
                st4<V>(E.C + o[i], z, n);
                if (E.kind == GEMM_BIAS_GELU)
                    st4<V>(h[i], make_float4(gelu_f(z.x), gelu_f(z.y), gelu_f(z.z), gelu_f(z.w)), n);
            }
            break;
        case GEMM_GELU_BACK: {
            float4 z[4];
#pragma unroll
            for (int i = 0; i < 4; i++) z[i] = in[i] ? ld4<V>(E.Z + o[i], n) : zero;
#pragma unroll
            for (int i = 0; i < 4; i++)
                if (in[i])
                    st4<V>(h[i],
                           make_float4(x[i].x * gelu_grad_f(z[i].x), x[i].y * gelu_grad_f(z[i].y),
                                       x[i].z * gelu_grad_f(z[i].z), x[i].w * gelu_grad_f(z[i].w)),
                           n);
            break;
        }
        case GEMM_ADAM: {
            float4 w[4], m[4], v[4];
#pragma unroll
            for (int i = 0; i < 4; i++) {
                w[i] = in[i] ? ld4<V>(E.w + o[i], n) : zero;
                m[i] = in[i] ? ld4<V>(E.m + o[i], n) : zero;
                v[i] = in[i] ? ld4<V>(E.v + o[i], n) : zero;
            }
#pragma unroll
            for (int i = 0; i < 4; i++) {
                adam_update(w[i].x, x[i].x, m[i].x, v[i].x, E.lr, E.c1, E.c2);
                adam_update(w[i].y, x[i].y, m[i].y, v[i].y, E.lr, E.c1, E.c2);
                adam_update(w[i].z, x[i].z, m[i].z, v[i].z, E.lr, E.c1, E.c2);
                adam_update(w[i].w, x[i].w, m[i].w, v[i].w, E.lr, E.c1, E.c2);
                if (!in[i]) continue;
                st4<V>(E.w + o[i], w[i], n);
                st4<V>(E.m + o[i], m[i], n);
                st4<V>(E.v + o[i], v[i], n);
                st4<V>(h[i], w[i], n);
            }
            break;
        }
        default:
#pragma unroll
            for (int i = 0; i < 4; i++)
                if (in[i]) st4<V>(E.C + o[i], x[i], n);
        }
    }
}

// (MNA and MNB: the weight gradients, see plan())
template <int BN, bool MNA, bool MNB>
__global__ void __launch_bounds__(128, MNA && MNB ? 4 : 1)
    k_gemm_tc(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, int M, int N,
              int K, int stages, int ldc, const __grid_constant__ GemmEpilogue E, int *err)
{
    static_assert(!MNB || BN >= 64, "an MN-major tile is made of 64-element boxes");
    constexpr int kTileB = tile_b(BN);
    constexpr uint32_t kIdesc = idesc(BN, MNA, MNB);
    extern __shared__ unsigned char smem_raw[];
    // tiles need 1024-byte alignment for the 128-byte swizzle
    unsigned char *base = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    unsigned char *sA = base;
    unsigned char *sB = base + (size_t)stages * kTileA;
    uint64_t *bars = reinterpret_cast<uint64_t *>(sB + (size_t)stages * kTileB);  // full[S], empty[S], done
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * stages + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int m0 = blockIdx.y * kBM, n0 = blockIdx.x * BN;
    const int ktiles = (K + kBK - 1) / kBK;
    const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + stages), done = smem_u32(bars + 2 * stages);

    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; s++) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(empty0 + 8 * s, 1);
        }
        mbar_init(done, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {  // tensor memory for the accumulator: BN columns x 128 lanes
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(BN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;

    int issued_loads = 0;  // producer: k-steps whose loads were issued
    if (warp == 0 && elect_one()) {
        // producer
        for (int kt = 0, s = 0, ph = 1; kt < ktiles; kt++) {
            if (kt >= stages && !mbar_wait(empty0 + 8 * s, ph)) {
                atomicExch(err, 1);
                *abort_flag = 1;
                break;
            }
            const uint32_t fb = full0 + 8 * s;
            const uint32_t a = smem_u32(sA + (size_t)s * kTileA), b = smem_u32(sB + (size_t)s * kTileB);
            mbar_expect_tx(fb, kTileA + kTileB);
            if constexpr (MNA) {
#pragma unroll
                for (int q = 0; q < kBM / 64; q++) tma_load_2d(a + q * 8192, &mapA, m0 + 64 * q, kt * kBK, fb);
            } else {
                tma_load_2d(a, &mapA, kt * kBK, m0, fb);
            }
            if constexpr (MNB) {
#pragma unroll
                for (int q = 0; q < BN / 64; q++) tma_load_2d(b + q * 8192, &mapB, n0 + 64 * q, kt * kBK, fb);
            } else {
                tma_load_2d(b, &mapB, kt * kBK, n0, fb);
            }
            issued_loads = kt + 1;
            if (++s == stages) s = 0, ph ^= 1;
        }
    } else if (warp == 1 && elect_one()) {
        // MMA issuer
        for (int kt = 0, s = 0, ph = 0; kt < ktiles; kt++) {
            if (!mbar_wait(full0 + 8 * s, ph)) {
                atomicExch(err, 1);
                *abort_flag = 1;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t a = smem_u32(sA + (size_t)s * kTileA), b = smem_u32(sB + (size_t)s * kTileB);
            const uint64_t da = MNA ? sw128_desc_mn(a) : sw128_desc(a);
            const uint64_t db = MNB ? sw128_desc_mn(b) : sw128_desc(b);
            // K = 16 per MMA: 32 bytes further along a K-major row, two 8-row groups of an MN-major tile
            constexpr uint64_t ka = MNA ? 2048 >> 4 : 2, kb = MNB ? 2048 >> 4 : 2;
#pragma unroll
            for (int k = 0; k < kBK / 16; k++)
                umma_f16(tmem, da + ka * k, db + kb * k, kIdesc, (kt > 0 || k > 0) ? 1u : 0u);
            umma_commit(empty0 + 8 * s);
            if (++s == stages) s = 0, ph ^= 1;
        }
        umma_commit(done);  // arrives when every MMA issued above has completed
    }
    // epilogue: every warp, its 32 lanes of tensor memory
    __syncwarp();
    const bool ok = mbar_wait(done, 0);
    if (!ok && lane == 0) atomicExch(err, 1);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (ok && !*abort_flag) {
        // every load has landed and every MMA has read it: the first stage's
        // A tile (16 KB; 16.5 KB with the first B tile after it when there is
        // one stage, else the next A tile) holds the warps' 32 x 33 blocks
        float(*blk)[33] = reinterpret_cast<float(*)[33]>(base) + 32 * warp;
        const int row0 = m0 + warp * 32;
#pragma unroll 1
        for (int c0 = 0; c0 < BN; c0 += 32) {
            uint32_t v[32];
            const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0;
            asm volatile(
                "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                  "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]),
                  "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]),
                  "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]),
                  "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
                : "r"(taddr));
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            __syncwarp();
#pragma unroll
            for (int q = 0; q < 32; q++) blk[lane][q] = __uint_as_float(v[q]);
            __syncwarp();
            if (row0 < M) {
                if (E.wide) epilogue_block<true>(E, blk, row0, n0 + c0 + 4 * (lane & 7), M, N, ldc);
                else epilogue_block<false>(E, blk, row0, n0 + c0 + 4 * (lane & 7), M, N, ldc);
            }
        }
    }
    if (issued_loads && *abort_flag) {
        // the producer of an aborted tile: let the last loads issued into each stage land
        // (bounded) before the CTA's shared memory goes away
        for (int kt = issued_loads - stages > 0 ? issued_loads - stages : 0; kt < issued_loads; kt++)
            mbar_wait(full0 + 8 * (kt % stages), (kt / stages) & 1);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(BN) : "memory");
    }
}

// ---- host: tensor maps through the driver entry point (no -lcuda) ----------
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn()
{
    static std::once_flag once;
    static EncodeTiledFn fn = nullptr;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
        else
            cudaGetLastError();
    });
    return fn;
}

// rows x cols BF16 matrix with row stride ld (elements); box of box_rows x 64.
// (For a K-strided operand the rows are k and the columns M or N.)
bool make_map(CUtensorMap *map, const __nv_bfloat16 *ptr, int rows, int cols, int ld, int box_rows)
{
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<__nv_bfloat16 *>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

bool gemm_tc_supported(int M, int N, int K, const GemmOperand &A, const GemmOperand &B)
{
    if (M < kBM || N < 128 || K < kBK) return false;
    if (!A.k_contiguous && B.k_contiguous) return false;  // no product has this pair of forms
    // rows that start on 16-byte boundaries (their length may be any: TMA fills what is past it)
    const int ca = A.k_contiguous ? K : M, cb = B.k_contiguous ? K : N;
    if (A.ld % 8 || B.ld % 8 || A.ld < ca || B.ld < cb) return false;
    if ((reinterpret_cast<uintptr_t>(A.p) & 15) || (reinterpret_cast<uintptr_t>(B.p) & 15)) return false;
    return encode_fn() != nullptr;
}

namespace {

// Tile width and stages.  The width with the fewest bytes into the busiest SM:
// waves of tiles times the 128 + BN operand rows that a tile reads in full (the
// L2 feeds an SM at about 64 bytes a cycle, less than its MMAs take).  A 256 x
// 1024 product makes 16 tiles of 128 x 128 for 152 SMs, and each then walks all
// of K alone; 64 tiles of 128 x 32 share that walk.  (32 columns at least, 64
// where B is MN-major.)  When there are more tiles than SMs, two CTAs share an
// SM, three where K is short, so that one's epilogue overlaps another's loads;
// else the stages fill the SM.  A weight update's time is its epilogue's traffic
// (26 bytes a weight): 64 columns and four CTAs an SM (128 registers) leave no
// short last wave and keep more of it in flight.  256 rows into 8192 x 1024 x
// 1024 x 4096: 245 -> 222 us the training step.
void plan(int M, int N, int K, bool mnb, bool update, int nsm, int *bn, int *stages)
{
    const long long mt = (M + kBM - 1) / kBM;
    long long best = 0, tiles = 0;
    for (int w = 128; w >= (mnb ? 64 : 32); w /= 2) {
        const long long t = mt * ((N + w - 1) / w), c = (t + nsm - 1) / nsm * (kBM + w);
        if (!best || c < best) {
            best = c;
            tiles = t;
            *bn = w;
        }
    }
    if (update && *bn == 128) {
        *bn = 64;
        tiles = mt * ((N + 63) / 64);
    }
    const int ktiles = (K + kBK - 1) / kBK, per = kTileA + tile_b(*bn);
    int st = (tiles <= nsm ? kStageBytes : update ? 50 * 1024 : ktiles <= 8 ? 70 * 1024 : 104 * 1024) / per;
    if (st > kMaxStages) st = kMaxStages;
    if (st > ktiles) st = ktiles;
    *stages = st < 2 ? 2 : st;
}

template <int BN, bool MNA, bool MNB>
cudaError_t launch(const CUtensorMap &ma, const CUtensorMap &mb, int M, int N, int K, int stages, int ldc,
                   const GemmEpilogue &E, int *err, cudaStream_t s)
{
    const size_t sm = smem_bytes(BN, stages);
    // the limit belongs to the kernel, not to this launch: always the same value,
    // or another thread's shape could lower it between here and the launch
    const cudaError_t e = cudaFuncSetAttribute(k_gemm_tc<BN, MNA, MNB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)smem_most(BN));
    if (e != cudaSuccess) return e;
    dim3 grid((N + BN - 1) / BN, (M + kBM - 1) / kBM);
    k_gemm_tc<BN, MNA, MNB><<<grid, 128, sm, s>>>(ma, mb, M, N, K, stages, ldc, E, err);
    return cudaGetLastError();
}

}  // namespace

cudaError_t gemm_tc(int M, int N, int K, const GemmOperand &A, const GemmOperand &B, int ldc, const GemmEpilogue &E,
                    int *err, cudaStream_t s)
{
    if (!gemm_tc_supported(M, N, K, A, B) || !err) return cudaErrorInvalidValue;
    int dev = 0, nsm = 0, bn = 0, stages = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    plan(M, N, K, !B.k_contiguous, E.kind == GEMM_ADAM, nsm, &bn, &stages);
    GemmEpilogue ep = E;
    // 16-byte accesses: every matrix (8 for the BF16 one) and row aligned for
    // them, and no row ending inside a group of four columns
    ep.wide = N % 4 == 0 && ldc % 4 == 0 && ep.ldh % 4 == 0 && (reinterpret_cast<uintptr_t>(E.H) & 7) == 0;
    for (const float *p : {(const float *)E.C, E.bias, E.Z, (const float *)E.w, (const float *)E.m, (const float *)E.v})
        ep.wide = ep.wide && (reinterpret_cast<uintptr_t>(p) & 15) == 0;
    CUtensorMap ma, mb;
    if (!(A.k_contiguous ? make_map(&ma, A.p, M, K, A.ld, kBM) : make_map(&ma, A.p, K, M, A.ld, kBK)) ||
        !(B.k_contiguous ? make_map(&mb, B.p, N, K, B.ld, bn) : make_map(&mb, B.p, K, N, B.ld, kBK)))
        return cudaErrorInvalidValue;
#define TMR_GEMM(BNN, MA, MB) launch<BNN, MA, MB>(ma, mb, M, N, K, stages, ldc, ep, err, s)
    if (A.k_contiguous && B.k_contiguous)
        return bn == 128 ? TMR_GEMM(128, false, false) : bn == 64 ? TMR_GEMM(64, false, false) : TMR_GEMM(32, false, false);
    if (A.k_contiguous) return bn == 128 ? TMR_GEMM(128, false, true) : TMR_GEMM(64, false, true);
    return bn == 128 ? TMR_GEMM(128, true, true) : TMR_GEMM(64, true, true);
#undef TMR_GEMM
}

}  // namespace tmr

extern "C" tmr_status tmr_gemm_bf16(int M, int N, int K, const void *A, int lda, const void *B, int ldb, float *C,
                                    int ldc, void *stream)
{
    tmr::set_last_error("");
    if (!A || !B || !C || M <= 0 || N <= 0 || K <= 0 || ldc < N) {
        tmr::set_last_error("tmr_gemm_bf16: bad argument");
        return TMR_ERR_INVALID_ARG;
    }
    if (!tmr::is_device_ptr(A) || !tmr::is_device_ptr(B) || !tmr::is_device_ptr(C)) {
        tmr::set_last_error("tmr_gemm_bf16: A, B and C must be device memory of the current device");
        return TMR_ERR_INVALID_ARG;
    }
    const tmr::GemmOperand oa{(const __nv_bfloat16 *)A, lda, true}, ob{(const __nv_bfloat16 *)B, ldb, true};
    tmr::GemmEpilogue ep{};
    ep.C = C;
    if (K % 8 || !tmr::gemm_tc_supported(M, N, K, oa, ob)) {
        tmr::set_last_error("tmr_gemm_bf16: needs M, N >= 128, K >= 64, K, lda, ldb multiples of 8, 16-byte alignment");
        return TMR_ERR_UNSUPPORTED;
    }
    int *err = nullptr;
    if (cudaMalloc(&err, sizeof(int)) != cudaSuccess) {
        cudaGetLastError();
        tmr::set_last_error("tmr_gemm_bf16: error flag");
        return TMR_ERR_OOM;
    }
    cudaStream_t s = (cudaStream_t)stream;
    int herr = 0;
    cudaError_t e = cudaMemsetAsync(err, 0, sizeof(int), s);
    if (e == cudaSuccess)
        e = tmr::gemm_tc(M, N, K, oa, ob, ldc, ep, err, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(err);
    if (e != cudaSuccess) {
        cudaGetLastError();
        tmr::set_last_error(cudaGetErrorString(e));
        return TMR_ERR_CUDA;
    }
    if (herr) {
        tmr::set_last_error("tmr_gemm_bf16: a barrier wait ran out");
        return TMR_ERR_TIMEOUT;
    }
    return TMR_OK;
}
