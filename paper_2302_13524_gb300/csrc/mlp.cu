// mlp.cu -- the learned initialiser's network: a three-layer perceptron
// x -> GELU(W1 x + b1) -> GELU(W2 h1 + b2) -> W3 h2 + b3, trained and run on
// the GPU by the kernels of this file.
//
// Weights are kept as FP32 master copies (updated by Adam) and as BF16 copies
// that feed the products; activations enter the products in BF16; every
// product accumulates in FP32 (mma.sync m16n8k16 BF16 tensor-core steps).  The
// loss is the mean squared error over every output, or its phase-invariant
// form (each target row rotated onto the output row first).  The forward
// products X W^T, the input gradients dZ W and the weight gradients dZ^T H run
// on the tensor cores with the layer's elementwise step as their epilogue
// (gemm_tc.cu); this file's mma.sync kernel, through generic element strides,
// takes the shapes that does not.  Rows of the BF16 matrices are padded to 16
// bytes (row_ld), which is what the tensor-core path asks of its operands, so that
// layers of any width take it.
#include <cuda_bf16.h>

#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>

#include "common.cuh"
#include "internal.h"
#include "mlp_math.cuh"
#include "tmr.h"

namespace tmr {

// C[M][N] (row-major, FP32) = sum_k A(m, k) B(k, n) with A(m, k) = A[m sam + k sak] and
// B(k, n) = B[k sbk + n sbn] in BF16.  64 x 64 tile per CTA, 4 warps of 32 x 32,
// K in steps of 32 through shared memory; out-of-range elements read as zero.
constexpr int GB_M = 64, GB_N = 64, GB_K = 32, GB_PAD = 8;

// Row stride of a BF16 matrix with n columns: 16-byte aligned rows.  The padding
// is zeroed where the matrix is allocated and never written.
__host__ __device__ constexpr int row_ld(int n) { return (n + 7) & ~7; }

__device__ __forceinline__ uint32_t pack_bf16(__nv_bfloat16 lo, __nv_bfloat16 hi)
{
    return (uint32_t)__bfloat16_as_ushort(lo) | ((uint32_t)__bfloat16_as_ushort(hi) << 16);
}

__global__ void __launch_bounds__(128) k_gemm_bf16(int M, int N, int K, const __nv_bfloat16 *__restrict__ A,
                                                  long long sam, long long sak,
                                                  const __nv_bfloat16 *__restrict__ B, long long sbk,
                                                  long long sbn, float *__restrict__ C, int ldc)
{
    __shared__ __nv_bfloat16 As[GB_M][GB_K + GB_PAD];
    __shared__ __nv_bfloat16 Bs[GB_N][GB_K + GB_PAD];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m0 = blockIdx.y * GB_M, n0 = blockIdx.x * GB_N;
    const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
    const int gid = lane >> 2, tig = lane & 3;
    float acc[2][4][4];
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
        for (int j = 0; j < 4; j++)
#pragma unroll
            for (int q = 0; q < 4; q++) acc[i][j][q] = 0.f;
    const __nv_bfloat16 zero = __float2bfloat16(0.f);
    for (int k0 = 0; k0 < K; k0 += GB_K) {
        // A tile: walk along whichever index is contiguous in memory
        for (int e = tid; e < GB_M * GB_K; e += 128) {
            int m, k;
            if (sak == 1) { m = e / GB_K; k = e % GB_K; }
            else { k = e / GB_M; m = e % GB_M; }
            const int gm = m0 + m, gk = k0 + k;
            As[m][k] = (gm < M && gk < K) ? A[gm * sam + gk * sak] : zero;
        }
        for (int e = tid; e < GB_N * GB_K; e += 128) {
            int n, k;
            if (sbk == 1) { n = e / GB_K; k = e % GB_K; }
            else { k = e / GB_N; n = e % GB_N; }
            const int gn = n0 + n, gk = k0 + k;
            Bs[n][k] = (gn < N && gk < K) ? B[gk * sbk + gn * sbn] : zero;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < GB_K; kk += 16) {
            uint32_t af[2][4], bfr[4][2];
#pragma unroll
            for (int i = 0; i < 2; i++) {
                const int r = wm + i * 16 + gid, c = kk + tig * 2;
                af[i][0] = pack_bf16(As[r][c], As[r][c + 1]);
                af[i][1] = pack_bf16(As[r + 8][c], As[r + 8][c + 1]);
                af[i][2] = pack_bf16(As[r][c + 8], As[r][c + 9]);
                af[i][3] = pack_bf16(As[r + 8][c + 8], As[r + 8][c + 9]);
            }
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const int n = wn + j * 8 + gid, c = kk + tig * 2;
                bfr[j][0] = pack_bf16(Bs[n][c], Bs[n][c + 1]);
                bfr[j][1] = pack_bf16(Bs[n][c + 8], Bs[n][c + 9]);
            }
#pragma unroll
            for (int i = 0; i < 2; i++)
#pragma unroll
                for (int j = 0; j < 4; j++)
                    asm volatile(
                        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
                        "{%8,%9}, {%0,%1,%2,%3};\n"
                        : "+f"(acc[i][j][0]), "+f"(acc[i][j][1]), "+f"(acc[i][j][2]), "+f"(acc[i][j][3])
                        : "r"(af[i][0]), "r"(af[i][1]), "r"(af[i][2]), "r"(af[i][3]), "r"(bfr[j][0]),
                          "r"(bfr[j][1]));
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int r = m0 + wm + i * 16 + gid, c = n0 + wn + j * 8 + tig * 2;
            if (r < M && c < N) C[(size_t)r * ldc + c] = acc[i][j][0];
            if (r < M && c + 1 < N) C[(size_t)r * ldc + c + 1] = acc[i][j][1];
            if (r + 8 < M && c < N) C[(size_t)(r + 8) * ldc + c] = acc[i][j][2];
            if (r + 8 < M && c + 1 < N) C[(size_t)(r + 8) * ldc + c + 1] = acc[i][j][3];
        }
}

static void gemm_sync(int M, int N, int K, const __nv_bfloat16 *A, long long sam, long long sak,
                      const __nv_bfloat16 *B, long long sbk, long long sbn, float *C, cudaStream_t s)
{
    dim3 grid((N + GB_N - 1) / GB_N, (M + GB_M - 1) / GB_M);
    k_gemm_bf16<<<grid, 128, 0, s>>>(M, N, K, A, sam, sak, B, sbk, sbn, C, N);
}

// A thread's elements of a matrix of n columns, row after row, without a division
// for each (64-bit ones take longer than the element's work).
struct RowWalk {
    size_t i, r, step, dr;
    int n, c, dc;
    __device__ RowWalk(int cols)
    {
        n = cols;
        i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
        step = (size_t)gridDim.x * blockDim.x;
        r = i / n, c = (int)(i - r * n);
        dr = step / n, dc = (int)(step - dr * n);
    }
    __device__ void next()
    {
        i += step, r += dr, c += dc;
        if (c >= n) c -= n, r++;
    }
};

// Z += b (per column); H (row stride ldh) = GELU(Z) in BF16 (gelu != 0) or Z itself copied to out.
__global__ void k_bias_act(int B, int N, float *Z, const float *b, __nv_bfloat16 *H, int ldh, int gelu)
{
    const size_t total = (size_t)B * N;
    for (RowWalk w(N); w.i < total; w.next()) {
        const float z = Z[w.i] + b[w.c];
        Z[w.i] = z;
        if (H) H[w.r * ldh + w.c] = __float2bfloat16(gelu ? gelu_f(z) : z);
    }
}

// One block per row: dY = 2 (Y - T) / (B N) and the row's sum of (Y - T)^2
// into part[row].  phase != 0 (the phase-invariant loss): the target row, read
// as t = T[:n] + i T[n:], n = N / 2, is first rotated onto the output row
// y = Y[:n] + i Y[n:]: t conj(c) / |c|, c = sum conj(y) t (unrotated where
// c = 0).  Sums in block_sum order.
__global__ void __launch_bounds__(256) k_loss_rows(int B, int N, int phase, const float *Y, const float *T,
                                                   __nv_bfloat16 *dY, float *part)
{
    const size_t o = (size_t)blockIdx.x * N;
    const float *y = Y + o, *t = T + o;
    __nv_bfloat16 *dy = dY + (size_t)blockIdx.x * row_ld(N);
    __shared__ float red[64], res[2];
    const float sc = 2.f / (float)((size_t)B * N);
    float acc = 0.f;
    if (phase) {
        const int n = N / 2;
        float cr = 0.f, ci = 0.f;
#pragma unroll 4
        for (int k = threadIdx.x; k < n; k += blockDim.x) {
            const float yr = y[k], yi = y[n + k], tr = t[k], ti = t[n + k];
            cr = fmaf(yr, tr, fmaf(yi, ti, cr));
            ci = fmaf(yr, ti, fmaf(-yi, tr, ci));
        }
        float v[2] = {cr, ci};
        block_sum<2>(v, red, res);
        const float ac = sqrtf(res[0] * res[0] + res[1] * res[1]);
        const float rr = ac > 0.f ? res[0] / ac : 1.f, ri = ac > 0.f ? -res[1] / ac : 0.f;  // conj(c) / |c|
#pragma unroll 4
        for (int k = threadIdx.x; k < n; k += blockDim.x) {
            const float tr = t[k], ti = t[n + k];
            const float e0 = y[k] - (tr * rr - ti * ri), e1 = y[n + k] - (tr * ri + ti * rr);
            acc = fmaf(e0, e0, acc);
            acc = fmaf(e1, e1, acc);
            dy[k] = __float2bfloat16(sc * e0);
            dy[n + k] = __float2bfloat16(sc * e1);
        }
    } else {
#pragma unroll 4
        for (int k = threadIdx.x; k < N; k += blockDim.x) {
            const float e = y[k] - t[k];
            acc = fmaf(e, e, acc);
            dy[k] = __float2bfloat16(sc * e);
        }
    }
    __syncthreads();  // res is read before red and res are used again
    float v[1] = {acc};
    block_sum<1>(v, red, res);
    if (threadIdx.x == 0) part[blockIdx.x] = res[0];
}

// loss = sum of the parts / total, FP64, one block of 256 threads (one thread
// walking the parts took longer than any product of the step)
__global__ void __launch_bounds__(256) k_loss_finish(int nparts, const float *part, float total, float *loss)
{
    double s = 0.0;
    for (int i = threadIdx.x; i < nparts; i += 256) s += part[i];
    __shared__ double red[8], out[1];
    double v[1] = {s};
    block_sum<1>(v, red, out);
    if (threadIdx.x == 0) *loss = (float)(out[0] / total);
}

// dZ = dH .* GELU'(Z) -> BF16 (row stride ldz)
__global__ void k_gelu_back(int B, int N, const float *dH, const float *Z, __nv_bfloat16 *dZ, int ldz)
{
    const size_t n = (size_t)B * N;
    for (RowWalk w(N); w.i < n; w.next())
        dZ[w.r * ldz + w.c] = __float2bfloat16(dH[w.i] * gelu_grad_f(Z[w.i]));
}

// Bias gradients of the three layers in one launch: g[c] = sum_r dZ[r][c] (dZ
// BF16, rows of N), and with adam != 0 the biases' Adam update instead of storing
// it.  A block of 32 x 8 threads takes 32 columns of one layer, thread (c, r)
// the rows r, r + 8, ...  (One thread per column, walking all rows, used 16
// blocks of the chip for 20 us a layer.)
struct BiasLayer {
    const __nv_bfloat16 *dZ;
    int N, block0;  // columns; first block of the layer
    float *g, *w, *m, *v;
};
struct BiasLayers {
    BiasLayer l[3];
};
__global__ void __launch_bounds__(256) k_bias_grad(int B, const __grid_constant__ BiasLayers P, int adam, float lr,
                                                   float c1, float c2)
{
    const BiasLayer &L = P.l[(int)blockIdx.x >= P.l[2].block0 ? 2 : (int)blockIdx.x >= P.l[1].block0 ? 1 : 0];
    const int c = ((int)blockIdx.x - L.block0) * 32 + threadIdx.x;
    __shared__ float red[8][33];
    float s = 0.f;
    if (c < L.N) {
#pragma unroll 8
        for (int r = threadIdx.y; r < B; r += 8) s += __bfloat162float(L.dZ[(size_t)r * row_ld(L.N) + c]);
    }
    red[threadIdx.y][threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.y != 0 || c >= L.N) return;
#pragma unroll
    for (int r = 1; r < 8; r++) s += red[r][threadIdx.x];
    if (!adam) {
        L.g[c] = s;
        return;
    }
    float w = L.w[c], m = L.m[c], v = L.v[c];
    adam_update(w, s, m, v, lr, c1, c2);
    L.w[c] = w;
    L.m[c] = m;
    L.v[c] = v;
}

// x -> BF16, four values a thread and step where both are aligned for it
__global__ void k_to_bf16(size_t n, const float *x, __nv_bfloat16 *y)
{
    const size_t t0 = blockIdx.x * (size_t)blockDim.x + threadIdx.x, step = (size_t)gridDim.x * blockDim.x;
    size_t done = 0;
    if (((reinterpret_cast<uintptr_t>(x) & 15) | (reinterpret_cast<uintptr_t>(y) & 7)) == 0) {
        const size_t n4 = n / 4;
#pragma unroll 4
        for (size_t i = t0; i < n4; i += step) {
            const float4 v = reinterpret_cast<const float4 *>(x)[i];
            const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
            reinterpret_cast<uint2 *>(y)[i] =
                make_uint2(*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi));
        }
        done = 4 * n4;
    }
    for (size_t i = done + t0; i < n; i += step) y[i] = __float2bfloat16(x[i]);
}
// the same of rows of n values into rows of stride ld
__global__ void k_rows_to_bf16(int rows, int n, const float *x, __nv_bfloat16 *y, int ld)
{
    const size_t total = (size_t)rows * n;
    for (RowWalk w(n); w.i < total; w.next()) y[w.r * ld + w.c] = __float2bfloat16(x[w.i]);
}

// wb: the weights' BF16 copy, row stride ldw
__global__ void k_adam(int rows, int cols, float *w, const float *g, float *m, float *v, __nv_bfloat16 *wb, int ldw,
                       float lr, float c1, float c2)
{
    const size_t n = (size_t)rows * cols;
    for (RowWalk k(cols); k.i < n; k.next()) {
        const size_t i = k.i;
        float wi = w[i], mi = m[i], vi = v[i];
        adam_update(wi, g[i], mi, vi, lr, c1, c2);
        m[i] = mi;
        v[i] = vi;
        w[i] = wi;
        wb[k.r * ldw + k.c] = __float2bfloat16(wi);
    }
}

// y = normalised sqrt intensities: x[r][i] = sqrt(max(y, 0)) / sqrt(mean_i y[r][i]) (BF16, padded rows)
__global__ void k_features(int K, const float *y, __nv_bfloat16 *x)
{
    const int r = blockIdx.x;
    const float *yr = y + (size_t)r * K;
    float s = 0.f;
    for (int i = threadIdx.x; i < K; i += blockDim.x) s += fmaxf(yr[i], 0.f);
    __shared__ float red[32], out[1];
    float v[1] = {s};
    block_sum<1>(v, red, out);
    const float inv = out[0] > 0.f ? rsqrtf(out[0] / (float)K) : 0.f;
    for (int i = threadIdx.x; i < K; i += blockDim.x)
        x[(size_t)r * row_ld(K) + i] = __float2bfloat16(sqrtf(fmaxf(yr[i], 0.f)) * inv);
}

// candidate start: t[n] = (out[n] + i out[N + n]) scaled to ||t||^2 = sum(y) / (J N)
__global__ void k_candidate(int N, int K, const float *out, const float *y, float2 *T)
{
    const int r = blockIdx.x;
    const float *o = out + (size_t)r * 2 * N;
    const float *yr = y + (size_t)r * K;
    float sy = 0.f, sn = 0.f;
    for (int i = threadIdx.x; i < K; i += blockDim.x) sy += fmaxf(yr[i], 0.f);
    for (int n = threadIdx.x; n < N; n += blockDim.x) sn += o[n] * o[n] + o[N + n] * o[N + n];
    __shared__ float red[64], res[2];
    float v[2] = {sy, sn};
    block_sum<2>(v, red, res);
    const float sc = res[1] > 0.f ? sqrtf(res[0] / (float)K) / sqrtf(res[1]) : 0.f;
    for (int n = threadIdx.x; n < N; n += blockDim.x)
        T[(size_t)r * N + n] = make_float2(o[n] * sc, o[N + n] * sc);
}

}  // namespace tmr

using namespace tmr;

struct tmr_mlp {
    int n_in, h1, h2, n_out;
    size_t np;  // parameters
    size_t off[6];   // each layer's weights and biases among them
    size_t woff[3];  // the layers' weights in wb
    cudaStream_t stream;
    float *w = nullptr, *m = nullptr, *v = nullptr, *g = nullptr;
    __nv_bfloat16 *wb = nullptr;  // the weights in BF16, padded rows
    long long step = 0;
    // batch scratch
    int cap = 0;
    __nv_bfloat16 *xb = nullptr, *h1b = nullptr, *h2b = nullptr, *dzb = nullptr, *dz2b = nullptr, *dyb = nullptr;
    float *z1 = nullptr, *z2 = nullptr, *y = nullptr, *dh = nullptr, *part = nullptr, *lossd = nullptr;
    int loss_kind = TMR_LOSS_MSE;
    int *tc_err = nullptr;  // tensor-core GEMM: the barrier-timeout flag
};

namespace {

tmr_status mfail(tmr_status st, const char *msg)
{
    set_last_error(msg);
    return st;
}

bool dev_ptr(const void *p) { return tmr::is_device_ptr(p); }

int ew_blocks(size_t n);

// C[M][N] = sum_k A(m, k) B(n, k), then the elementwise step E (row stride N),
// on the tcgen05 tensor cores (gemm_tc.cu) when the shape allows; otherwise the
// mma.sync tile kernel above, the product into E.C (which the caller sets to
// scratch where E itself does not store it) and the step as its own kernel.
void gemm(tmr_mlp *m, int M, int N, int K, const GemmOperand &A, const GemmOperand &B, const GemmEpilogue &E)
{
    cudaStream_t s = m->stream;
    if (m->tc_err && gemm_tc_supported(M, N, K, A, B)) {
        if (gemm_tc(M, N, K, A, B, N, E, m->tc_err, s) == cudaSuccess) return;
        cudaGetLastError();
    }
    gemm_sync(M, N, K, A.p, A.k_contiguous ? A.ld : 1, A.k_contiguous ? 1 : A.ld, B.p, B.k_contiguous ? 1 : B.ld,
              B.k_contiguous ? B.ld : 1, E.C, s);
    const size_t n = (size_t)M * N;
    const int nb = ew_blocks(n);
    switch (E.kind) {
    case GEMM_BIAS:
    case GEMM_BIAS_GELU: k_bias_act<<<nb, 256, 0, s>>>(M, N, E.C, E.bias, E.H, E.ldh, E.kind == GEMM_BIAS_GELU); break;
    case GEMM_GELU_BACK: k_gelu_back<<<nb, 256, 0, s>>>(M, N, E.C, E.Z, E.H, E.ldh); break;
    case GEMM_ADAM: k_adam<<<nb, 256, 0, s>>>(M, N, E.w, E.C, E.m, E.v, E.H, E.ldh, E.lr, E.c1, E.c2); break;
    default: break;
    }
}

int ew_blocks(size_t n)
{
    size_t b = (n + 255) / 256;
    return (int)(b > 152 * 8 ? 152 * 8 : (b < 1 ? 1 : b));
}

// rows x n values to BF16, padded rows
void to_bf16(int rows, int n, const float *x, __nv_bfloat16 *y, cudaStream_t s)
{
    const size_t total = (size_t)rows * n;
    if (row_ld(n) == n) k_to_bf16<<<ew_blocks(total), 256, 0, s>>>(total, x, y);
    else k_rows_to_bf16<<<ew_blocks(total), 256, 0, s>>>(rows, n, x, y, row_ld(n));
}

tmr_status ensure_batch(tmr_mlp *m, int B)
{
    if (B <= m->cap) return TMR_OK;
    void **bufs[] = {(void **)&m->xb, (void **)&m->h1b, (void **)&m->h2b, (void **)&m->dzb, (void **)&m->dz2b,
                     (void **)&m->dyb, (void **)&m->z1, (void **)&m->z2, (void **)&m->y, (void **)&m->dh,
                     (void **)&m->part};
    for (void **b : bufs)
        if (*b) {
            cudaFree(*b);
            *b = nullptr;
        }
    const int hid = m->h1 > m->h2 ? m->h1 : m->h2, io = m->n_in > m->n_out ? m->n_in : m->n_out;
    const int hmax = io > hid ? io : hid;
    const size_t rows = (size_t)B;
    bool zeroed = false;
    auto padded = [&](__nv_bfloat16 **p, int width) {
        const size_t bytes = sizeof(__nv_bfloat16) * rows * row_ld(width);
        if (cudaMalloc(p, bytes) != cudaSuccess) return false;
        if (row_ld(width) == width) return true;
        zeroed = true;
        return cudaMemsetAsync(*p, 0, bytes, m->stream) == cudaSuccess;
    };
    bool ok = padded(&m->xb, m->n_in) && padded(&m->h1b, m->h1) && padded(&m->h2b, m->h2) && padded(&m->dzb, m->h1) &&
              padded(&m->dz2b, m->h2) && padded(&m->dyb, m->n_out) &&
              cudaMalloc(&m->z1, sizeof(float) * rows * m->h1) == cudaSuccess &&
              cudaMalloc(&m->z2, sizeof(float) * rows * m->h2) == cudaSuccess &&
              cudaMalloc(&m->y, sizeof(float) * rows * m->n_out) == cudaSuccess &&
              cudaMalloc(&m->dh, sizeof(float) * rows * hmax) == cudaSuccess &&
              cudaMalloc(&m->part, sizeof(float) * rows) == cudaSuccess &&
              // mlp_propose goes on on another stream
              (!zeroed || cudaStreamSynchronize(m->stream) == cudaSuccess);
    if (!ok) {
        cudaGetLastError();
        return mfail(TMR_ERR_OOM, "MLP batch buffers");
    }
    m->cap = B;
    return TMR_OK;
}

GemmEpilogue bias_step(float *z, const float *bias, __nv_bfloat16 *h, int ldh)
{
    GemmEpilogue E;
    E.kind = h ? GEMM_BIAS_GELU : GEMM_BIAS;
    E.C = z;
    E.bias = bias;
    E.H = h;
    E.ldh = ldh;
    return E;
}

// forward from BF16 features m->xb into y (FP32 [B][out]); keeps Z1, Z2, H1, H2
void forward_core(tmr_mlp *m, int B, float *y)
{
    const __nv_bfloat16 *W1 = m->wb + m->woff[0], *W2 = m->wb + m->woff[1], *W3 = m->wb + m->woff[2];
    const float *b1 = m->w + m->off[1], *b2 = m->w + m->off[3], *b3 = m->w + m->off[5];
    const int li = row_ld(m->n_in), l1 = row_ld(m->h1), l2 = row_ld(m->h2);
    gemm(m, B, m->h1, m->n_in, {m->xb, li, true}, {W1, li, true}, bias_step(m->z1, b1, m->h1b, l1));
    gemm(m, B, m->h2, m->h1, {m->h1b, l1, true}, {W2, l1, true}, bias_step(m->z2, b2, m->h2b, l2));
    gemm(m, B, m->n_out, m->h2, {m->h2b, l2, true}, {W3, l2, true}, bias_step(y, b3, nullptr, 0));
}

// One Adam step's size and bias corrections
struct AdamStep {
    float lr, c1, c2;
};

// The loss (device scalar) and, from m->y, the gradient w.r.t. every parameter
// into g; with `step`, every parameter is updated by it instead (g is scratch).
void backward_core(tmr_mlp *m, int B, const float *T, float *loss, float *g, const AdamStep *step)
{
    cudaStream_t s = m->stream;
    const __nv_bfloat16 *W2 = m->wb + m->woff[1], *W3 = m->wb + m->woff[2];
    const int li = row_ld(m->n_in), l1 = row_ld(m->h1), l2 = row_ld(m->h2), lo = row_ld(m->n_out);
    k_loss_rows<<<B, 256, 0, s>>>(B, m->n_out, m->loss_kind == TMR_LOSS_PHASE, m->y, T, m->dyb, m->part);
    k_loss_finish<<<1, 256, 0, s>>>(B, m->part, (float)((size_t)B * m->n_out), loss);
    // dZ = (dZ_next W) .* GELU'(Z)
    auto back = [&](const float *z, __nv_bfloat16 *dz, int ldz) {
        GemmEpilogue E;
        E.kind = GEMM_GELU_BACK;
        E.C = m->dh;
        E.Z = z;
        E.H = dz;
        E.ldh = ldz;
        return E;
    };
    // dW = dZ^T H: the gradient, or the update of the layer's weights
    auto weights = [&](int layer, int ldw) {
        const size_t o = m->off[2 * layer];
        GemmEpilogue E;
        E.C = g + o;
        if (step) {
            E.kind = GEMM_ADAM;
            E.w = m->w + o;
            E.m = m->m + o;
            E.v = m->v + o;
            E.H = m->wb + m->woff[layer];
            E.ldh = ldw;
            E.lr = step->lr;
            E.c1 = step->c1;
            E.c2 = step->c2;
        }
        return E;
    };
    // every dZ is made before the weights it was made with change
    gemm(m, B, m->h2, m->n_out, {m->dyb, lo, true}, {W3, l2, false}, back(m->z2, m->dz2b, l2));
    gemm(m, m->n_out, m->h2, B, {m->dyb, lo, false}, {m->h2b, l2, false}, weights(2, l2));
    gemm(m, B, m->h1, m->h2, {m->dz2b, l2, true}, {W2, l1, false}, back(m->z1, m->dzb, l1));
    gemm(m, m->h2, m->h1, B, {m->dz2b, l2, false}, {m->h1b, l1, false}, weights(1, l1));
    gemm(m, m->h1, m->n_in, B, {m->dzb, l1, false}, {m->xb, li, false}, weights(0, li));
    BiasLayers L;
    const __nv_bfloat16 *dz[3] = {m->dzb, m->dz2b, m->dyb};
    const int width[3] = {m->h1, m->h2, m->n_out};
    int blocks = 0;
    for (int i = 0; i < 3; i++) {
        const size_t o = m->off[2 * i + 1];
        L.l[i] = {dz[i], width[i], blocks, g + o, m->w + o, m->m + o, m->v + o};
        blocks += (width[i] + 31) / 32;
    }
    k_bias_grad<<<blocks, dim3(32, 8), 0, s>>>(B, L, step != nullptr, step ? step->lr : 0.f, step ? step->c1 : 1.f,
                                               step ? step->c2 : 1.f);
}

}  // namespace

namespace tmr {
// used by the learned start of tmr_retrieve: features of rows [r0, r0+B) of y
// -> candidate starts T (rows r0 ..)
cudaError_t mlp_propose(tmr_mlp *m, const float *y, int B, int N, int J, float2 *T, cudaStream_t s)
{
    if (ensure_batch(m, B) != TMR_OK) return cudaErrorMemoryAllocation;
    cudaStream_t keep = m->stream;
    m->stream = s;
    k_features<<<B, 256, 0, s>>>(J * N, y, m->xb);
    forward_core(m, B, m->y);
    k_candidate<<<B, 256, 0, s>>>(N, J * N, m->y, y, T);
    m->stream = keep;
    return cudaGetLastError();
}
int mlp_in(const tmr_mlp *m) { return m->n_in; }
int mlp_out(const tmr_mlp *m) { return m->n_out; }
}  // namespace tmr

extern "C" {

tmr_status tmr_mlp_create(tmr_mlp **out, int n_in, int n_h1, int n_h2, int n_out, unsigned long long seed,
                          void *stream)
{
    set_last_error("");
    if (!out || n_in <= 0 || n_h1 <= 0 || n_h2 <= 0 || n_out <= 0) return mfail(TMR_ERR_INVALID_ARG, "bad MLP size");
    tmr_mlp *m = new tmr_mlp();
    m->n_in = n_in;
    m->h1 = n_h1;
    m->h2 = n_h2;
    m->n_out = n_out;
    m->stream = (cudaStream_t)stream;
    const size_t sz[6] = {(size_t)n_h1 * n_in, (size_t)n_h1, (size_t)n_h2 * n_h1, (size_t)n_h2,
                          (size_t)n_out * n_h2, (size_t)n_out};
    size_t o = 0;
    for (int i = 0; i < 6; i++) {
        m->off[i] = o;
        o += sz[i];
    }
    m->np = o;
    size_t nwb = 0;
    const int fan[3][2] = {{n_h1, n_in}, {n_h2, n_h1}, {n_out, n_h2}};
    for (int l = 0; l < 3; l++) {
        m->woff[l] = nwb;
        nwb += (size_t)fan[l][0] * row_ld(fan[l][1]);
    }
    const bool ok = cudaMalloc(&m->w, sizeof(float) * o) == cudaSuccess &&
                    cudaMalloc(&m->m, sizeof(float) * o) == cudaSuccess &&
                    cudaMalloc(&m->v, sizeof(float) * o) == cudaSuccess &&
                    cudaMalloc(&m->g, sizeof(float) * o) == cudaSuccess &&
                    cudaMalloc(&m->wb, sizeof(__nv_bfloat16) * nwb) == cudaSuccess &&
                    cudaMemsetAsync(m->wb, 0, sizeof(__nv_bfloat16) * nwb, m->stream) == cudaSuccess &&
                    cudaMalloc(&m->lossd, sizeof(float) * 4) == cudaSuccess &&
                    cudaMalloc(&m->tc_err, sizeof(int)) == cudaSuccess &&
                    cudaMemset(m->tc_err, 0, sizeof(int)) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        tmr_mlp_destroy(m);
        return mfail(TMR_ERR_OOM, "MLP parameters");
    }
    // He-style start: W ~ U(-s, s) with s = sqrt(3 / fan_in) (Philox), biases 0
    float *hw = (float *)malloc(sizeof(float) * o);
    for (int l = 0; l < 3; l++) {
        const int fan_in = l == 0 ? n_in : (l == 1 ? n_h1 : n_h2);
        const float s = sqrtf(3.f / (float)fan_in);
        for (size_t i = 0; i < sz[2 * l]; i++) {
            const uint4 r = philox4x32_10(make_uint4((uint32_t)i, (uint32_t)(i >> 32), (uint32_t)l, 0u),
                                          make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)));
            hw[m->off[2 * l] + i] = s * (2.f * ((float)r.x * 0x1p-32f) - 1.f);
        }
        for (size_t i = 0; i < sz[2 * l + 1]; i++) hw[m->off[2 * l + 1] + i] = 0.f;
    }
    tmr_status st = tmr_mlp_set_params(m, hw);
    free(hw);
    if (st != TMR_OK) {
        tmr_mlp_destroy(m);
        return st;
    }
    *out = m;
    return TMR_OK;
}

size_t tmr_mlp_num_params(const tmr_mlp *m) { return m ? m->np : 0; }

tmr_status tmr_mlp_set_params(tmr_mlp *m, const float *params)
{
    set_last_error("");
    if (!m || !params) return mfail(TMR_ERR_INVALID_ARG, "NULL argument");
    if (cudaMemcpyAsync(m->w, params, sizeof(float) * m->np, cudaMemcpyDefault, m->stream) != cudaSuccess ||
        cudaMemsetAsync(m->m, 0, sizeof(float) * m->np, m->stream) != cudaSuccess ||
        cudaMemsetAsync(m->v, 0, sizeof(float) * m->np, m->stream) != cudaSuccess)
        return mfail(TMR_ERR_CUDA, "set params");
    to_bf16(m->h1, m->n_in, m->w + m->off[0], m->wb + m->woff[0], m->stream);
    to_bf16(m->h2, m->h1, m->w + m->off[2], m->wb + m->woff[1], m->stream);
    to_bf16(m->n_out, m->h2, m->w + m->off[4], m->wb + m->woff[2], m->stream);
    m->step = 0;
    if (cudaStreamSynchronize(m->stream) != cudaSuccess) return mfail(TMR_ERR_CUDA, "set params sync");
    return TMR_OK;
}

tmr_status tmr_mlp_get_params(tmr_mlp *m, float *params)
{
    set_last_error("");
    if (!m || !params) return mfail(TMR_ERR_INVALID_ARG, "NULL argument");
    int tc_err = 0;
    if (cudaMemcpyAsync(params, m->w, sizeof(float) * m->np, cudaMemcpyDefault, m->stream) != cudaSuccess ||
        cudaMemcpyAsync(&tc_err, m->tc_err, sizeof(int), cudaMemcpyDeviceToHost, m->stream) != cudaSuccess ||
        cudaStreamSynchronize(m->stream) != cudaSuccess)
        return mfail(TMR_ERR_CUDA, "get params");
    if (tc_err) return mfail(TMR_ERR_TIMEOUT, "a tensor-core GEMM barrier wait ran out");
    return TMR_OK;
}

tmr_status tmr_mlp_forward(tmr_mlp *m, const float *X, int B, float *Y)
{
    set_last_error("");
    if (!m || !X || !Y || B <= 0) return mfail(TMR_ERR_INVALID_ARG, "bad argument");
    if (!dev_ptr(X) || !dev_ptr(Y)) return mfail(TMR_ERR_INVALID_ARG, "X and Y must be device memory");
    tmr_status st = ensure_batch(m, B);
    if (st != TMR_OK) return st;
    to_bf16(B, m->n_in, X, m->xb, m->stream);
    forward_core(m, B, Y);
    return cudaGetLastError() == cudaSuccess ? TMR_OK : mfail(TMR_ERR_CUDA, "forward kernels");
}

// the batch's loss and, without `step`, its gradient (into grad, or scratch when
// NULL), with it one update
static tmr_status mlp_batch(tmr_mlp *m, const float *X, const float *T, int B, float *loss, float *grad,
                            const AdamStep *step)
{
    set_last_error("");
    if (!m || !X || !T || B <= 0) return mfail(TMR_ERR_INVALID_ARG, "bad argument");
    if (!dev_ptr(X) || !dev_ptr(T) || (loss && !dev_ptr(loss)) || (grad && !dev_ptr(grad)))
        return mfail(TMR_ERR_INVALID_ARG, "arrays must be device memory");
    tmr_status st = ensure_batch(m, B);
    if (st != TMR_OK) return st;
    to_bf16(B, m->n_in, X, m->xb, m->stream);
    forward_core(m, B, m->y);
    backward_core(m, B, T, loss ? loss : m->lossd, grad ? grad : m->g, step);
    return cudaGetLastError() == cudaSuccess ? TMR_OK : mfail(TMR_ERR_CUDA, "network kernels");
}

tmr_status tmr_mlp_grad(tmr_mlp *m, const float *X, const float *T, int B, float *loss, float *grad)
{
    return mlp_batch(m, X, T, B, loss, grad, nullptr);
}

tmr_status tmr_mlp_train_step(tmr_mlp *m, const float *X, const float *T, int B, float lr, float *loss)
{
    if (!m) return mlp_batch(m, X, T, B, loss, nullptr, nullptr);  // refused there
    const float t = (float)(m->step + 1);
    const AdamStep step = {lr, 1.f - powf(0.9f, t), 1.f - powf(0.999f, t)};
    const tmr_status st = mlp_batch(m, X, T, B, loss, nullptr, &step);
    if (st == TMR_OK) m->step++;
    return st;
}

tmr_status tmr_mlp_set_loss(tmr_mlp *m, int kind)
{
    set_last_error("");
    if (!m) return mfail(TMR_ERR_INVALID_ARG, "NULL network");
    if (kind != TMR_LOSS_MSE && kind != TMR_LOSS_PHASE) return mfail(TMR_ERR_INVALID_ARG, "unknown loss");
    if (kind == TMR_LOSS_PHASE && m->n_out % 2 != 0)
        return mfail(TMR_ERR_INVALID_ARG, "the phase-invariant loss needs an even number of outputs");
    m->loss_kind = kind;
    return TMR_OK;
}

void tmr_mlp_destroy(tmr_mlp *m)
{
    if (!m) return;
    if (m->stream) cudaStreamSynchronize(m->stream);
    else cudaDeviceSynchronize();
    void *p[] = {m->w, m->m, m->v, m->g, m->wb, m->xb, m->h1b, m->h2b, m->dzb, m->dz2b, m->dyb,
                 m->z1, m->z2, m->y, m->dh, m->part, m->lossd, m->tc_err};
    for (void *q : p)
        if (q) cudaFree(q);
    delete m;
}

}  // extern "C"
