// solver_row.cuh -- the per-row solver (Algorithm 1) with one CTA per row.
//
// The same iteration as k_solver (solver_impl.cuh): initialisation, then
// L-BFGS steps each made of one forward batch w_j = F(d_j .* p), the exact
// minimiser of the quartic phi(a) = f(t + a p), the update t += a p,
// z += a w, one adjoint batch for the new gradient (Eq. derivative) and the
// compact-form direction from the Gram scalars.  What differs is the layout,
// chosen so that a row needs no thread-block cluster:
//   * every mask of the row is a team of NT = N/16 threads in one CTA, each
//     thread holding 16 points of z_j and w_j in registers; the transforms
//     are register Stockham passes of radix 16 after a first pass of the
//     remaining radix (2048 = 8 x 16 x 16: two exchanges through shared
//     memory per transform), the last pass's twiddles formed from per-thread
//     bases and the others' in a small table made on the device (FP64
//     sincospi rounded to FP32);
//   * the masks and the row's intensities live in shared memory (the masks
//     are copied once per CTA and shared by all its rows), next to full-length
//     t, g and the direction p, and one exchange buffer per team;
//   * the L-BFGS pairs (2 (m + 1) vectors of N complex values, 192 KB at
//     N = 2048, m = 5) live in the SM's tensor memory, which the FP32 solver
//     has no other use for: each thread keeps the elements it owns in the
//     A and G phases (i = tid + e BT) in columns of its own lane, so the two
//     passes over the pairs of every iteration read tensor memory instead of
//     L2; before the first pair exists, the same columns hold the vectors of
//     the Lanczos start where they fit (k N complex values: 256 KB, all 512
//     columns, at N = 2048, J = 4, k = 16), else those stay in global memory;
//   * every exchange and every reduction is inside the CTA: block barriers
//     instead of cluster barriers, no distributed shared memory.
// Rows come from the same atomic work counter; a persistent launch of one
// CTA per SM (or two, when shared memory allows) walks the matrix.
//
// A row too large for one CTA (N = 4096, or more than four masks of N = 2048)
// takes the same layout over a small cluster (CLU): each CTA holds two or more
// of its masks and a slice of its vectors, so that a row occupies half or a
// quarter of the SMs that one mask per CTA (solver_impl.cuh) gives it, and the
// serial parts of an iteration (reductions, scalars, barriers: half of it at one
// mask per CTA) are shared by that many more rows.  N = 4096, J = 4, M = 4096,
// 20 iterations: 21.6 ms against 29.0 (19.4 with the fields in tensor memory, ZT below).
// For a few rows, which do not fill the chip either way, it is the slower one: see
// tune_rows in api.cu.
#pragma once

#include "solver_impl.cuh"
#include "tmem.cuh"

namespace tmr {

constexpr int kRowPts = 16;

template <int N_>
struct RowCfg {
    static constexpr int N = N_;
    static constexpr int E = kRowPts;  // points per thread of one transform
    static constexpr int NT = N_ / E;  // threads per team (one mask)
    static constexpr int R = 16;       // radix of every pass but the first
    static constexpr int BPT = E / R;  // butterflies per thread in the last pass
    using Plan = FftPlan<N_, E, R>;
    static constexpr int NCONST = Plan::TW_SMALL;  // twiddles of the non-final passes
    static constexpr int LBUF = fft_buf_len(N_);
};

// Variants exist for N = 512 .. 2048 with J * N / 16 <= 512 threads.
__host__ __device__ constexpr bool row_variant_fits(int N, int J) { return J >= 1 && J * (N / kRowPts) <= 512; }

// The same layout over a cluster (CLU): each CTA holds JB of the row's masks
// and a 1/JC slice of its vectors, JC = J / JB.  JB: the most masks that fit
// 512 threads, at least 2; 0 when the row fits one CTA or no such split exists.
__host__ __device__ constexpr int rowc_masks(int N, int J)
{
    if ((N != 2048 && N != 4096) || J > kMaxMasks || row_variant_fits(N, J)) return 0;
    for (int jb = 512 / (N / kRowPts); jb >= 2; jb--)
        if (J % jb == 0 && J / jb >= 2) return jb;
    return 0;
}

template <int N>
__host__ __device__ size_t rowc_smem(int J)
{
    using C = RowCfg<N>;
    const int JB = rowc_masks(N, J), JC = J / JB, NW = JB * C::NT / 32;
    const size_t SL = (N + JC - 1) / JC;
    const size_t f2 = ((size_t)C::NCONST + 1) / 2 * 2 + (size_t)JB * N /*masks*/ + (size_t)JB * C::LBUF /*exchange; the
                      first also gathers p*/ + 2 * SL /*t, g*/ + (JC - 1) * SL /*peers' sums*/ + kMaxLanczos * kMaxLanczos;
    size_t bytes = f2 * sizeof(float2) +
                   sizeof(float) * ((size_t)JB * N /*y*/ + (size_t)kParts * NW + 2 * (size_t)JC * kParts);
    bytes = (bytes + 15) & ~(size_t)15;
    return bytes + kGramBytes;
}

template <int N>
__host__ __device__ size_t row_smem(int J, int m)
{
    using C = RowCfg<N>;
    (void)m;
    const int NW = J * C::NT / 32;
    size_t f2 = ((size_t)C::NCONST + 1) / 2 * 2 /*twiddles, even count*/ + (size_t)J * N /*masks*/ +
                (size_t)J * C::LBUF /*team exchange buffers*/ + 3 * (size_t)N /*p, t, g*/;
    size_t bytes = f2 * sizeof(float2) + sizeof(float) * ((size_t)J * N /*y*/ + (size_t)kParts * (NW > 0 ? NW : 1));
    bytes = (bytes + 15) & ~(size_t)15;
    return bytes + kGramBytes;
}

// Tensor-memory columns of one CTA.  Thread tid owns elements tid + e BT,
// e < EPT = ceil(N / BT), of every pair and Lanczos vector.  A warp's block of
// pair columns holds (m + 1) slots x EPT elements x (s re, s im, y re, y im);
// its block of Lanczos columns EPT elements x KM vectors x (re, im), KM = k
// rounded up to a multiple of 4; the up to four warps that share a lane
// quarter take consecutive blocks.  Every row variant with m <= 6 needs at
// most 504 columns for its pairs; the Lanczos vectors go to tensor memory when
// their blocks fit in 512 columns (klz = k steps, else 0).  The allocation is
// the next power of two of the larger need (at least 32).
struct RowShape {
    int threads, ept;  // threads of the CTA, vector elements per thread
    __host__ __device__ int quarter_warps() const { return (threads / 32 + 3) / 4; }
    __host__ __device__ int pair_block(int m) const { return 4 * ept * (m + 1); }
    __host__ __device__ int lanczos_block(int k) const { return 2 * ept * ((k + 3) & ~3); }
    __host__ __device__ int klz(bool lanczos_start, int k) const
    {
        return lanczos_start && k >= 1 && k <= kMaxLanczos && quarter_warps() * lanczos_block(k) <= 512 ? k : 0;
    }
    // z: the row's fields take 2 kRowPts columns more of each warp, after the pairs
    __host__ __device__ int cols(int m, int klz, bool z = false) const
    {
        int need = quarter_warps() * (pair_block(m) + (z ? 2 * kRowPts : 0));
        if (klz > 0) {
            const int lz = quarter_warps() * lanczos_block(klz);
            if (lz > need) need = lz;
        }
        int c = 32;
        while (c < need) c *= 2;
        return c;
    }
};
// Whether the fields z fit beside the pairs without taking residency: as many
// CTAs share an SM as its registers (512 threads) and the pairs alone allow.
__host__ __device__ inline bool row_fields_fit(const RowShape &s, int m, int klz)
{
    const int with = s.cols(m, klz, true), without = s.cols(m, klz), by_regs = 512 / s.threads;
    if (with > 512) return false;
    const int a = 512 / with, b = 512 / without;
    return a >= b || a >= by_regs;
}
// JB masks in the CTA, nloc vector elements
__host__ __device__ inline RowShape row_shape(int N, int JB, int nloc)
{
    const int bt = JB * (N / kRowPts);
    return RowShape{bt, (nloc + bt - 1) / bt};
}

// The same of the variant with one CTA per row.
__host__ __device__ inline int row_ept(int N, int J) { return row_shape(N, J, N).ept; }
__host__ __device__ inline int row_quarter_warps(int N, int J) { return row_shape(N, J, N).quarter_warps(); }
__host__ __device__ inline int row_tmem_block(int N, int J, int m) { return row_shape(N, J, N).pair_block(m); }
__host__ __device__ inline int row_tmem_lanczos_block(int N, int J, int k) { return row_shape(N, J, N).lanczos_block(k); }
__host__ __device__ inline int row_tmem_klz(int N, int J, bool lanczos_start, int k)
{
    return row_shape(N, J, N).klz(lanczos_start, k);
}
__host__ __device__ inline int row_tmem_cols(int N, int J, int m, int klz) { return row_shape(N, J, N).cols(m, klz); }

// No global pair workspace: the pairs are in tensor memory.
__host__ __device__ inline size_t row_pair_stride(int N, int m)
{
    (void)N;
    (void)m;
    return 0;
}

// ZT: between a step's update and the next step's line search the fields z wait
// in tensor memory.  32 registers a thread are then free for both transforms and
// for the sweeps over the pairs, which keep three loads in flight instead of
// spilling or waiting for each: 8192 rows, 20 iterations, J = 4, N = 2048 15.17 ->
// 14.46 ms, N = 1024 10.65 -> 9.39; 4096 rows of N = 4096 (CLU) 21.6 -> 19.6.
template <int N, int COST = COST_INTENSITY, bool CLU = false, bool ZT = true>
__global__ void __launch_bounds__(512, 1) k_solver_row(SolverParams P)
{
    using C = RowCfg<N>;
    constexpr int NT = C::NT, E = C::E, R = C::R, BPT = C::BPT, NCONST = C::NCONST, LBUF = C::LBUF;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // JT masks in all, J of them in this CTA, JC CTAs (rank jr), my slice [lo, lo + nmine)
    const int JT = P.J, J = CLU ? rowc_masks(N, P.J) : P.J, JC = CLU ? JT / J : 1, m = P.m, M = P.M;
    cg::cluster_group cluster = cg::this_cluster();
    const int jr = CLU ? (int)cluster.block_rank() : 0;
    const int SL = (N + JC - 1) / JC, lo = CLU ? jr * N / JC : 0, nmine = CLU ? (jr + 1) * N / JC - lo : N;
    const int BT = J * NT;
    const int NW = BT / 32;
    const int tid = threadIdx.x;
    const int team = tid / NT, ttid = tid - team * NT;
    const int lane = tid & 31, warp = tid >> 5;
    const size_t K = (size_t)JT * N, KL = (size_t)J * N;  // intensities of the row, and of this CTA
    const float JN = (float)K;
    const float gsc = cost_grad_scale(COST);  // the gradient's scale (-4 intensity, 2 amplitude)

    // ---- shared memory ----
    float2 *tws = reinterpret_cast<float2 *>(smem_raw);
    float2 *msk = tws + (NCONST + 1) / 2 * 2;     // [J][N]
    float2 *bufs = msk + (size_t)J * N;           // [J][LBUF]
    float2 *buf = bufs + (size_t)team * LBUF;     // this team's exchange buffer
    // direction p (or the vector being transformed); in a cluster it is gathered
    // in the first exchange buffer, which is free until it has been read
    float2 *X = CLU ? bufs : bufs + (size_t)J * LBUF;
    float2 *ts = CLU ? bufs + (size_t)J * LBUF : X + N;  // t (my slice)
    float2 *gs = ts + SL;                                // g (my slice)
    float2 *Yr = gs + SL;                                // CLU: the peers' sums for my slice [JC - 1][SL]
    float2 *lzG = CLU ? Yr + (size_t)(JC - 1) * SL : X;  // Gram matrix of the Lanczos vectors
    float *ys = reinterpret_cast<float *>(CLU ? lzG + kMaxLanczos * kMaxLanczos : gs + SL);  // [J][N] intensities (scaled)
    float *red = ys + (size_t)J * N;                // [kParts][NW]
    float *part = red + kParts * NW;                // CLU: [2][JC][kParts]
    Gram &Gm = *reinterpret_cast<Gram *>(
        smem_raw + ((reinterpret_cast<unsigned char *>(CLU ? part + 2 * JC * kParts : part) - smem_raw + 15) & ~(size_t)15));

    // L-BFGS pairs in tensor memory: element e (i = tid + e BT) of the pair in
    // slot a at columns tcol(a, e) .. + 3 (s, then y)
    __shared__ uint32_t tmem_base;
    const RowShape shape = row_shape(N, J, SL);
    const int klz = shape.klz(P.lanczos && P.init == INIT_SPECTRAL && !P.T_init, P.power_iters);
    const int ncols = shape.cols(m, klz, ZT);
    if (warp == 0) tmem_alloc_warp(&tmem_base, (uint32_t)ncols);
    tmem_fence_before_sync();
    __syncthreads();
    tmem_fence_after_sync();
    const int EPT = shape.ept;
    const uint32_t tquarter = tmem_base + ((uint32_t)(32 * (warp & 3)) << 16);
    const uint32_t tlane = tquarter + (uint32_t)((warp >> 2) * shape.pair_block(m));
    auto tcol = [&](int a, int e) { return tlane + (uint32_t)(4 * (a * EPT + e)); };
    const uint32_t tfields =
        tquarter + (uint32_t)(shape.quarter_warps() * shape.pair_block(m) + (warp >> 2) * 2 * kRowPts);
    auto put_fields = [&](const float2 (&z)[E]) {
        if constexpr (ZT) tmem_st32(tfields, z);
    };
    auto get_fields = [&](float2 (&z)[E]) {
        if constexpr (ZT) {
            tmem_wait_st();
            tmem_ld32(tfields, z);
            tmem_wait_ld();
            tmem_reg_ready(z);
        }
    };

    // f(k, s, y) for element e of the np pairs by age, three loads in flight (six
    // measure the same).  Loads past np repeat one: under a condition their
    // registers would stay taken around the whole loop.
    auto for_pairs = [&](int np, int e, auto &&f) {
        constexpr int Q = 3;
#pragma unroll
        for (int k0 = 0; k0 < kMaxMem; k0 += Q) {
            if (k0 >= np) break;
            uint32_t r[Q][4];
#pragma unroll
            for (int q = 0; q < Q; q++) tmem_ld4(tcol(Gm.slot[k0 + q < np ? k0 + q : k0], e), r[q]);
            tmem_wait_ld();
#pragma unroll
            for (int q = 0; q < Q; q++) {
                tmem_reg_ready(r[q]);
                if (k0 + q < np)
                    f(k0 + q, make_float2(__uint_as_float(r[q][0]), __uint_as_float(r[q][1])),
                      make_float2(__uint_as_float(r[q][2]), __uint_as_float(r[q][3])));
            }
        }
    };

    // twiddles of the passes between the first and the last:
    // tw_p[(r - 1) Ns + j] = exp(-2 pi i r j / (Ns R)) at tw_off(p)
    for (int p = 1; p < C::Plan::P - 1; p++) {
        const int Rp = C::Plan::radix(p), Ns = C::Plan::ns(p), off = C::Plan::tw_off(p);
        for (int i = tid; i < (Rp - 1) * Ns; i += BT) {
            const int r = 1 + i / Ns, j = i - (r - 1) * Ns;
            double s, c;
            sincospi(-2.0 * (double)r * (double)j / ((double)Ns * Rp), &s, &c);
            tws[off + i] = make_float2((float)c, (float)s);
        }
    }
    for (int i = tid; i < J * N; i += BT) msk[i] = P.masks[jr * J * N + i];
    const float2 *dm = msk + (size_t)team * N;  // this team's mask
    const float *yt = ys + (size_t)team * N;    // this team's intensities
    float2 wb[BPT];  // last-pass twiddle bases exp(-2 pi i b / N), b = ttid + i NT
#pragma unroll
    for (int i = 0; i < BPT; i++) {
        double s, c;
        sincospi(-2.0 * (double)(ttid + i * NT) / (double)N, &s, &c);
        wb[i] = make_float2((float)c, (float)s);
    }
    __syncthreads();

    // x <- F(d .* x) and x <- conj(d) .* F^H x for this team's mask.  Only the
    // team's own warps meet inside, so that one team's exchange can run beside
    // another's butterflies (N = 2048, J = 4: 14.74 ms a launch of 20 iterations
    // against 14.97 with block barriers).
    const TeamBarrier<NT> team_bar{1 + team};
    auto fwd = [&](float2 (&x)[E]) {
#pragma unroll
        for (int e = 0; e < E; e++) x[e] = cmul(x[e], dm[ttid + e * NT]);
        block_fft_rbx<N, NT, R, -1>(x, buf, tws, wb, ttid, team_bar);
    };
    auto adj = [&](float2 (&x)[E]) {
        block_fft_rbx<N, NT, R, +1>(x, buf, tws, wb, ttid, team_bar);
#pragma unroll
        for (int e = 0; e < E; e++) x[e] = cmulc(x[e], dm[ttid + e * NT]);
    };
    if constexpr (CLU) cluster.sync();  // every CTA runs before anyone touches its shared memory
    // after a transform every thread has passed its last exchange, so the team
    // buffer is free: park the natural-order result there (unpadded)
    auto park = [&](const float2 (&x)[E]) {
#pragma unroll
        for (int e = 0; e < E; e++) buf[ttid + e * NT] = x[e];
    };
    // sum over this CTA's masks of the parked results, element i of the vector
    auto local_sum = [&](int i) {
        float2 acc = bufs[i];
#pragma unroll
        for (int j = 1; j < kMaxMasks; j++)
            if (j < J) acc = cadd(acc, bufs[j * LBUF + i]);
        return acc;
    };
    // Make the parked results of every mask available to team_sum.  In a cluster
    // each CTA adds its own masks for the peers' slices and pushes the sums
    // into their Yr.  (A cluster barrier follows every read of Yr before the next
    // share: a reduction's, or the gather's of the next vector.)
    auto share = [&]() {
        __syncthreads();
        if constexpr (CLU) {
            for (int o = 0; o < JC; o++) {
                if (o == jr) continue;
                const int b = o * N / JC, n = (o + 1) * N / JC - b;
                float2 *dst = cluster.map_shared_rank(Yr, o) + (size_t)(jr < o ? jr : jr - 1) * SL;
                for (int i = tid; i < n; i += BT) dst[i] = local_sum(b + i);
            }
            cluster.sync();
        }
    };
    // sum over all masks, element i of my slice, times s (CTAs in rank order)
    auto team_sum = [&](int i, float s) {
        float2 acc = local_sum(lo + i);
        if constexpr (CLU) {
            float2 tot = make_float2(0.f, 0.f);
            for (int r = 0; r < JC; r++) tot = cadd(tot, r == jr ? acc : Yr[(size_t)(r < jr ? r : r - 1) * SL + i]);
            acc = tot;
        }
        return cscale(acc, s);
    };
    auto load_team = [&](const float2 *src, float2 (&x)[E]) {
#pragma unroll
        for (int e = 0; e < E; e++) x[e] = src[ttid + e * NT];
    };
    // x <- the whole vector whose slices are src.  In a cluster the slices are
    // first pushed into every CTA's X, once every CTA is done with the parked
    // results there (X is its first exchange buffer).
    auto load_vec = [&](const float2 *src, float2 (&x)[E]) {
        if constexpr (CLU) {
            cluster.sync();
            for (int o = 0; o < JC; o++) {
                float2 *dst = cluster.map_shared_rank(X, o) + lo;
                for (int i = tid; i < nmine; i += BT) dst[i] = src[i];
            }
            cluster.sync();
            load_team(X, x);
            __syncthreads();  // X is read before the transform reuses it
        } else {
            __syncthreads();
            load_team(src, x);
        }
    };
    // Block-wide sums of nv <= 32 per-thread values: warp sums, then thread k
    // adds the NW warp sums of value k in warp order into Gm.red[k].  With
    // all = false only warp 0 (threads 0 .. 31) goes on to read the sums, so
    // a warp barrier replaces the block barrier after them.
    int sel = 0;
    auto block_reduce = [&](float (&v)[32], int nv, bool all = true) {
        if (nv <= 6) {
            // constant indices only: a runtime index would move v to local memory
#pragma unroll
            for (int k = 0; k < 6; k++) {
                if (k < nv) {
                    const float t = warp_sum(v[k]);
                    if (lane == 0) red[k * NW + warp] = t;
                }
            }
        } else {
            warp_reduce32(v, lane);
            if (lane < nv) red[lane * NW + warp] = v[0];
        }
        __syncthreads();
        float acc = 0.f;
        if (tid < nv) {
            // at most 16 warps, the loads in flight together; the amplitude cost's line
            // search, which holds its fields through a dozen reductions an
            // iteration, has registers for four at a time
            constexpr int U = COST == COST_AMPLITUDE ? 4 : 16;
#pragma unroll
            for (int w0 = 0; w0 < 16; w0 += U) {
                if (w0 >= NW) break;
#pragma unroll
                for (int w = w0; w < w0 + U; w++)
                    if (w < NW) acc += red[tid * NW + w];
            }
        }
        if constexpr (CLU) {
            // the CTAs' sums into every CTA's part, then added in rank order
            // (two buffers in turn, as in k_solver)
            float *pb = part + sel * JC * kParts;
            sel ^= 1;
            if (tid < nv)
                for (int o = 0; o < JC; o++) cluster.map_shared_rank(pb, o)[jr * kParts + tid] = acc;
            cluster.sync();
            if (tid < nv) {
                acc = 0.f;
#pragma unroll
                for (int o = 0; o < kMaxMasks / 2; o++)
                    if (o < JC) acc += pb[o * kParts + tid];
            }
        }
        if (tid < nv) Gm.red[tid] = acc;
        if (all) __syncthreads();
        else __syncwarp();
    };

    while (true) {
        if constexpr (CLU) {
            if (jr == 0 && tid == 0) {
                const int r = (int)atomicAdd(P.queue, 1u);
                for (int o = 0; o < JC; o++) cluster.map_shared_rank(&Gm.row, o)[0] = r;
            }
            cluster.sync();
        } else {
            if (tid == 0) Gm.row = (int)atomicAdd(P.queue, 1u);
            __syncthreads();
        }
        const int row = Gm.row;
        if (row >= M) break;  // nobody touches another CTA's shared memory after this barrier

        // ---- intensities, their sum and finiteness ----
        {
            float pv[32] = {0.f};
            const float *yr = P.y + (size_t)row * K + jr * KL;
            for (size_t i = tid; i < KL; i += BT) {
                const float v = yr[i];
                ys[i] = v;
                if (isfinite(v)) pv[0] += v;
                else pv[1] += 1.f;
            }
            block_reduce(pv, 2);
            if (tid == 0) {
                Gm.status = ROW_MAXITER;
                Gm.done = 0;
                Gm.np = 0;
                Gm.f = 0.f;
                Gm.stop = 0;
                Gm.early = 0;
                Gm.sumy = Gm.red[0];
                const int js = row_scale_exp(Gm.red[0], (int)K);
                Gm.yscale = ldexpf(1.f, -2 * js);
                Gm.tsc = ldexpf(1.f, js);
                if (Gm.red[1] > 0.f || !isfinite(Gm.red[0])) { Gm.status = ROW_NUMERIC; Gm.stop = 1; Gm.early = 1; }
                else if (Gm.red[0] == 0.f) { Gm.status = ROW_ZERO; Gm.stop = 1; Gm.early = 1; }
            }
            __syncthreads();
            // the row is solved with y 4^-j and t 2^-j (exact scales; see k_solver)
            const float ysc = Gm.yscale;
            for (size_t i = tid; i < KL; i += BT) ys[i] *= ysc;
            __syncthreads();
        }
        const float sumy = Gm.sumy * Gm.yscale;
        float2 z[E];
#pragma unroll
        for (int e = 0; e < E; e++) z[e] = make_float2(0.f, 0.f);

        if (!Gm.stop) {
            // ---- initialisation ----
            if (P.T_init) {
                const float tinv = 1.f / Gm.tsc;
                for (int i = tid; i < nmine; i += BT) ts[i] = cscale(P.T_init[(size_t)row * N + lo + i], tinv);
            } else if (P.init == INIT_BP) {
                float2 u[E];
#pragma unroll
                for (int e = 0; e < E; e++) u[e] = make_float2(sqrtf(fmaxf(yt[ttid + e * NT], 0.f)), 0.f);
                adj(u);
                park(u);
                share();
                for (int i = tid; i < nmine; i += BT) ts[i] = team_sum(i, 1.f / JN);
            } else {
                // seed: the proposed start (learned initialiser) where it is
                // finite and nonzero, else the Philox vector
                bool seeded = false;
                if (P.T_cand && P.seed_from_cand) {
                    float pv[32] = {0.f};
                    for (int i = tid; i < nmine; i += BT) {
                        const float2 v = P.T_cand[(size_t)row * N + lo + i];
                        ts[i] = v;
                        pv[0] += cabs2(v);
                    }
                    block_reduce(pv, 1);
                    seeded = isfinite(Gm.red[0]) && Gm.red[0] > 0.f;
                    if (seeded && jr == 0 && tid == 0 && P.cand_wins) atomicAdd(P.cand_wins, 1u);
                }
                if (!seeded)
                    for (int i = tid; i < nmine; i += BT) ts[i] = philox_cnormal(P.seed, (uint32_t)row, (uint32_t)(lo + i));
                if (P.init == INIT_SPECTRAL && P.lanczos) {
                    const float mean = sumy / (float)K;
                    auto applyA = [&]() {
                        float2 x[E];
                        load_vec(ts, x);
                        fwd(x);
#pragma unroll
                        for (int e = 0; e < E; e++) {
                            float tv = yt[ttid + e * NT] / mean;
                            if (P.clip > 0.f && tv > P.clip) tv = P.clip;
                            x[e] = cscale(x[e], tv);
                        }
                        adj(x);
                        park(x);
                        share();
                        for (int i = tid; i < nmine; i += BT) gs[i] = team_sum(i, 1.f / JN);
                        __syncthreads();
                    };
                    float2 *V = P.krylov + (size_t)(blockIdx.x / JC) * lanczos_region(N, P.power_iters);
                    // (the direction p is not in use yet: one CTA per row keeps
                    // the Gram matrix of the Lanczos vectors in its buffer X)
                    if (klz)
                        lanczos_start_tmem(klz, nmine, EPT,
                                           tquarter + (uint32_t)((warp >> 2) * shape.lanczos_block(klz)), ts,
                                           gs, lzG, Gm.red, &Gm.SY[0][0], &Gm.YY[0][0], applyA, block_reduce);
                    else
                        lanczos_start(P.power_iters, nmine, ts, gs, V + lo, (size_t)N,
                                      V + (size_t)P.power_iters * N + jr * kMaxLanczos * kMaxLanczos, Gm.red,
                                      &Gm.SY[0][0], &Gm.YY[0][0], applyA, block_reduce);
                } else if (P.init == INIT_SPECTRAL) {
                    const float mean = sumy / (float)K;
                    for (int it = 0; it < P.power_iters; it++) {
                        // t <- A t, A = Q^H diag(tau) Q / (J N), tau = min(y / mean, clip);
                        // the norm is restored every 8th step and at the end
                        float2 x[E];
                        load_vec(ts, x);
                        fwd(x);
#pragma unroll
                        for (int e = 0; e < E; e++) {
                            float tv = yt[ttid + e * NT] / mean;
                            if (P.clip > 0.f && tv > P.clip) tv = P.clip;
                            x[e] = cscale(x[e], tv);
                        }
                        adj(x);
                        park(x);
                        share();
                        const bool renorm = ((it & 7) == 7) || (it == P.power_iters - 1);
                        float pv[32] = {0.f};
                        for (int i = tid; i < nmine; i += BT) {
                            const float2 s = team_sum(i, 1.f / JN);
                            ts[i] = s;
                            pv[0] = fmaf(s.x, s.x, fmaf(s.y, s.y, pv[0]));
                        }
                        if (renorm) {
                            block_reduce(pv, 1);
                            const float nrm = Gm.red[0];
                            const float inv = nrm > 0.f ? rsqrtf(nrm) : 0.f;
                            for (int i = tid; i < nmine; i += BT) ts[i] = cscale(ts[i], inv);
                        }
                    }
                }
                // rescale to the Parseval norm ||t||^2 = sum(y) / (J N)
                float pv[32] = {0.f};
                for (int i = tid; i < nmine; i += BT) pv[0] += cabs2(ts[i]);
                block_reduce(pv, 1);
                const float nrm = Gm.red[0];
                const float sc = nrm > 0.f ? sqrtf(sumy / JN) / sqrtf(nrm) : 0.f;
                for (int i = tid; i < nmine; i += BT) ts[i] = cscale(ts[i], sc);
            }

            // ---- per-row selection: a proposed start (learned initialiser) against this one ----
            if (P.T_cand && P.judge_cand) {
                const float tinv = 1.f / Gm.tsc;
                for (int i = tid; i < nmine; i += BT) gs[i] = cscale(P.T_cand[(size_t)row * N + lo + i], tinv);
                float fv[2];
                for (int c = 0; c < 2; c++) {  // f at the start above, then at the proposal
                    float2 x[E];
                    load_vec(c == 0 ? ts : gs, x);
                    fwd(x);
                    float pv[32] = {0.f};
#pragma unroll
                    for (int e = 0; e < E; e++) {
                        cost_coef(COST, x[e], yt[ttid + e * NT], pv[0]);
                    }
                    block_reduce(pv, 1);
                    fv[c] = Gm.red[0];
                }
                if (fv[1] < fv[0]) {  // NaN proposals lose
                    for (int i = tid; i < nmine; i += BT) ts[i] = gs[i];
                    if (jr == 0 && tid == 0 && P.cand_wins) atomicAdd(P.cand_wins, 1u);
                }
            }

            // ---- f and gradient at the start ----
            {
                load_vec(ts, z);
                fwd(z);
                put_fields(z);
                float2 u[E];
                float pv[32] = {0.f};
#pragma unroll
                for (int e = 0; e < E; e++) u[e] = cscale(z[e], cost_coef(COST, z[e], yt[ttid + e * NT], pv[0]));
                adj(u);
                park(u);
                share();
                for (int i = tid; i < nmine; i += BT) {
                    const float2 g = team_sum(i, gsc);
                    gs[i] = g;
                    pv[1] += cabs2(g);
                }
                block_reduce(pv, 2);
                if (warp == 0) {
                    if (lane == 0) {
                        Gm.f = Gm.red[0];
                        Gm.gg = Gm.red[1];
                        Gm.np = 0;
                        if (!isfinite(Gm.f) || !isfinite(Gm.gg)) { Gm.status = ROW_NUMERIC; Gm.stop = 1; }
                        else if (P.iters > 0 && (Gm.f == 0.f || Gm.gg == 0.f)) { Gm.status = ROW_CONVERGED; Gm.stop = 1; }
                    }
                    lbfgs_reset(Gm, lane);
                }
                __syncthreads();
            }

            // ---- L-BFGS iterations ----
            for (int it = 0; it < P.iters && !Gm.stop; it++) {
                const int np = Gm.np;
                const int sn_slot = Gm.slot[np];  // the free slot (age np) of the new pair
                // A: direction p = -(gamma g + sum c1 s + sum c2 y) into X
                {
                    const float gam = Gm.gamma;
                    // every thread runs all EPT steps (the tensor-memory loads
                    // are warp-wide); steps past N only load
                    tmem_fence_after_sync();
#pragma unroll 1
                    for (int e = 0; e < EPT; e++) {
                        const int i = tid + e * BT;
                        const bool in = i < nmine;
                        float2 acc = in ? cscale(gs[i], gam) : make_float2(0.f, 0.f);
                        for_pairs(np, e, [&](int k, float2 sa, float2 ya) {
                            const float c1 = Gm.c1[k], c2 = Gm.c2[k];
                            acc.x = fmaf(c1, sa.x, fmaf(c2, ya.x, acc.x));
                            acc.y = fmaf(c1, sa.y, fmaf(c2, ya.y, acc.y));
                        });
                        if constexpr (CLU) {
                            // to every CTA; my own copy waits in the new pair's
                            // cells, X being an exchange buffer until then
                            if (in)
                                for (int o = 0; o < JC; o++)
                                    cluster.map_shared_rank(X, o)[lo + i] = make_float2(-acc.x, -acc.y);
                            tmem_st2(tcol(sn_slot, e), -acc.x, -acc.y);
                        } else {
                            if (in) X[i] = make_float2(-acc.x, -acc.y);
                        }
                    }
                    if constexpr (CLU) tmem_wait_st();
                }
                if constexpr (CLU) cluster.sync();
                else __syncthreads();
                // C: w = F(d .* p)
                float2 w[E];
                load_team(X, w);
                if constexpr (CLU) __syncthreads();  // X is read before the transform reuses it
                fwd(w);
                get_fields(z);
                // D: the step -- the amplitude cost's line search, or the quartic's exact minimiser
                if constexpr (COST == COST_AMPLITUDE) {
                    const float al = amp_line_search(
                        z, w, [&](int e) { return yt[ttid + e * NT]; }, [](int) { return true; }, block_reduce,
                        Gm.red, Gm.red + 16);
                    if (tid == 0) {
                        Gm.alpha = al;
                        if (!isfinite(al)) { Gm.status = ROW_NUMERIC; Gm.stop = 1; }
                        else if (al == 0.f) { Gm.status = ROW_CONVERGED; Gm.stop = 1; }
                    }
                    __syncthreads();
                } else {
                    float pv[32] = {0.f};
#pragma unroll
                    for (int e = 0; e < E; e++) {
                        const float a = cdotr(z[e], w[e]);
                        const float b = cabs2(w[e]);
                        const float r = yt[ttid + e * NT] - cabs2(z[e]);
                        pv[0] = fmaf(r, r, pv[0]);
                        pv[1] = fmaf(-4.f * r, a, pv[1]);
                        pv[2] += fmaf(4.f * a, a, -2.f * r * b);
                        pv[3] = fmaf(4.f * a, b, pv[3]);
                        pv[4] = fmaf(b, b, pv[4]);
                    }
                    block_reduce(pv, 5, false);
                    if (warp == 0) {
                        const float al = quartic_argmin_warp(Gm.red, lane);
                        if (lane == 0) {
                            Gm.alpha = al;
                            if (!isfinite(al)) { Gm.status = ROW_NUMERIC; Gm.stop = 1; }
                            else if (al == 0.f) { Gm.status = ROW_CONVERGED; Gm.stop = 1; }
                        }
                    }
                    __syncthreads();
                }
                if (Gm.stop) break;
                const float al = Gm.alpha;
                // E: fields, residual, t += a p, then the adjoint
                float2 u[E];
                float fpart = 0.f;
#pragma unroll
                for (int e = 0; e < E; e++) {
                    z[e] = make_float2(fmaf(al, w[e].x, z[e].x), fmaf(al, w[e].y, z[e].y));
                    u[e] = cscale(z[e], cost_coef(COST, z[e], yt[ttid + e * NT], fpart));
                }
                put_fields(z);
                adj(u);
                park(u);
                share();
                // G: new gradient, new pair, batched dot products
                {
                    float pv[32];
#pragma unroll
                    for (int k = 0; k < 32; k++) pv[k] = 0.f;
                    float dn[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
                    for (int e = 0; e < EPT; e++) {
                        const int i = tid + e * BT;
                        const bool in = i < nmine;
                        float2 gn = make_float2(0.f, 0.f), sn = gn, yn = gn, pn = gn;
                        if constexpr (CLU) {
                            uint32_t r[2];
                            tmem_ld2(tcol(sn_slot, e), r);
                            tmem_wait_ld();
                            tmem_reg_ready(r);
                            pn = make_float2(__uint_as_float(r[0]), __uint_as_float(r[1]));
                        }
                        if (in) {
                            gn = team_sum(i, gsc);
                            if constexpr (!CLU) pn = X[i];
                            sn = cscale(pn, al);
                            yn = csub(gn, gs[i]);
                            ts[i] = cadd(ts[i], sn);
                            gs[i] = gn;
                        }
                        tmem_st4(tcol(sn_slot, e), sn.x, sn.y, yn.x, yn.y);
                        for_pairs(np, e, [&](int k, float2 sa, float2 ya) {
                            pv[4 * k + 0] += cdotr(sa, yn);  // live pairs by age
                            pv[4 * k + 1] += cdotr(ya, yn);
                            pv[4 * k + 2] += cdotr(sa, gn);
                            pv[4 * k + 3] += cdotr(ya, gn);
                        });
                        // the new pair (age np), added to its place after the loop
                        dn[0] += cdotr(sn, yn);
                        dn[1] += cdotr(yn, yn);
                        dn[2] += cdotr(sn, gn);
                        dn[3] += cdotr(yn, gn);
                        pv[kIdxSS] += cabs2(sn);
                        pv[kIdxGG] += cabs2(gn);
                    }
                    tmem_wait_st();  // the new pair is read back from the next iteration on
                    tmem_fence_before_sync();
#pragma unroll
                    for (int k = 0; k < kSlots; k++)
                        if (k == np) {
#pragma unroll
                            for (int q = 0; q < 4; q++) pv[4 * k + q] = dn[q];
                        }
                    pv[kIdxF] = fpart;
                    block_reduce(pv, kParts, false);
                    if (warp == 0) lbfgs_gram_update(Gm, lane, m, it, P.iters, P.tol);
                    __syncthreads();
                }
            }
        }

        // ---- outputs (rows decided before initialisation come back as zero) ----
        const bool early = Gm.early != 0;
        const float tsc = Gm.tsc;
        for (int i = tid; i < nmine; i += BT)
            P.T_out[(size_t)row * N + lo + i] = early ? make_float2(0.f, 0.f) : cscale(ts[i], tsc);
        if (jr == 0 && tid == 0) {
            if (P.row_status) P.row_status[row] = Gm.status;
            if (P.row_iters) P.row_iters[row] = Gm.done;
            if (P.row_loss) {
                // the intensity cost scales as y^2 = t^4, the amplitude cost as y = t^2
                const double f2 = COST == COST_AMPLITUDE ? (double)tsc * tsc : (double)tsc * tsc * tsc * tsc;
                P.row_loss[row] = early ? (Gm.status == ROW_ZERO ? 0.f : __int_as_float(0x7fc00000))
                                        : (float)((double)Gm.f * f2);
            }
        }
        if (P.Zd) {
            if (early) {
#pragma unroll
                for (int e = 0; e < E; e++) z[e] = make_float2(0.f, 0.f);
            } else {
                get_fields(z);
            }
#pragma unroll
            for (int e = 0; e < E; e++) {
                const int pat = (jr * J + team) * N + ttid + e * NT;
                if (pat < P.Nd) P.Zd[(size_t)pat * M + row] = cscale(z[e], tsc);
            }
        }
        __syncthreads();
    }
    tmem_fence_before_sync();
    __syncthreads();
    if (warp == 0) {
        tmem_fence_after_sync();
        tmem_dealloc_warp(tmem_base, (uint32_t)ncols);
    }
}

// Shared memory and resident CTAs per SM of a launch.  Every CTA holds
// RowShape::cols columns of the SM's 512 for its whole life, so at most
// 512 / cols CTAs may share an SM; where registers and shared memory would
// let more in, the shared-memory request is raised until they do not, and no
// allocation has to wait for the columns of another CTA of the same launch.
// (A concurrent launch on another stream that holds tensor memory can delay
// an allocation until its CTAs on that SM exit; they never wait on this one.)
template <int N, int COST, bool ZT>
cudaError_t row_launch_shape(int J, int m, int cols, size_t *smem_out, int *per_sm_out)
{
    const int BT = J * RowCfg<N>::NT;
    const int cap = 512 / cols;
    const auto kernel = k_solver_row<N, COST, false, ZT>;
    size_t sm = row_smem<N>(J, m);
    int dev = 0, occ = 0, sm_per_mp = 0, optin = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sm_per_mp, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev)) != cudaSuccess)
        return e;
    if ((e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return e;
    for (int pass = 0; pass < 2; pass++) {
        if (sm > (size_t)optin) return cudaErrorInvalidConfiguration;
        if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm)) !=
            cudaSuccess)
            return e;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, BT, sm)) != cudaSuccess)
            return e;
        if (occ < 1) return cudaErrorInvalidConfiguration;
        if (occ <= cap) break;
        if (pass == 1) return cudaErrorInvalidConfiguration;
        const size_t need = (size_t)sm_per_mp / (size_t)(cap + 1) + 1;
        if (need > sm) sm = (need + 15) & ~(size_t)15;
    }
    *smem_out = sm;
    *per_sm_out = occ;
    return cudaSuccess;
}

template <int N, int COST, bool ZT>
cudaError_t launch_solver_row_zt(const SolverParams &p, cudaStream_t s, int *ctas_out)
{
    if (!row_variant_fits(N, p.J) || p.m < 1 || p.m > kMaxMem) return cudaErrorInvalidValue;
    const int BT = p.J * RowCfg<N>::NT;
    size_t sm = 0;
    int occ = 0, dev = 0, nsm = 0;
    const int klz = row_tmem_klz(N, p.J, p.lanczos && p.init == INIT_SPECTRAL && !p.T_init, p.power_iters);
    cudaError_t e = row_launch_shape<N, COST, ZT>(p.J, p.m, row_shape(N, p.J, N).cols(p.m, klz, ZT), &sm, &occ);
    if (e != cudaSuccess) return e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    long long grid = (long long)occ * nsm;
    if (grid > p.M) grid = p.M;
    if (grid > p.pair_ctas) grid = p.pair_ctas;  // the resident CTAs the handle sized its workspaces for
    if (p.lanczos && p.init == INIT_SPECTRAL && grid > p.krylov_units) grid = p.krylov_units;
    if (grid < 1) grid = 1;
    if (ctas_out) *ctas_out = (int)grid;
    k_solver_row<N, COST, false, ZT><<<(int)grid, BT, sm, s>>>(p);
    return cudaGetLastError();
}

// The fields in tensor memory where they fit beside the pairs, else in registers
// (solver_row_regs.cu).
template <int N, int COST = COST_INTENSITY>
cudaError_t launch_solver_row_t(const SolverParams &p, cudaStream_t s, int *ctas_out)
{
    if (!row_variant_fits(N, p.J) || p.m < 1 || p.m > kMaxMem) return cudaErrorInvalidValue;
    const int klz = row_tmem_klz(N, p.J, p.lanczos && p.init == INIT_SPECTRAL && !p.T_init, p.power_iters);
    if (!row_fields_fit(row_shape(N, p.J, N), p.m, klz)) return launch_solver_row_regs(N, p, s, ctas_out);
    return launch_solver_row_zt<N, COST, true>(p, s, ctas_out);
}

// The row layout over clusters of JC CTAs.  Shared memory (above 114 KB for
// every supported shape; raised to that otherwise) keeps it at one such CTA per
// SM, so no tensor-memory allocation waits for a CTA of another cluster, which
// might wait for this one in turn.
template <int N, int COST = COST_INTENSITY>
cudaError_t launch_solver_rowc_t(const SolverParams &p, cudaStream_t s, int *clusters_out)
{
    const int JB = rowc_masks(N, p.J);
    if (JB == 0 || p.m < 1 || p.m > kMaxMem) return cudaErrorInvalidValue;
    const int JC = p.J / JB;
    if (!row_fields_fit(row_shape(N, JB, (N + JC - 1) / JC), p.m, 0)) return cudaErrorInvalidValue;
    size_t sm = rowc_smem<N>(p.J);
    const auto kernel = k_solver_row<N, COST, true>;
    if (sm < 116 * 1024) sm = 116 * 1024;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = JC;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.blockDim = dim3(JB * RowCfg<N>::NT);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.gridDim = dim3(JC);
    int maxc = 0;
    e = cudaOccupancyMaxActiveClusters(&maxc, kernel, &cfg);
    if (e != cudaSuccess) return e;
    if (maxc < 1) return cudaErrorInvalidConfiguration;
    int nc = maxc < p.M ? maxc : p.M;
    if (p.lanczos && p.init == INIT_SPECTRAL && nc > p.krylov_units) nc = p.krylov_units;  // one region each
    if (nc < 1) nc = 1;
    cfg.gridDim = dim3(nc * JC);
    if (clusters_out) *clusters_out = nc;
    return cudaLaunchKernelEx(&cfg, kernel, p);
}

}  // namespace tmr
