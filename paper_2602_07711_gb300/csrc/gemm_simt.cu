// Complex64 GEMM on the CUDA cores (FFMA): the eigenvector transforms of EigT steps 2 and 4
// (Sec. 4.1, Eq. EIG_SOLVER) in the plain complex64 mode.
//   C[b] = alpha * A[b] B[b],  A: M x K, B: K x N, C: M x N, row-major, batch strides sA/sB/sC.
// x-pass (right multiply by V_x^-T or V_x^T):  A = the grid viewed as (N_y N_z) x N_x rows, B = operand.
// y-pass (left multiply by V_y^-1 or V_y):      A = operand (sA = 0), B = slice l, batch = N_z.
//
// The FP32 pipe bounds it (8 flop per complex product), so the work is arranged to issue little else: a thread
// holds TM x TN complex accumulators as packed f32x2 pairs of two rows (real parts, imaginary parts) and multiplies
// in packed instructions, two per product, which take two cycles of the pipe and one issue slot each.  A is staged
// as planes of real and imaginary parts, so that a pair of rows comes from shared memory as an operand; only B's
// values are duplicated (and negated) in registers.  (Pairs of (re, im) need both operands duplicated or swapped:
// as many register moves as products, 353 us for the x-pass below.)  NW warps of 4 x 8 lanes share a tile of
// 4 NW TM x 8 TN outputs; K is staged 16 at a time through a three-stage cp.async ring.  Every component is summed in
// the order of k by the same four multiply-adds, so a result does not depend on the tile.  The tile is chosen per
// call: grid sizes are seldom multiples of one (at 200^3, 64 x 64 tiles left 39% of the y-pass to padding).
// Measured: the passes at 200^3 405/493 us (4 x 4 accumulators, scalar FMAs, no ring: 28 TFLOP/s) -> 244/302 us
// (52 and 42 TFLOP/s; 200 rows are 6.25 warps).  Small grids: 8.1/7.6 us at 32^3 -> 4.3/3.9 us.
#include "common.cuh"
#include "packed.cuh"

namespace {
constexpr int GK = 16, GST = 3;
template <int TM, int TN, int NW>
struct Tile {
    static constexpr int BM = 4 * NW * TM, BN = 8 * TN, NT = 32 * NW;
    static constexpr int LDA = BM + 4;                       // floats per staged k of a plane of A (16-byte rows)
    static constexpr int STAGE = GK * (2 * LDA + 2 * BN);    // floats
    static constexpr size_t SMEM = (size_t)GST * STAGE * sizeof(float);
};

// copies of 4 and 8 bytes, zeros where !ok
__device__ __forceinline__ void gcp4(float* dst, const float* src, bool ok) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst), n = ok ? 4u : 0u;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void gcp8(float* dst, const float2* src, bool ok) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst), n = ok ? 8u : 0u;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(d), "l"(src), "r"(n) : "memory");
}

// TM rows of a thread from a staged plane of A, as pairs of rows: quads at 4 ly + 16 i, then a pair for TM % 4
template <int TM>
__device__ __forceinline__ void load_a(float2 (&v)[TM / 2], const float* row, int ly) {
#pragma unroll
    for (int i = 0; i < TM / 4; ++i) {
        const float4 w = *reinterpret_cast<const float4*>(row + 16 * i + 4 * ly);
        v[2 * i] = make_float2(w.x, w.y);
        v[2 * i + 1] = make_float2(w.z, w.w);
    }
    if (TM % 4) v[TM / 2 - 1] = *reinterpret_cast<const float2*>(row + 16 * (TM / 4) + 2 * ly);
}
// TN columns from a staged row of B: pairs at 2 lx + 16 j, then one for odd TN
template <int TN>
__device__ __forceinline__ void load_b(float2 (&v)[TN], const float2* row, int lx) {
#pragma unroll
    for (int j = 0; j < TN / 2; ++j) {
        const float4 w = *reinterpret_cast<const float4*>(row + 16 * j + 2 * lx);
        v[2 * j] = make_float2(w.x, w.y);
        v[2 * j + 1] = make_float2(w.z, w.w);
    }
    if (TN & 1) v[TN - 1] = row[16 * (TN / 2) + lx];
}

template <int TM, int TN, int NW>
__global__ void __launch_bounds__(32 * NW, TM * TN > 24 ? 2 : 4)
cgemm_kernel(int M, int N, int K, const float2* __restrict__ A, long lda, long sA, const float2* __restrict__ B, long ldb,
             long sB, float2* __restrict__ C, long ldc, long sC, float alpha, const double* alpha_dev, int aidx, int rows_per,
             int astride) {
    typedef Tile<TM, TN, NW> T;
    extern __shared__ float4 gsm[];
    float* ring = reinterpret_cast<float*>(gsm);
    const int tid = threadIdx.x, warp = tid >> 5, ly = (tid >> 3) & 3, lx = tid & 7;
    const int m0 = blockIdx.y * T::BM, n0 = blockIdx.x * T::BN;
    A += blockIdx.z * sA;
    B += blockIdx.z * sB;
    C += blockIdx.z * sC;
    const int nk = (K + GK - 1) / GK;
    auto fetch = [&](int kb) {
        if (kb < nk) {
            float* As = ring + (kb % GST) * T::STAGE;
            float* Bs = As + 2 * GK * T::LDA;
            // A: 16 consecutive threads take the 16 k of a row
#pragma unroll
            for (int q = 0; q < T::BM * GK / T::NT; ++q) {
                const int e = tid + T::NT * q, r = e >> 4, kk = e & 15, gr = m0 + r, gk = kb * GK + kk;
                const bool ok = gr < M && gk < K;
                const float* src = reinterpret_cast<const float*>(A + (ok ? (long)gr * lda + gk : 0));
                gcp4(As + kk * T::LDA + r, src, ok);
                gcp4(As + (GK + kk) * T::LDA + r, src + 1, ok);
            }
#pragma unroll
            for (int q = 0; q < (T::BN * GK + T::NT - 1) / T::NT; ++q) {
                const int e = tid + T::NT * q, kk = e / T::BN, c = e % T::BN, gk = kb * GK + kk, gc = n0 + c;
                const bool ok = gk < K && gc < N;
                if (T::BN * GK % T::NT == 0 || kk < GK)
                    gcp8(Bs + 2 * (kk * T::BN + c), B + (ok ? (long)gk * ldb + gc : 0), ok);
            }
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    float2 re[TM / 2][TN], im[TM / 2][TN];
#pragma unroll
    for (int i = 0; i < TM / 2; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) re[i][j] = im[i][j] = make_float2(0.f, 0.f);
    grid_wait();
    grid_trigger();
    for (int b = 0; b < GST - 1; ++b) fetch(b);
    for (int kb = 0; kb < nk; ++kb) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(GST - 2) : "memory");
        __syncthreads();          // stage kb landed for every thread; the stage of kb - 1 is free
        fetch(kb + GST - 1);
        if (m0 + warp * 4 * TM >= M) continue;   // rows of padding only: leave the pipe to the other warps
        const float* As = ring + (kb % GST) * T::STAGE + warp * 4 * TM;
        const float2* Bs = reinterpret_cast<const float2*>(ring + (kb % GST) * T::STAGE + 2 * GK * T::LDA);
#pragma unroll
        for (int kk = 0; kk < GK; ++kk) {
            float2 ar[TM / 2], ai[TM / 2], b[TN];
            load_a<TM>(ar, As + kk * T::LDA, ly);
            load_a<TM>(ai, As + (GK + kk) * T::LDA, ly);
            load_b<TN>(b, Bs + kk * T::BN, lx);
#pragma unroll
            for (int j = 0; j < TN; ++j) {
                const float2 br = bc2(b[j].x), bi = bc2(b[j].y), bn = bc2(-b[j].y);
#pragma unroll
                for (int i = 0; i < TM / 2; ++i) {
                    re[i][j] = fma2(ar[i], br, re[i][j]);
                    re[i][j] = fma2(ai[i], bn, re[i][j]);
                    im[i][j] = fma2(ar[i], bi, im[i][j]);
                    im[i][j] = fma2(ai[i], br, im[i][j]);
                }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int r = i < TM / 4 * 4 ? 16 * (i / 4) + 4 * ly + i % 4 : 16 * (TM / 4) + 2 * ly + i % 2;
        const int gr = m0 + warp * 4 * TM + r;
        if (gr >= M) continue;
        float al = alpha;
        if (alpha_dev) al *= (float)alpha_dev[aidx + (rows_per > 0 ? (gr / rows_per) * astride : 0)];
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            const int gc = n0 + (j < TN / 2 * 2 ? 16 * (j / 2) + 2 * lx + (j & 1) : 16 * (TN / 2) + lx);
            const float x = i & 1 ? re[i / 2][j].y : re[i / 2][j].x, y = i & 1 ? im[i / 2][j].y : im[i / 2][j].x;
            if (gc < N) C[(long)gr * ldc + gc] = make_float2(al * x, al * y);
        }
    }
}

struct Args {
    int M, N, K;
    const float2* A;
    long lda, sA;
    const float2* B;
    long ldb, sB;
    float2* C;
    long ldc, sC;
    int batch;
    float alpha;
    const double* alpha_dev;
    int aidx, rows_per, astride, follows;
};
template <int TM, int TN, int NW>
void run(const Args& a, cudaStream_t s) {
    typedef Tile<TM, TN, NW> T;
    const dim3 grid((a.N + T::BN - 1) / T::BN, (a.M + T::BM - 1) / T::BM, a.batch);
    if (T::SMEM > 48 * 1024)
        cudaFuncSetAttribute(cgemm_kernel<TM, TN, NW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)T::SMEM);
    launch_after(a.follows, cgemm_kernel<TM, TN, NW>, grid, T::NT, T::SMEM, s, a.M, a.N, a.K, a.A, a.lda, a.sA, a.B, a.ldb,
                 a.sB, a.C, a.ldc, a.sC, a.alpha, a.alpha_dev, a.aidx, a.rows_per, a.astride);
}
template <int TM, int NW>
void run_n(const Args& a, int tn, cudaStream_t s) {
    switch (tn) {
        case 8: run<TM, 8, NW>(a, s); break;
        case 7: run<TM, 7, NW>(a, s); break;
        case 6: run<TM, 6, NW>(a, s); break;
        case 5: run<TM, 5, NW>(a, s); break;
        default: run<TM, 4, NW>(a, s);
    }
}
}  // namespace

void launch_cgemm_simt(int M, int N, int K, const float2* A, long lda, long sA, const float2* B, long ldb, long sB,
                       float2* C, long ldc, long sC, int batch, float alpha, const double* alpha_dev, int aidx,
                       cudaStream_t s, int rows_per, int astride, int follows) {
    // The tile with the least time for the whole grid of tiles: an SM works through its share of them at a rate
    // proportional to their area, padding included (of the rows, that of a warp: 32), but no faster than one warp
    // per scheduler; a tile's fixed cost (the first loads, the epilogue) is worth about 1500 outputs.  Widths 64, 56,
    // 48, 40 and 32; ties go to the wider.  32 x 32 tiles serve the small grids, which leave most SMs without a
    // large tile.
    constexpr double SMS = 152.0;
    int bm = 128, tn = 8;
    double best = 1e300;
    auto consider = [&](int m, int n) {
        const int tiles_m = (M + m - 1) / m, rows = (M + 31) / 32 * 32;
        const double share = ceil((double)tiles_m * ((N + 8 * n - 1) / (8 * n)) * batch / SMS);
        const double t = fmax(share * 8.0 * n * rows / tiles_m, 8.0 * n * m) + share * 1500.0;
        if (t < best) { best = t; bm = m; tn = n; }
    };
    for (int n = 8; n >= 4; --n) consider(128, n);
    consider(32, 4);
    const Args a = {M, N, K, A, lda, sA, B, ldb, sB, C, ldc, sC, batch, alpha, alpha_dev, aidx, rows_per, astride, follows};
    if (bm == 128) run_n<8, 4>(a, tn, s);
    else run<2, 4, 4>(a, s);
}
