// 3x3x3 convolutions of the learned correction on the tcgen05 tensor cores (BF16 operands, FP32 accumulation
// in tensor memory), as implicit GEMMs.  An extension of the method (the paper has no network); the network
// itself lives in learned.cu, the activation layout in cells.cuh.
//
// Layout: activations are cells of 8 channels (16 bytes) on grids with a zero halo, [channel group][z][y][x].
// Consecutive points of a padded plane are consecutive cells, which is the canonical K-major, no-swizzle operand
// layout (a core matrix is 8 points x 16 bytes), and a tap's view of the staged points is the same layout at
// another start address.  So a run of points with everything its 27 taps need is three contiguous pieces of
// memory per channel group, fetched by bulk copies without any gather.  (The layout before, channel-first
// rows transposed into cells by eight warps per tile, made that gather the bound, at 9% of the tensor pipe.)
//
// Forward and data gradient (the same convolution with flipped, transposed weights):
//   out[o][p] = act(bias[o] + sum_{t, i} W(o, i, t) in[i][p + off_t])
//   A tile is R x 128 consecutive points of a padded plane, taken along the flattened (y, x) index, in S consecutive
//   planes: rows follow one another across the halo, so the waste is the two halo points per row and not the
//   remainder of a row to 128.  Per 128 points and plane one accumulator of 128 x Np (Np: outputs padded to 16) in
//   tensor memory, R S Np <= 256 columns, two buffers.
//   The tensor unit bounds it: it takes 64 cycles for an MMA of M = 128, K = 16 with any N up to 128, so N = Np = 32
//   outputs alone used an eighth of its rate (84% busy).  So an MMA takes one view of the points (one input plane,
//   dy, dx) for up to three output planes at once: their accumulators are adjacent columns, and the weights of
//   the three dz are adjacent rows, stored from dz = 2 down.  9 (S + 2) MMAs serve S planes instead of 27 S.
//   The K dimension runs over 16-channel chunks, then the input planes, then dy, dx: every output sums chunk, tap, 16
//   channels in that order whatever R and S are.  A stage is one chunk of one input plane: the points of the tile
//   plus a row and a point on both sides (or three runs for the three dy where rows are longer than a tile); the
//   27 taps' weights of a chunk have two buffers of their own.
//   Persistent, one CTA per SM: warp 0 issues the bulk copies, warps 1 and 10 the MMAs (M = 128, K = 16) of one
//   128-point block each (one warp alone could not issue them fast enough: 118 cycles an MMA), warps 2-9 run the epilogue
//   of the previous tile.
//   Measured at 160^3, width 28: the 84 -> 28 layer 4.14 ms before cells, 1.38 with one output plane per MMA, 1.05 with
//   one MMA warp and four epilogue warps, 0.90 with two and eight, 0.80 since a stage's copies
//   are issued without forming their addresses anew; the forward pass 9.2, 3.17, 2.46, 2.09, 1.89 ms.
// Weight gradient:  gW[o][i][t] = sum_p g[o][p] in[i][p + off_t].
//   Both operands are read as MN-major cells (channels x points): M = output channels (64, or 128), N = all
//   input channels of a block (up to 160), K = 256 points of a flattened plane (the gradient's halo is zero, so
//   rows run on).  A CTA holds the accumulators of one dz and either 9 taps (narrow inputs) or the 3 taps of
//   one dy in tensor memory for its whole share of the points and adds them to gW (FP32 atomics) at the end.
//   The copies bound it: one warp issues a 4 KiB copy per channel group and tile.  Measured on two 96^3 fields, 84 ->
//   28 layer: 0.65 ms with tiles of 256 points, 1.19 ms with 128; 7.6 ms with M = 128 rows of which 28 were used, N =
//   16 inputs at a time and a gathered slab per input chunk.  A training pass: 24.2 -> 3.9 ms.
// Every mbarrier wait is bounded; an expired wait raises HELM_DEV_WAIT, the CTA waits (bounded) for its bulk
// copies and MMAs in flight, frees its tensor memory and exits.
#include "cells.cuh"
#include <algorithm>

namespace {

constexpr long CT_WAIT = 1L << 22;                 // bound of every mbarrier wait (polls)
constexpr int CT_NPMAX = 64;                       // largest padded output-channel count of a launch
constexpr int CT_RMAX = 2;                         // 128-point blocks of a tile at most
constexpr int CT_PLANES = 128;                     // S Np at most: output planes of a tile times outputs
constexpr int CT_THREADS = 192;                    // producer warp, MMA warp, four epilogue warps
constexpr int CV_THREADS = CT_THREADS + 5 * 32;    // convolutions: eight epilogue warps (2 .. 9), one MMA warp per 128-point
                                                   // block (warps 1 and 10)
constexpr int CT_NST = 8;                          // most stages
constexpr int CT_CHUNK = 128;                      // cells of a bulk copy at most (whole runs measured the same)
constexpr int CT_RUN = 3 * (128 * CT_RMAX + 2);    // cells of a staged run at most
constexpr int CT_SMEM = 229376;                    // dynamic shared memory of a CTA at most (224 KiB)
constexpr int WG_KT = 256;                         // points of a weight-gradient tile at most
// Points a CTA sums in tensor memory before it adds to gW.  The accumulators of the tensor cores are FP32 with
// truncation, so long chains of additions lose digits: with one wave of CTAs (112,000 points for the
// 84 -> 28 layer on two 96^3 fields) the gradient moved by 2.8e-5 against chains a quarter as long.
constexpr int WG_POINTS = 16384;

__device__ __forceinline__ uint32_t s32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_init(uint32_t b, uint32_t n) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(b), "r"(n) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint32_t b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(b) : "memory");
}
__device__ __forceinline__ void bar_expect(uint32_t b, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool bar_wait(uint32_t b, uint32_t parity, long limit) {
    for (long it = 0; it < limit; ++it) {
        uint32_t ok;
        asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
                     : "=r"(ok)
                     : "r"(b), "r"(parity)
                     : "memory");
        if (ok) return true;
    }
    return false;
}
// the same by every lane of a warp, with one answer
__device__ __forceinline__ bool warp_wait(uint32_t b, uint32_t parity, long limit) {
    return __all_sync(0xffffffffu, bar_wait(b, parity, limit));
}
// bulk copy global -> shared (16-byte aligned addresses, size a multiple of 16), completion on bar
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t b) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(b)
                 : "memory");
}
// shared-memory matrix descriptor, no swizzle: start, LBO (the stride between 8-element groups along K) and
// SBO (along M or N) in bytes, multiples of 16; a core matrix is 8 rows of 16 contiguous bytes
__device__ __forceinline__ uint64_t ndesc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = (uint64_t)((addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}
// instruction descriptor, kind::f16 with BF16 A and B, FP32 D; a_mn/b_mn = 1 for MN-major operands
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, int a_mn, int b_mn) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16) |
           ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// The MMAs of a stage differ in their start addresses alone, so the issuing thread keeps the upper words of the
// descriptors and adds to the lower ones (start address / 16 in the low 14 bits; shared memory ends below 2^18, so
// the sums stay in the field).  The whole warp runs the issuing loop and `lead` (one elected lane) predicates the
// instruction: the operands are then warp-uniform values in uniform registers.
__device__ __forceinline__ void mma_bf16(uint32_t lead, uint32_t d, uint32_t alo, uint32_t ahi, uint32_t blo, uint32_t bhi,
                                         uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n.reg .pred p, q;\n.reg .b64 da, db;\nmov.b64 da, {%1, %2};\nmov.b64 db, {%3, %4};\nsetp.ne.b32 p, %6, 0;\n"
        "setp.ne.b32 q, %7, 0;\n@q tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n}\n" ::"r"(d), "r"(alo), "r"(ahi),
        "r"(blo), "r"(bhi), "r"(idesc), "r"(acc), "r"(lead));
}
// 1 in one lane of the (converged) warp.  The MMA instructions are predicated on this value directly: the compiler
// then issues them back to back; predicated on lane == 0, or on a copy of this in a variable that other code sets too,
// an MMA took twice as long (weight gradient of 28 -> 28 channels on two 96^3 fields 341 against 781 us)
__device__ __forceinline__ uint32_t elect_one() {
    uint32_t r;
    asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}\n" : "=r"(r));
    return r;
}
__device__ __forceinline__ void mma_commit(uint32_t b) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(b) : "memory");
}
__device__ __forceinline__ void tc_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
    uint32_t r[16];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}
// tensor memory: the MMA warp allocates all 512 columns (one CTA per SM) and frees them at the end
__device__ __forceinline__ void tmem_alloc(uint32_t* slot) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(s32(slot)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_free(uint32_t tmem) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
}

// ---- forward / data gradient ------------------------------------------------------------------------------
struct ConvArgs {
    CellGrid g;
    const bf16* in;      // cells of Gin groups
    int Gin;
    const bf16* wt;      // arranged weights [nkc][9][2][3][Np][8]
    int Np;
    const float* bias;   // [Cout] or NULL
    void* out;
    int Gout, ooff;      // groups of the output tensor, the first output channel in it
    int Cout;            // outputs of this launch (at most 64)
    int relu;
    const bf16* mask;    // CONV_GRAD: cells of Gout groups; the output is 0 where mask <= 0
    float* gb;           // CONV_GRAD: += sum of the output over points, per channel
    int R, S;            // 128-point blocks and planes per tile
    int ntp, nzg;        // tiles per plane, groups of S planes
    int ntiles;
    int dstride;         // staged cells between the views of consecutive dy
    int L;               // staged cells per channel group
    int split;           // three runs (one per dy) instead of one
    int nst, stage;      // stages, bytes of one
    unsigned* status;
};

template <int OUT>
__global__ void __launch_bounds__(CV_THREADS, 1) conv_cells_kernel(const __grid_constant__ ConvArgs a) {
    extern __shared__ __align__(128) unsigned char csm[];
    __shared__ __align__(8) uint64_t full[CT_NST], empty[CT_NST], wfull[2], wempty[2], accf[2], acce[2], drainb;
    __shared__ uint32_t tslot;
    __shared__ int fail_any;
    __shared__ float sbias[CT_NPMAX];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nkc = (a.Gin + 1) / 2;
    const uint32_t base = (s32(csm) + 127u) & ~127u;
    const uint32_t wbytes = 27u * 2u * (uint32_t)a.Np * 16u, sbytes = (uint32_t)a.L * 16u;
    const uint32_t ring = base + 2u * wbytes;   // (wbytes is a multiple of 128)
    if (threadIdx.x == 0) {
        for (int s = 0; s < CT_NST; ++s) { bar_init(s32(&full[s]), 1); bar_init(s32(&empty[s]), CT_RMAX); }
        for (int b = 0; b < 2; ++b) {
            bar_init(s32(&wfull[b]), 1);
            bar_init(s32(&wempty[b]), CT_RMAX);
            bar_init(s32(&accf[b]), CT_RMAX);
            bar_init(s32(&acce[b]), 8);
        }
        bar_init(s32(&drainb), CT_RMAX);
        fail_any = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (threadIdx.x < CT_NPMAX) sbias[threadIdx.x] = a.bias && threadIdx.x < a.Cout ? a.bias[threadIdx.x] : 0.f;
    if (warp == 1) tmem_alloc(&tslot);
    tc_before();
    __syncthreads();
    tc_after();
    const uint32_t tmem = tslot;
    const CellGrid& g = a.g;
    bool ok = true;
    long issued = 0, wissued = 0;   // stages and weight chunks whose copies were issued
    if (warp == 0) {
        // a stage's pieces: runs (two channel groups, times three dy in the split form) in chunks of CT_CHUNK cells, one for
        // each lane (at most 18).  What a lane's copy has in common for all stages is formed here: the time from a free
        // stage to its copies is on the pipeline's path (a division and a product more per stage cost 3%)
        const int nrun = a.split ? 6 : 2, run = a.split ? a.dstride : a.L, nch = (run + CT_CHUNK - 1) / CT_CHUNK;
        const int rn = lane / nch, c = (lane - rn * nch) * CT_CHUNK, cg = rn & 1, dy = rn >> 1;
        const bool copies = rn < nrun;
        const uint32_t dst = ring + (uint32_t)cg * sbytes + (uint32_t)(dy * a.dstride + c) * 16u;
        const uint32_t bytes = (uint32_t)min(CT_CHUNK, run - c) * 16u;
        const bf16* src = a.in + 8 * (cg * g.vol + (long)dy * g.pitch + c);
        // a second group that does not exist: the zeros behind the tensor, at another place for every CTA
        const bf16* zeros = a.in + 8 * ((long)g.B * a.Gin * g.vol + blockIdx.x * 24 % (CELL_SLACK - CT_RUN) + c);
        for (int tile = blockIdx.x; tile < a.ntiles && ok; tile += gridDim.x) {
            const int tp = tile % a.ntp, zg = tile / a.ntp, z0 = zg % a.nzg * a.S, b = zg / a.nzg;
            const int planes = min(a.S, g.Z - z0) + 2;   // input planes
            // first staged cell of a plane: one row and one point before the tile's first point
            const long q0 = (long)tp * 128 * a.R;
            for (int kc = 0; kc < nkc && ok; ++kc) {
                const int wb = (int)(wissued & 1);
                if (wissued >= 2) ok = warp_wait(s32(&wempty[wb]), (uint32_t)((wissued / 2 - 1) & 1), CT_WAIT);
                if (!ok) break;
                if (lane == 0) bar_expect(s32(&wfull[wb]), wbytes);
                __syncwarp();
                for (uint32_t o = (uint32_t)lane * (CT_CHUNK * 16u); o < wbytes; o += 32u * CT_CHUNK * 16u)
                    bulk_g2s(base + (uint32_t)wb * wbytes + o, reinterpret_cast<const unsigned char*>(a.wt) + (size_t)kc * wbytes + o,
                             min(CT_CHUNK * 16u, wbytes - o), s32(&wfull[wb]));
                ++wissued;
                const bool none = cg && 2 * kc + 1 == a.Gin;
                const bf16* from = none ? zeros : src + 8 * (((long)b * a.Gin + 2 * kc) * g.vol + (long)z0 * g.plane + q0);
                const long step = none ? 0 : 8 * g.plane;
                for (int zp = 0; zp < planes; ++zp, ++issued) {
                    const int s = (int)(issued % a.nst);
                    if (issued >= a.nst) ok = warp_wait(s32(&empty[s]), (uint32_t)((issued / a.nst - 1) & 1), CT_WAIT);
                    if (!ok) break;
                    const uint32_t fb = s32(&full[s]);
                    if (lane == 0) bar_expect(fb, 2u * sbytes);
                    __syncwarp();
                    if (copies) bulk_g2s(dst + (uint32_t)s * (uint32_t)a.stage, from, bytes, fb);
                    from += step;
                }
            }
        }
    } else if (warp == 1 || warp >= 10) {
        const int r = warp == 1 ? 0 : warp - 9;   // this warp's 128-point block of every tile
        const uint32_t lead = elect_one();
        long it = 0, wit = 0;
        int lt = 0;
        for (int tile = blockIdx.x; tile < a.ntiles && ok; tile += gridDim.x, ++lt) {
            const int tp = tile % a.ntp, z0 = tile / a.ntp % a.nzg * a.S, buf = lt & 1;
            const int S = min(a.S, g.Z - z0);
            // (the last tile of a plane may be short)
            const bool mine = r < a.R && (tp * a.R + r) * 128 < g.span;
            if (lt >= 2) ok = warp_wait(s32(&acce[buf]), (uint32_t)(((lt >> 1) - 1) & 1), CT_WAIT);
            if (!ok) break;
            tc_after();
            const uint32_t Np = (uint32_t)a.Np, acc = tmem + (uint32_t)(buf * 256) + (uint32_t)(r * a.S) * Np;
            for (int kc = 0; kc < nkc && ok; ++kc, ++wit) {
                const int wb = (int)(wit & 1);
                ok = warp_wait(s32(&wfull[wb]), (uint32_t)((wit >> 1) & 1), CT_WAIT);
                if (!ok) break;
                // B: a view's weights [2 channel groups][dz = 2, 1, 0][Np][8]: next channel group 3 Np*16 bytes, next 8
                // rows 128
                const uint64_t bd = ndesc(base + (uint32_t)wb * wbytes, 3u * Np * 16u, 128u);
                const uint32_t bhi = (uint32_t)(bd >> 32);
                for (int zp = 0; zp < S + 2; ++zp, ++it) {
                    const int s = (int)(it % a.nst);
                    ok = warp_wait(s32(&full[s]), (uint32_t)((it / a.nst) & 1), CT_WAIT);
                    if (!ok) break;
                    tc_after();
                    // A: a tap's view of the points; next channel group sbytes, next 8 points 128
                    const uint64_t ad = ndesc(ring + (uint32_t)s * (uint32_t)a.stage + (uint32_t)r * 2048u, sbytes, 128u);
                    const uint32_t ahi = (uint32_t)(ad >> 32);
                    // input plane zp serves the output planes s0 .. s1 (dz = zp - s0 .. zp - s1)
                    const int s0 = max(0, zp - 2), s1 = min(S - 1, zp);
                    const uint32_t row0 = (uint32_t)(2 - zp + s0) * Np;
                    const uint32_t id = idesc_bf16(128, (s1 - s0 + 1) * a.Np, 0, 0);
                    uint32_t blo = (uint32_t)bd + row0;
                    const bool opens = kc == 0 && zp < S;   // plane zp's first tap: its accumulator starts here
                    const uint32_t d = acc + (uint32_t)s0 * Np;
                    if (mine) {
#pragma unroll
                        for (int t = 0; t < 9; ++t, blo += 6u * Np) {
                            const uint32_t al = (uint32_t)ad + (uint32_t)((t / 3) * a.dstride + t % 3);
                            if (t == 0 && opens) {
                                if (zp > s0) mma_bf16(lead, d, al, ahi, blo, bhi, idesc_bf16(128, (zp - s0) * a.Np, 0, 0), 1u);
                                mma_bf16(lead, acc + (uint32_t)zp * Np, al, ahi, (uint32_t)bd + 2u * Np, bhi,
                                         idesc_bf16(128, a.Np, 0, 0), 0u);
                            } else {
                                mma_bf16(lead, d, al, ahi, blo, bhi, id, 1u);
                            }
                        }
                    }
                    if (lead) mma_commit(s32(&empty[s]));
                    __syncwarp();
                }
                if (ok && lead) mma_commit(s32(&wempty[wb]));
                __syncwarp();
            }
            if (ok && lead) mma_commit(s32(&accf[buf]));
            __syncwarp();
        }
    } else {
        const int w = warp & 3, half = (warp - 2) >> 2;   // tensor-memory lanes 32 w .. 32 w + 31; every second plane
        float bsum[CT_NPMAX / 16] = {0.f, 0.f, 0.f, 0.f};
        int lt = 0;
        for (int tile = blockIdx.x; tile < a.ntiles && ok; tile += gridDim.x, ++lt) {
            const int tp = tile % a.ntp, zg = tile / a.ntp, z0 = zg % a.nzg * a.S, b = zg / a.nzg, buf = lt & 1;
            const int nr = min(a.R, (g.span - tp * 128 * a.R + 127) / 128), S = min(a.S, g.Z - z0);
            ok = warp_wait(s32(&accf[buf]), (uint32_t)((lt >> 1) & 1), CT_WAIT);
            if (!ok) break;
            tc_after();
            for (int r = 0; r < nr; ++r) {
                const int rel = (tp * a.R + r) * 128 + 32 * w + lane;   // point y pitch + x
                const int y = rel / g.pitch, x = rel - y * g.pitch;
                const bool in = y < g.Y && x < g.X;
                for (int sp = half; sp < S; sp += 2) {
                    const int z = z0 + sp;
                    const long q = (long)(z + 1) * g.plane + g.pitch + 1 + rel;   // its cell in a channel group
#pragma unroll
                    for (int cb = 0; cb < CT_NPMAX; cb += 16) {
                        if (cb >= a.Np) break;
                        float v[16];
                        tmem_ld16(tmem + ((uint32_t)(32 * w) << 16) + (uint32_t)(buf * 256 + (r * a.S + sp) * a.Np + cb), v);
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            v[j] += sbias[cb + j];
                            if (a.relu) v[j] = fmaxf(v[j], 0.f);
                        }
                        if constexpr (OUT == CONV_PLANAR) {
                            if (in)
#pragma unroll
                                for (int j = 0; j < 16; ++j)
                                    if (cb + j < a.Cout)
                                        reinterpret_cast<float*>(a.out)[(((size_t)b * a.Cout + cb + j) * g.Z + z) * g.Y * g.X +
                                                                        (size_t)y * g.X + x] = v[j];
                        } else {
                            const int c0 = a.ooff + cb;
                            if constexpr (OUT == CONV_GRAD) {
#pragma unroll
                                for (int h = 0; h < 2; ++h) {
                                    uint4 m = make_uint4(0u, 0u, 0u, 0u);
                                    if (in && cb + 8 * h < a.Cout)
                                        m = *reinterpret_cast<const uint4*>(a.mask + 8 * (((long)b * a.Gout + c0 / 8 + h) * g.vol + q));
#pragma unroll
                                    for (int j = 0; j < 8; ++j)
                                        if (!(cell_value(m, j) > 0.f)) v[8 * h + j] = 0.f;
                                }
                                bsum[cb / 16] += lane_fold16(v, lane);
                            }
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                if (!in || cb + 8 * h >= a.Cout) continue;
                                if constexpr (OUT == CONV_F32CELLS) {
                                    float4* o = reinterpret_cast<float4*>(a.out) + 2 * (((long)b * a.Gout + c0 / 8 + h) * g.vol + q);
                                    o[0] = make_float4(v[8 * h], v[8 * h + 1], v[8 * h + 2], v[8 * h + 3]);
                                    o[1] = make_float4(v[8 * h + 4], v[8 * h + 5], v[8 * h + 6], v[8 * h + 7]);
                                } else if (a.ooff % 8 == 0) {
                                    *reinterpret_cast<uint4*>(reinterpret_cast<bf16*>(a.out) +
                                                              8 * (((long)b * a.Gout + c0 / 8 + h) * g.vol + q)) = pack_cell(v + 8 * h);
                                } else {   // a channel offset inside a cell: channel by channel
#pragma unroll
                                    for (int j = 0; j < 8; ++j)
                                        if (cb + 8 * h + j < a.Cout) {
                                            const int c = c0 + 8 * h + j;
                                            reinterpret_cast<bf16*>(a.out)[8 * (((long)b * a.Gout + c / 8) * g.vol + q) + c % 8] =
                                                __float2bfloat16(v[8 * h + j]);
                                        }
                                }
                            }
                        }
                    }
                }
            }
            tc_before();
            __syncwarp();
            if (lane == 0) bar_arrive(s32(&acce[buf]));
        }
        if constexpr (OUT == CONV_GRAD) {
            const int c = lane_fold16_channel(lane);
#pragma unroll
            for (int k = 0; k < CT_NPMAX / 16; ++k)
                if (!(lane & 1) && 16 * k + c < a.Cout) atomicAdd(&a.gb[16 * k + c], bsum[k]);
        }
    }
    if (!ok) {
        atomicOr(a.status, (unsigned)HELM_DEV_WAIT);
        fail_any = 1;
    }
    __syncthreads();
    if (fail_any) {
        if (warp == 0 && lane == 0) {   // the copies of the last (at most nst, two) issued stages and chunks may still be in flight
            for (long k = issued > a.nst ? issued - a.nst : 0; k < issued; ++k)
                bar_wait(s32(&full[k % a.nst]), (uint32_t)((k / a.nst) & 1), CT_WAIT);
            for (long k = wissued > 2 ? wissued - 2 : 0; k < wissued; ++k)
                bar_wait(s32(&wfull[k & 1]), (uint32_t)((k >> 1) & 1), CT_WAIT);
        } else if ((warp == 1 || warp >= 10) && elect_one()) {   // the lane that issued (the election is deterministic)
            mma_commit(s32(&drainb));
            bar_wait(s32(&drainb), 0, CT_WAIT);
        }
    }
    tc_before();
    __syncthreads();
    if (warp == 1) tmem_free(tmem);
}

// ---- weight gradient ---------------------------------------------------------------------------------
struct WgradArgs {
    CellGrid g;
    const bf16* in;      // cells of Gin groups
    int Gin;
    const bf16* gr;      // gradient cells of Ggr groups, halo zero
    int Ggr;
    int Cin, Cout, M;    // M = 64 or 128 accumulator rows
    int Nb, nblk;        // input channels of a block (a multiple of 16), blocks
    int ndy;             // 3: a CTA holds the 9 taps of its dz; 1: the 3 taps of its (dz, dy)
    int kt, ntp, ntiles, nst, stage;   // points of a tile (a multiple of 16, at most WG_KT), ...
    float* gw;           // [Cout][Cin][27]
    unsigned* status;
};

__global__ void __launch_bounds__(CT_THREADS, 1) wgrad_cells_kernel(const __grid_constant__ WgradArgs a) {
    extern __shared__ __align__(128) unsigned char csm[];
    __shared__ __align__(8) uint64_t full[CT_NST], empty[CT_NST], accf, drainb;
    __shared__ uint32_t tslot;
    __shared__ int fail_any;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t base = (s32(csm) + 127u) & ~127u;
    const CellGrid& g = a.g;
    const int ib = blockIdx.x % a.nblk, tg = blockIdx.x / a.nblk;
    const int dz = a.ndy == 3 ? tg : tg / 3, dy0 = a.ndy == 3 ? 0 : tg % 3;
    const int ng = min(a.Nb / 8, a.Gin - ib * (a.Nb / 8));   // input groups of this block that exist
    const uint32_t abytes = (uint32_t)(a.Ggr * a.kt) * 16u, brow = (uint32_t)(a.kt + 2) * 16u;
    if (threadIdx.x == 0) {
        for (int s = 0; s < CT_NST; ++s) { bar_init(s32(&full[s]), 1); bar_init(s32(&empty[s]), 1); }
        bar_init(s32(&accf), 1);
        bar_init(s32(&drainb), 1);
        fail_any = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(&tslot);
    tc_before();
    __syncthreads();
    tc_after();
    const uint32_t tmem = tslot;
    bool ok = true;
    long issued = 0;
    if (warp == 0) {
        for (int tile = blockIdx.y; tile < a.ntiles && ok; tile += gridDim.y) {
            const int tp = tile % a.ntp, zb = tile / a.ntp, z = zb % g.Z, b = zb / g.Z;
            const int ks = min(a.kt / 16, (g.span - tp * a.kt + 15) / 16);   // K steps of 16 points
            const int s = (int)(issued % a.nst);
            if (issued >= a.nst)
                ok = warp_wait(s32(&empty[s]), (uint32_t)((issued / a.nst - 1) & 1), CT_WAIT);
            if (!ok) break;
            const uint32_t st = base + (uint32_t)s * (uint32_t)a.stage, fb = s32(&full[s]);
            const uint32_t an = (uint32_t)ks * 256u, bn = an + 32u;
            if (lane == 0) bar_expect(fb, (uint32_t)a.Ggr * an + (uint32_t)(a.ndy * ng) * bn);
            __syncwarp();
            const long q = (long)tp * a.kt;   // first point, from the plane's first
            for (int k = lane; k < a.Ggr + a.ndy * ng; k += 32) {
                if (k < a.Ggr) {
                    bulk_g2s(st + (uint32_t)k * (uint32_t)a.kt * 16u,
                             a.gr + 8 * (((long)b * a.Ggr + k) * g.vol + (long)(z + 1) * g.plane + g.pitch + 1 + q), an, fb);
                } else {
                    const int e = k - a.Ggr, dy = e / ng, cg = e % ng;
                    bulk_g2s(st + abytes + (uint32_t)(dy * (a.Nb / 8) + cg) * brow,
                             a.in + 8 * (((long)b * a.Gin + ib * (a.Nb / 8) + cg) * g.vol + (long)(z + dz) * g.plane +
                                         (long)(dy0 + dy) * g.pitch + q),
                             bn, fb);
                }
            }
            ++issued;
        }
    } else if (warp == 1) {
        {
            const uint32_t lead = elect_one();
            const uint32_t idesc = idesc_bf16(a.M, a.Nb, 1, 1);
            int n = 0;
            for (int tile = blockIdx.y; tile < a.ntiles && ok; tile += gridDim.y, ++n) {
                const int ks = min(a.kt / 16, (g.span - (tile % a.ntp) * a.kt + 15) / 16);
                const int s = n % a.nst;
                ok = warp_wait(s32(&full[s]), (uint32_t)((n / a.nst) & 1), CT_WAIT);
                if (!ok) break;
                tc_after();
                const uint32_t ga = base + (uint32_t)s * (uint32_t)a.stage, xa = ga + abytes;
                // both operands MN-major: next 8 points (K) 128 bytes, next channel group one run of cells.  Without
                // swizzling the leading-byte offset is the K stride and the stride-byte offset the M/N stride
                const uint64_t ad = ndesc(ga, 128u, (uint32_t)a.kt * 16u), bd = ndesc(xa, 128u, brow);
                const uint32_t alo = (uint32_t)ad, ahi = (uint32_t)(ad >> 32), bhi = (uint32_t)(bd >> 32);
                for (int t = 0; t < 3 * a.ndy; ++t) {
                    const uint32_t blo = (uint32_t)bd + (uint32_t)((t / 3) * (a.Nb / 8) * (a.kt + 2) + t % 3);
                    const uint32_t acc = tmem + (uint32_t)(t * a.Nb);
#pragma unroll
                    for (int kk = 0; kk < WG_KT / 16; ++kk)
                        if (kk < ks)
                            mma_bf16(lead, acc, alo + (uint32_t)(16 * kk), ahi, blo + (uint32_t)(16 * kk), bhi, idesc,
                                     (n | kk) ? 1u : 0u);
                }
                if (lead) mma_commit(s32(&empty[s]));
                    __syncwarp();
            }
            if (ok && lead) mma_commit(s32(&accf));
        }
    } else if (blockIdx.y < a.ntiles) {
        const int w = warp & 3;
        ok = warp_wait(s32(&accf), 0, CT_WAIT * 4);
        if (ok) {
            tc_after();
            // accumulator rows: 128 -> lane 32 w + l; 64 -> 16 rows in the first half of each warp's lanes
            const int o = a.M == 128 ? 32 * w + lane : 16 * w + lane;
            const bool live = (a.M == 128 || lane < 16) && o < a.Cout;
            for (int t = 0; t < 3 * a.ndy; ++t) {
                const int tap = 9 * dz + 3 * dy0 + t;
                for (int cb = 0; cb < a.Nb; cb += 16) {
                    float v[16];
                    tmem_ld16(tmem + ((uint32_t)(32 * w) << 16) + (uint32_t)(t * a.Nb + cb), v);
                    if (live)
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            const int i = ib * a.Nb + cb + j;
                            if (i < a.Cin) atomicAdd(&a.gw[((size_t)o * a.Cin + i) * 27 + tap], v[j]);
                        }
                }
            }
        }
    }
    if (!ok) {
        atomicOr(a.status, (unsigned)HELM_DEV_WAIT);
        fail_any = 1;
    }
    __syncthreads();
    if (fail_any) {
        if (warp == 0 && lane == 0) {
            for (long k = issued > a.nst ? issued - a.nst : 0; k < issued; ++k)
                bar_wait(s32(&full[k % a.nst]), (uint32_t)((k / a.nst) & 1), CT_WAIT);
        } else if (warp == 1 && elect_one()) {
            mma_commit(s32(&drainb));
            bar_wait(s32(&drainb), 0, CT_WAIT);
        }
    }
    tc_before();
    __syncthreads();
    if (warp == 1) tmem_free(tmem);
}

// arranged[kc][3 dy + dx][cg][2 - dz][o][j] = W(o0 + o, 16 kc + 8 cg + j, t), t = 9 dz + 3 dy + dx, for the output slice
// o0 .. o0 + Np - 1, zero beyond Cout / Cin; W(o, i, t) = w[(o Cin + i) 27 + t] (wmode 0) or
// w[(i Cout + o) 27 + 26 - t] (wmode 1: the data gradient's flipped, transposed weights)
__global__ void arrange_w_kernel(const bf16* __restrict__ w, int Cin, int Cout, int o0, int wmode, int Np, int nkc,
                                 bf16* __restrict__ dst) {
    const size_t n = (size_t)nkc * 27 * 2 * Np * 8;
    for (size_t id = blockIdx.x * (size_t)blockDim.x + threadIdx.x; id < n; id += (size_t)gridDim.x * blockDim.x) {
        size_t r = id;
        const int j = (int)(r % 8);
        r /= 8;
        const int o = (int)(r % Np);
        r /= Np;
        const int dz = 2 - (int)(r % 3);
        r /= 3;
        const int cg = (int)(r % 2);
        r /= 2;
        const int t = 9 * dz + (int)(r % 9);
        const int kc = (int)(r / 9);
        const int i = 16 * kc + 8 * cg + j, oo = o0 + o;
        bf16 v = __float2bfloat16(0.f);
        if (oo < Cout && i < Cin)
            v = wmode ? w[((size_t)i * Cout + oo) * 27 + 26 - t] : w[((size_t)oo * Cin + i) * 27 + t];
        dst[id] = v;
    }
}

int sm_count() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        cudaGetLastError();
    return sms > 0 ? sms : 152;
}

}  // namespace

size_t conv_scratch_bytes(int Cin, int Cout) {
    const int Np = std::min((Cout + 15) / 16 * 16, CT_NPMAX), nkc = (Cin + 15) / 16;
    return (size_t)nkc * 27 * 2 * Np * 8 * sizeof(bf16);
}

helm_status conv_prepare() {
    HELM_CUDA_TRY(cudaFuncSetAttribute(conv_cells_kernel<CONV_CELLS>, cudaFuncAttributeMaxDynamicSharedMemorySize, CT_SMEM));
    HELM_CUDA_TRY(cudaFuncSetAttribute(conv_cells_kernel<CONV_PLANAR>, cudaFuncAttributeMaxDynamicSharedMemorySize, CT_SMEM));
    HELM_CUDA_TRY(cudaFuncSetAttribute(conv_cells_kernel<CONV_F32CELLS>, cudaFuncAttributeMaxDynamicSharedMemorySize, CT_SMEM));
    HELM_CUDA_TRY(cudaFuncSetAttribute(conv_cells_kernel<CONV_GRAD>, cudaFuncAttributeMaxDynamicSharedMemorySize, CT_SMEM));
    HELM_CUDA_TRY(cudaFuncSetAttribute(wgrad_cells_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, CT_SMEM));
    return HELM_OK;
}

// One convolution; mode: CONV_CELLS ....  wscr holds conv_scratch_bytes(Cin, Cout).
helm_status conv_cells(const CellGrid& g, int mode, const bf16* in, int Cin, const bf16* w, int wmode, const float* bias,
                       void* out, int Cout, int Cout_total, int ooff, int relu, const bf16* mask, float* gb, bf16* wscr,
                       unsigned* status, cudaStream_t s) {
    const int Gin = cell_groups(Cin), nkc = (Gin + 1) / 2;
    const int sms = sm_count();
    // output slices of at most 64 channels (one accumulator width each); the launches follow one another on s
    for (int o0 = 0; o0 < Cout; o0 += CT_NPMAX) {
        ConvArgs a;
        a.g = g;
        a.in = in; a.Gin = Gin;
        a.Cout = std::min(Cout - o0, CT_NPMAX);
        a.Np = (a.Cout + 15) / 16 * 16;
        a.wt = wscr;
        a.bias = bias ? bias + o0 : nullptr;
        a.out = mode == CONV_PLANAR ? (void*)((float*)out + (size_t)o0 * g.Z * g.Y * g.X) : out;
        a.Gout = cell_groups(Cout_total);
        a.ooff = ooff + o0;
        a.relu = relu;
        a.mask = mask;
        a.gb = gb ? gb + o0 : nullptr;
        a.status = status;
        // the largest tile whose count still gives every SM two (small grids: shorter runs, then fewer planes), within
        // 256 accumulator columns: more planes save MMAs, longer runs share their halo rows
        int R = CT_RMAX, S = std::max(1, CT_PLANES / a.Np);
        auto tiles = [&](int r, int sp) { return (long)g.B * ((g.Z + sp - 1) / sp) * ((g.span + 128 * r - 1) / (128 * r)); };
        while (R > 1 && tiles(R, S) < 2L * sms) R /= 2;
        while (S > 1 && tiles(R, S) < 2L * sms) S = (S + 1) / 2;
        a.R = R;
        a.S = S;
        a.ntp = (g.span + 128 * R - 1) / (128 * R);
        a.nzg = (g.Z + S - 1) / S;
        a.ntiles = (int)tiles(R, S);
        // one run with the rows between the three dy views, or three runs where that is shorter (long rows)
        a.split = g.pitch > 128 * R + 2;
        a.dstride = a.split ? 128 * R + 2 : g.pitch;
        a.L = a.split ? 3 * a.dstride : 128 * R + 2 + 2 * g.pitch;
        a.stage = (2 * a.L * 16 + 127) / 128 * 128;
        const int wbytes = 27 * 2 * a.Np * 16;
        a.nst = std::min(CT_NST, (CT_SMEM - 128 - 2 * wbytes) / a.stage);
        const size_t na = (size_t)nkc * 27 * 2 * a.Np * 8;
        arrange_w_kernel<<<(unsigned)((na + 255) / 256), 256, 0, s>>>(w, Cin, Cout, o0, wmode, a.Np, nkc, wscr);
        const size_t smem = (size_t)a.nst * a.stage + 2 * wbytes + 128;
        const unsigned grid = (unsigned)std::min((long)a.ntiles, (long)sms);
        if (mode == CONV_CELLS) conv_cells_kernel<CONV_CELLS><<<grid, CV_THREADS, smem, s>>>(a);
        else if (mode == CONV_PLANAR) conv_cells_kernel<CONV_PLANAR><<<grid, CV_THREADS, smem, s>>>(a);
        else if (mode == CONV_F32CELLS) conv_cells_kernel<CONV_F32CELLS><<<grid, CV_THREADS, smem, s>>>(a);
        else conv_cells_kernel<CONV_GRAD><<<grid, CV_THREADS, smem, s>>>(a);
        HELM_CUDA_TRY(cudaGetLastError());
    }
    return HELM_OK;
}

// gw += d loss/d W for the gradient cells gr of the layer output (Cout <= 128)
helm_status wgrad_cells(const CellGrid& g, const bf16* in, int Cin, const bf16* gr, int Cout, float* gw, unsigned* status,
                        cudaStream_t s) {
    WgradArgs a;
    a.g = g;
    a.in = in; a.Gin = cell_groups(Cin);
    a.gr = gr; a.Ggr = cell_groups(Cout);
    a.Cin = Cin; a.Cout = Cout;
    a.M = Cout <= 64 ? 64 : 128;
    a.gw = gw;
    a.status = status;
    // accumulators in tensor memory (512 columns): the 9 taps of a dz up to 48 inputs, else 3 taps of up to 160
    const int Nin = 8 * a.Gin;
    a.ndy = Nin <= 48 ? 3 : 1;
    a.nblk = (Nin + 159) / 160;
    a.Nb = ((Nin + 15) / 16 + a.nblk - 1) / a.nblk * 16;
    // the MMAs read M / 8 groups of gradient rows; those beyond Ggr fall into the staged inputs (their accumulator
    // rows are not used), so a stage is at least as long as all of them
    auto stage = [&](int kt) {
        return (std::max(a.M / 8 * kt * 16, a.Ggr * kt * 16 + a.ndy * (a.Nb / 8) * (kt + 2) * 16) + 127) / 128 * 128;
    };
    a.kt = 3 * stage(WG_KT) + 128 <= CT_SMEM ? WG_KT : WG_KT / 2;   // at least three stages
    a.stage = stage(a.kt);
    a.nst = std::min(CT_NST, (CT_SMEM - 128) / a.stage);
    a.ntp = (g.span + a.kt - 1) / a.kt;
    a.ntiles = (int)((long)g.B * g.Z * a.ntp);
    // whole waves of CTAs (one per SM), each with at most WG_POINTS points
    const int groups = (a.ndy == 3 ? 3 : 9) * a.nblk, sms = sm_count();
    const int one = std::max(1, sms / groups), per = WG_POINTS / a.kt;
    const int waves = (a.ntiles + per * one - 1) / (per * one);
    const int split = std::min(a.ntiles, std::max(1, waves * sms / groups));
    wgrad_cells_kernel<<<dim3((unsigned)groups, (unsigned)split), CT_THREADS, (size_t)a.nst * a.stage + 128, s>>>(a);
    HELM_CUDA_TRY(cudaGetLastError());
    return HELM_OK;
}
