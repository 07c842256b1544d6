// EigT step 3 (Sec. 4.1): the N_x N_y independent complex tridiagonal systems of
// Eq. Indep_precond_system along z,
//   (gamma_z + b_1) u_1 + zeta_z u_2 = y_1
//   u_{l-1} + b_l u_l + u_{l+1} = y_l
//   zeta_z u_{N-1} + (gamma_z + b_N) u_N = y_N,
//   b_l = alpha_x d_{x,i} + alpha_y d_{y,j} + h_z^2 k0^2(z_l) - 2(alpha_x + alpha_y + 1).
//
// Every context with a preconditioner factorises its systems at set-up; the solves below run over the stored factors or
// recompute them, with the same operations and the same bits.
#include "common.cuh"
#include <cuda_bf16.h>
#include <cuda_fp16.h>

namespace {

struct ZParams {
    int nx, ny, nz;
    const float2* dxs;   // alpha_x d_{x,i}
    const float2* dys;   // alpha_y d_{y,j}
    const float2* cz;    // h_z^2 k0^2(z_l) - 2(alpha_x + alpha_y + 1)
    float2 gz;           // gamma_z
    float zz;            // zeta_z
};

__device__ inline float2 f2(float a, float b) { return make_float2(a, b); }

// The steps of the factorised solve, every operation rounded as written (explicit fma/mul/add, so that no
// kernel contracts differently): the set-up factors, the forward and backward sweeps over stored factors
// and the sweeps that recompute the factors all produce the same bits.
// pivot step: m_l = 1 / (b_l - a_l c'_{l-1}) with b_l = s + cz_l (+ gamma_z at the ends), then c'_l = sup_l m_l
// (*dmag, when given: |Re| + |Im| of the pivot, for the tiny-pivot check of the set-up)
__device__ __forceinline__ float2 zpivot(float2 s, float2 czl, bool end, float2 gz, float a, float sup, float2& c,
                                         float* dmag = nullptr) {
    float bx = __fadd_rn(s.x, czl.x), by = __fadd_rn(s.y, czl.y);
    if (end) { bx = __fadd_rn(bx, gz.x); by = __fadd_rn(by, gz.y); }
    const float dx = __fmaf_rn(-c.x, a, bx), dy = __fmaf_rn(-c.y, a, by);
    if (dmag) *dmag = fabsf(dx) + fabsf(dy);
    // 1/|pivot|^2 by the hardware reciprocal (at most one ulp off, one instruction: the recurrence is the
    // critical path of every line), then m = conj(pivot) / |pivot|^2
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__fmaf_rn(dx, dx, __fmul_rn(dy, dy))));
    const float2 m = make_float2(__fmul_rn(dx, r), __fmul_rn(-dy, r));
    c = make_float2(__fmul_rn(m.x, sup), __fmul_rn(m.y, sup));
    return m;
}
// forward: d_l = (y_l - a_l d_{l-1}) m_l
__device__ __forceinline__ float2 zfwd(float2 y, float2 d, float a, float2 m) {
    const float tx = __fmaf_rn(-d.x, a, y.x), ty = __fmaf_rn(-d.y, a, y.y);
    return make_float2(__fmaf_rn(tx, m.x, __fmul_rn(-ty, m.y)), __fmaf_rn(tx, m.y, __fmul_rn(ty, m.x)));
}
// backward: x_l = d_l - sup_l (m_l x_{l+1})
__device__ __forceinline__ float2 zbwd(float2 d, float2 m, float2 x, float sup) {
    const float px = __fmaf_rn(m.x, x.x, __fmul_rn(-m.y, x.y)), py = __fmaf_rn(m.x, x.y, __fmul_rn(m.y, x.x));
    return make_float2(__fmaf_rn(-px, sup, d.x), __fmaf_rn(-py, sup, d.y));
}

// y + a b with the product rounded as written (so that every kernel that forms a generated right-hand side
// gives the same bits)
__device__ __forceinline__ float2 zaddmul(float2 y, float2 a, float2 b) {
    return make_float2(__fadd_rn(y.x, __fmaf_rn(a.x, b.x, -__fmul_rn(a.y, b.y))),
                       __fadd_rn(y.y, __fmaf_rn(a.y, b.x, __fmul_rn(a.x, b.y))));
}

// ---- factorised z-solve (EigT) -------------------------------------------------------------------
// The systems of a context never change, so their Thomas factorisation is computed once at set-up:
//   m_l = 1 / (b_l - a_l c'_{l-1}),   c'_l = sup_l m_l,   (a_l, sup_l the sub- and super-diagonal)
// and stored per point (complex64).  An application is then one thread per line: forward
// d_l = (y_l - a_l d_{l-1}) m_l written over the output, backward x_l = d_l - sup_l m_l x_{l+1}, i.e.
// one complex product per step and sweep, no divisions, no interface system.  The backward sweep
// re-reads d and m soon after the forward sweep wrote/read them, mostly from L2.  Lines of consecutive
// x are consecutive threads, so every step is a contiguous row access.
constexpr int ZU = 8;   // steps whose loads are issued together

__global__ void __launch_bounds__(128) zfactor_kernel(ZParams p, float2* __restrict__ m, unsigned* status) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
    if (i >= p.nx) return;
    const size_t plane = (size_t)p.nx * p.ny, base = (size_t)j * p.nx + i;
    const float2 dxy = make_float2(__fadd_rn(p.dxs[i].x, p.dys[j].x), __fadd_rn(p.dxs[i].y, p.dys[j].y));
    float2 cprev = f2(0.f, 0.f);
    float minpiv = 1e30f;
    for (int l = 0; l < p.nz; ++l) {
        const float a = l == 0 ? 0.f : (l == p.nz - 1 ? p.zz : 1.f);
        const float sup = l == p.nz - 1 ? 0.f : (l == 0 ? p.zz : 1.f);
        float dm;
        const float2 mi = zpivot(dxy, p.cz[l], l == 0 || l == p.nz - 1, p.gz, a, sup, cprev, &dm);
        minpiv = fminf(minpiv, dm);
        m[base + (size_t)l * plane] = mi;
    }
    if (!(minpiv > 1e-30f)) atomicOr(status, (unsigned)HELM_DEV_PIVOT);
}

__global__ void __launch_bounds__(128) zsolve_fact_kernel(int nx, int ny, int nz, float zz, const float2* __restrict__ m,
                                                         const float2* in, float2* out) {
    // blockIdx.y = (right-hand side of a batch group) * ny + j; the factors m are shared
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y % ny, vb = blockIdx.y / ny;
    if (i >= nx) return;
    const size_t plane = (size_t)nx * ny, base = (size_t)j * nx + i, voff = (size_t)vb * plane * nz;
    if (vb) {
        in += voff;
        out += voff;
    }
    float2 d = f2(0.f, 0.f);
    for (int l0 = 0; l0 < nz; l0 += ZU) {
        float2 yv[ZU], mv[ZU];
#pragma unroll
        for (int u = 0; u < ZU; ++u)
            if (l0 + u < nz) {
                yv[u] = in[base + (size_t)(l0 + u) * plane];
                mv[u] = m[base + (size_t)(l0 + u) * plane];
            }
#pragma unroll
        for (int u = 0; u < ZU; ++u) {
            const int l = l0 + u;
            if (l < nz) {
                const float a = l == 0 ? 0.f : (l == nz - 1 ? zz : 1.f);
                d = zfwd(yv[u], d, a, mv[u]);
                out[base + (size_t)l * plane] = d;
            }
        }
    }
    float2 x = f2(0.f, 0.f);
    for (int l1 = nz; l1 > 0; l1 -= ZU) {
        float2 dv[ZU], mv[ZU];
#pragma unroll
        for (int u = 0; u < ZU; ++u) {
            const int l = l1 - 1 - u;
            if (l >= 0) {
                dv[u] = out[base + (size_t)l * plane];
                mv[u] = m[base + (size_t)l * plane];
            }
        }
#pragma unroll
        for (int u = 0; u < ZU; ++u) {
            const int l = l1 - 1 - u;
            if (l >= 0) {
                const float sup = l == nz - 1 ? 0.f : (l == 0 ? zz : 1.f);
                x = zbwd(dv[u], mv[u], x, sup);
                out[base + (size_t)l * plane] = x;
            }
        }
    }
}

// Factorised solve, L2-resident form (even N_x).  The backward sweep reads
// d and m again; when every line runs at once those re-reads (16 B/pt) miss the L2, so here a persistent
// grid of a few 64-thread CTAs per SM keeps about 20k-40k lines in flight (their d and m stay in L2) and
// walks the rest in turn.  Each thread takes two adjacent lines (16-byte accesses) and streams its inputs
// through a private ring of ZB blocks of ZU steps in shared memory by cp.async (one group per block, no
// block barrier); a landed block is read into registers at once and its ZU dependent steps then run back
// to back, so the shared-memory latency is paid once per block rather than once per step.
// GEN = 1, 2 (PFFT's boundary correction; 2: no input grid): the right-hand side of ZGen is formed as the forward
// sweep consumes a block.  Its two factors that vary with the slice and x ride in the ring beside y and m; those
// that vary with the slice and y are read one block ahead into registers (they are contiguous in the slice
// index), the rest are constant along a line.  One thread per line without a ring, re-reading all eight
// factors at every step, took 235 us at 256^3; this takes 119 us (GEN = 1) and 107 us (GEN = 2).
constexpr int ZRT = 64, ZU2 = 8;
__host__ __device__ constexpr int zring_arrays(int gen) { return gen == 0 ? 2 : (gen == 1 ? 4 : 3); }
__host__ __device__ constexpr int zring_depth(int gen) { return gen == 1 ? 3 : 4; }   // blocks in the ring
__host__ __device__ constexpr size_t zring_bytes(int gen) {   // 64 KiB, 96 KiB, 96 KiB
    return (size_t)zring_depth(gen) * ZU2 * zring_arrays(gen) * ZRT * sizeof(float4);
}

__device__ __forceinline__ void zcp16(void* smem, const void* gmem) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(a), "l"(gmem) : "memory");
}
__device__ __forceinline__ void zcommit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void zwait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }
__device__ __forceinline__ void zwait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// nb > 1: nb right-hand side grids back to back (a batch group), sharing the factors m
template <int GEN>
__global__ void __launch_bounds__(ZRT) zsolve_ring_kernel(int nx, int ny, int nz, float zz,
                                                         const float4* __restrict__ m, const float4* in, float4* out,
                                                         int nb, const __grid_constant__ ZGen g) {
    constexpr int ZB = zring_depth(GEN), NA = zring_arrays(GEN);
    constexpr int AQ = GEN == 1 ? 2 : 1;   // first of the two Q arrays in a slot (y: 0, m: the last without GEN)
    constexpr int AM = GEN == 2 ? 0 : 1;
    extern __shared__ float4 zring[];   // [ZB * ZU2][NA][ZRT]
    const int tid = threadIdx.x;
    const int hx = nx / 2, npairs = hx * ny;
    const int nblk = (nz + ZU2 - 1) / ZU2;
    const size_t plane = (size_t)hx * ny;   // in float4 (two lines) units
    auto slot = [&](int st, int a) -> float4* { return &zring[((size_t)st * NA + a) * ZRT + tid]; };
    for (int prb = blockIdx.x * ZRT + tid; prb < npairs * nb; prb += gridDim.x * ZRT) {
        const int pr = prb % npairs, vb = prb / npairs;
        const size_t off = (size_t)pr;   // pair pr = (j, i/2) is float4 pr of every plane
        const size_t voff = (size_t)vb * plane * nz;   // this right-hand side's grid (the factors are shared)
        const int j = pr / hx;
        const float4* q0 = GEN ? reinterpret_cast<const float4*>(g.q0) + (pr - j * hx) : nullptr;
        const float4* q1 = GEN ? reinterpret_cast<const float4*>(g.q1) + (pr - j * hx) : nullptr;
        // ---- forward: d_l = (y_l - a_l d_{l-1}) m_l, steps in increasing l
        auto fetch_f = [&](int b) {
            if (b < nblk) {
#pragma unroll
                for (int u = 0; u < ZU2; ++u) {
                    const int l = b * ZU2 + u;
                    if (l < nz) {
                        if (GEN != 2) zcp16(slot((b % ZB) * ZU2 + u, 0), in + voff + off + (size_t)l * plane);
                        zcp16(slot((b % ZB) * ZU2 + u, AM), m + off + (size_t)l * plane);
                        if (GEN) {
                            zcp16(slot((b % ZB) * ZU2 + u, AQ), q0 + (size_t)l * hx);
                            zcp16(slot((b % ZB) * ZU2 + u, AQ + 1), q1 + (size_t)l * hx);
                        }
                    }
                }
            }
            zcommit();
        };
        for (int b = 0; b < ZB - 1; ++b) fetch_f(b);
        float2 d0 = f2(0.f, 0.f), d1 = d0;
        float2 p0 = d0, p1 = d0;                         // GEN: the factors constant along the line pair
        float4 c2 = make_float4(0.f, 0.f, 0.f, 0.f), c3 = c2;
        float4 n2[ZU2 / 2], n3[ZU2 / 2];                 // p2, p3 of the next block, two steps per float4
        const float4* p2 = nullptr;
        const float4* p3 = nullptr;
        if (GEN) {
            p0 = g.p0[j];
            p1 = g.p1[j];
            c2 = reinterpret_cast<const float4*>(g.q2)[pr - j * hx];
            c3 = reinterpret_cast<const float4*>(g.q3)[pr - j * hx];
            p2 = reinterpret_cast<const float4*>(g.p2 + (size_t)j * g.nzp);
            p3 = reinterpret_cast<const float4*>(g.p3 + (size_t)j * g.nzp);
#pragma unroll
            for (int u = 0; u < ZU2 / 2; ++u) { n2[u] = p2[u]; n3[u] = p3[u]; }
        }
        for (int b = 0; b < nblk; ++b) {
            fetch_f(b + ZB - 1);
            zwait<ZB - 1>();   // block b has landed
            float4 y[ZU2], mm[ZU2];
#pragma unroll
            for (int u = 0; u < ZU2; ++u) {
                y[u] = GEN == 2 ? make_float4(0.f, 0.f, 0.f, 0.f) : *slot((b % ZB) * ZU2 + u, 0);
                mm[u] = *slot((b % ZB) * ZU2 + u, AM);
                if (GEN) {
                    const float4 a = *slot((b % ZB) * ZU2 + u, AQ), e = *slot((b % ZB) * ZU2 + u, AQ + 1);
                    const float2 r2 = u & 1 ? f2(n2[u / 2].z, n2[u / 2].w) : f2(n2[u / 2].x, n2[u / 2].y);
                    const float2 r3 = u & 1 ? f2(n3[u / 2].z, n3[u / 2].w) : f2(n3[u / 2].x, n3[u / 2].y);
                    float2 v0 = f2(y[u].x, y[u].y), v1 = f2(y[u].z, y[u].w);
                    v0 = zaddmul(v0, p0, f2(a.x, a.y));
                    v0 = zaddmul(v0, p1, f2(e.x, e.y));
                    v0 = zaddmul(v0, r2, f2(c2.x, c2.y));
                    v0 = zaddmul(v0, r3, f2(c3.x, c3.y));
                    v1 = zaddmul(v1, p0, f2(a.z, a.w));
                    v1 = zaddmul(v1, p1, f2(e.z, e.w));
                    v1 = zaddmul(v1, r2, f2(c2.z, c2.w));
                    v1 = zaddmul(v1, r3, f2(c3.z, c3.w));
                    y[u] = make_float4(v0.x, v0.y, v1.x, v1.y);
                }
            }
            if (GEN && b + 1 < nblk)
#pragma unroll
                for (int u = 0; u < ZU2 / 2; ++u) {
                    n2[u] = p2[(b + 1) * (ZU2 / 2) + u];
                    n3[u] = p3[(b + 1) * (ZU2 / 2) + u];
                }
#pragma unroll
            for (int u = 0; u < ZU2; ++u) {
                const int l = b * ZU2 + u;
                if (l < nz) {
                    const float a = l == 0 ? 0.f : (l == nz - 1 ? zz : 1.f);
                    d0 = zfwd(f2(y[u].x, y[u].y), d0, a, f2(mm[u].x, mm[u].y));
                    d1 = zfwd(f2(y[u].z, y[u].w), d1, a, f2(mm[u].z, mm[u].w));
                    out[voff + off + (size_t)l * plane] = make_float4(d0.x, d0.y, d1.x, d1.y);
                }
            }
        }
        zwait_all();
        __threadfence_block();
        // ---- backward: x_l = d_l - s_l m_l x_{l+1}, steps in decreasing l (block b holds l = nz-1-(b ZU2 + u))
        auto fetch_b = [&](int b) {
            if (b < nblk) {
#pragma unroll
                for (int u = 0; u < ZU2; ++u) {
                    const int l = nz - 1 - (b * ZU2 + u);
                    if (l >= 0) {
                        zcp16(slot((b % ZB) * ZU2 + u, 0), out + voff + off + (size_t)l * plane);
                        zcp16(slot((b % ZB) * ZU2 + u, 1), m + off + (size_t)l * plane);
                    }
                }
            }
            zcommit();
        };
        for (int b = 0; b < ZB - 1; ++b) fetch_b(b);
        float2 x0 = f2(0.f, 0.f), x1 = x0;
        for (int b = 0; b < nblk; ++b) {
            fetch_b(b + ZB - 1);
            zwait<ZB - 1>();
            float4 dv[ZU2], mm[ZU2];
#pragma unroll
            for (int u = 0; u < ZU2; ++u) {
                dv[u] = *slot((b % ZB) * ZU2 + u, 0);
                mm[u] = *slot((b % ZB) * ZU2 + u, 1);
            }
#pragma unroll
            for (int u = 0; u < ZU2; ++u) {
                const int l = nz - 1 - (b * ZU2 + u);
                if (l >= 0) {
                    const float sup = l == nz - 1 ? 0.f : (l == 0 ? zz : 1.f);
                    x0 = zbwd(f2(dv[u].x, dv[u].y), f2(mm[u].x, mm[u].y), x0, sup);
                    x1 = zbwd(f2(dv[u].z, dv[u].w), f2(mm[u].z, mm[u].w), x1, sup);
                    out[voff + off + (size_t)l * plane] = make_float4(x0.x, x0.y, x1.x, x1.y);
                }
            }
        }
        zwait_all();
    }
}

// EigT form without the factor stream: the pivots depend only on the line's lateral shift
// s_ij = alpha_x d_{x,i} + alpha_y d_{y,j} and the plane, so the sweeps recompute them step by step (the same
// operations as zfactor_kernel, one reciprocal per step).  The forward sweep writes no forward values either: it only
// saves the recurrences' state (c'_{l-1}, d_{l-1}) at the start of every block of ZU2 steps to a small scratch (2
// bytes per point, [block][pair] so that a warp's saves are contiguous rows), and the backward sweep recomputes a
// block's factors and forward values from its checkpoint and from y, read a second time.  HBM and L2 see y read twice
// and x written: for 16-bit grids 12 bytes a point where forward values in FP32 took 28.
// A grid is one thread per pair of lines (32k threads at 256^3, three to four 64-thread CTAs per SM), so latency is
// hidden by prefetch depth: a six-block ring per thread (48 steps ahead).  Block b lives in slot b mod 6 in both
// sweeps, so the last six blocks need no second read.  ALL: grids of few CTAs hold every block of their lines
// (and the checkpoints) in shared memory: one read, all loads in flight at once.
// The recurrence is the bound where the grid is small (one reciprocal and six dependent operations a step), and
// everything else is kept off it: cz comes from shared memory, and the blocks without an end row run without
// per-step conditions, behind which each step's loads used to wait.
// CTAs of 32 threads, for a fuller last wave, gain nothing.
// Measured (with per-step conditions; without; without forward values): 256^3, FP16 chain 105, 74, 59 us; 200^3 FP32
// 63, 41, 40; 150 x 100 x 75 25, 15, 13; 32^3 10.6, 8.9, 7.5.
constexpr int ZPB = 6;   // ring depth (blocks) of the pivot-recomputing kernel
// a step of a line pair: FP32 16 bytes, 16-bit 8; then cz, and for ALL the checkpoints
constexpr size_t zpiv_smem(int nz, bool h16, bool all) {
    return (size_t)(all ? (nz + ZU2 - 1) / ZU2 : ZPB) * ZU2 * ZRT * (h16 ? 8 : 16) + (size_t)(nz + 1) / 2 * sizeof(float4) +
           (all ? (size_t)((nz + ZU2 - 1) / ZU2) * 2 * ZRT * sizeof(float4) : 0);
}
constexpr size_t ZPIV_ALL_MAX = 112 * 1024;   // two CTAs per SM
template <bool B>
struct BoolC {
    constexpr operator bool() const { return B; }
};
__device__ __forceinline__ void zwait_piv() { asm volatile("cp.async.wait_group %0;\n" ::"n"(ZPB - 1) : "memory"); }

__device__ __forceinline__ void zcp8(void* smem, const void* gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(gmem) : "memory");
}
// a pair of lines' complex values from / to four 16-bit values (memory order re0, im0, re1, im1), H = 1 BF16,
// 2 FP16 (clamped to the finite range); widening is exact
template <int H>
__device__ __forceinline__ float4 h4_to_f4(uint2 w) {
    if (H == 2) {
        const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&w.x));
        const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&w.y));
        return make_float4(a.x, a.y, b.x, b.y);
    }
    return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xFFFF0000u), __uint_as_float(w.y << 16),
                       __uint_as_float(w.y & 0xFFFF0000u));
}
// a step's input values of a line pair as stored, and widened
template <bool BF> struct ZPairOf { typedef float4 T; };
template <> struct ZPairOf<true> { typedef uint2 T; };
template <int H>
__device__ __forceinline__ float4 zwiden(float4 v) { return v; }
template <int H>
__device__ __forceinline__ float4 zwiden(uint2 v) { return h4_to_f4<H>(v); }
template <int H>
__device__ __forceinline__ uint32_t zpack16(float lo, float hi) {
    if (H == 2) {
        const __half2 v = __floats2half2_rn(fminf(fmaxf(lo, -65504.f), 65504.f), fminf(fmaxf(hi, -65504.f), 65504.f));
        return *reinterpret_cast<const uint32_t*>(&v);
    }
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}

// H (1 BF16, 2 FP16): y read and x written (times oscale) in 16 bits (uint2 per line pair); H = 0: float4.  in may
// equal out.
template <int H, bool ALL>
__global__ void __launch_bounds__(ZRT, ALL ? 2 : 4) zsolve_piv_kernel(int nx, int ny, int nz, float zz, float2 gz,
                                                                      const float2* __restrict__ dxs,
                                                                      const float2* __restrict__ dys,
                                                                      const float2* __restrict__ cz, const void* inv,
                                                                      void* outv, float4* __restrict__ ck, int nb,
                                                                      float oscale = 1.f, double* h16d = nullptr,
                                                                      float gain = 1.f) {
    constexpr bool BF = H != 0;
    typedef typename ZPairOf<BF>::T Y;   // a step's input values of a line pair
    extern __shared__ float4 zsm[];      // ring [depth * ZU2][ZRT], cz [nz], ALL: checkpoints [block][2][ZRT]
    const Y* in = reinterpret_cast<const Y*>(inv);
    Y* out = reinterpret_cast<Y*>(outv);
    const int tid = threadIdx.x;
    const int hx = nx / 2, npairs = hx * ny, nall = npairs * nb;
    const int nblk = (nz + ZU2 - 1) / ZU2, depth = ALL ? nblk : ZPB;
    const size_t plane = (size_t)hx * ny;   // in line pairs
    Y* ring = reinterpret_cast<Y*>(zsm);
    float4* after = zsm + (size_t)depth * ZU2 * ZRT * sizeof(Y) / sizeof(float4);
    float2* scz = reinterpret_cast<float2*>(after);
    float4* sck = after + (nz + 1) / 2;
    for (int l = tid; l < nz; l += ZRT) scz[l] = cz[l];
    __syncthreads();
    grid_wait();
    grid_trigger();
    // FP16 chain with dynamic stage scales (h16d): the output scale from the bound of ||T2|| (h16d[1]),
    // recorded in h16d[5]; the squared norm of what is stored accumulates into h16d[2]
    float nacc = 0.f;
    if (BF && h16d) {
        const double n2 = chain_value(h16d + 1);
        float sc = 1.f;
        if (n2 > 0.0) {
            int e = 15 - (int)ceil(log2((double)gain * sqrt(n2)));
            e = e < -100 ? -100 : (e > 100 ? 100 : e);
            sc = ldexpf(1.f, e);
        }
        oscale *= sc;
        if (blockIdx.x == 0 && threadIdx.x == 0) h16d[5] = sc;
    }
    auto slot = [&](int blk, int u) -> Y* { return ring + (size_t)((ALL ? blk : blk % ZPB) * ZU2 + u) * ZRT + tid; };
    for (int prb = blockIdx.x * ZRT + tid; prb < nall; prb += gridDim.x * ZRT) {
        const int pr = prb % npairs, vb = prb / npairs;
        const int j = pr / hx, i0 = 2 * (pr - j * hx);
        const size_t base = (size_t)vb * plane * nz + (size_t)pr;
        // the input of block blk (steps l = blk ZU2 + u) into its slot; one group per call, empty ones included
        auto fetch = [&](int blk) {
            if (blk >= 0 && blk < nblk) {
                const Y* src = in + base + (size_t)(blk * ZU2) * plane;
                const int n = min(ZU2, nz - blk * ZU2);
#pragma unroll
                for (int u = 0; u < ZU2; ++u)
                    if (u < n) {
                        if (BF) zcp8(slot(blk, u), src + (size_t)u * plane);
                        else zcp16(slot(blk, u), src + (size_t)u * plane);
                    }
            }
            zcommit();
        };
        for (int b = 0; b < depth - (ALL ? 0 : 1); ++b) fetch(b);
        const float2 s0 = make_float2(__fadd_rn(dxs[i0].x, dys[j].x), __fadd_rn(dxs[i0].y, dys[j].y));
        const float2 s1 = make_float2(__fadd_rn(dxs[i0 + 1].x, dys[j].x), __fadd_rn(dxs[i0 + 1].y, dys[j].y));
        // blocks whose steps are all interior (off-diagonals 1, no corner) run without per-step conditions: with
        // them, every step's loads waited inside the recurrence
        auto interior = [&](int blk) { return blk > 0 && blk * ZU2 + ZU2 < nz; };
        // block blk forward from the state c0, c1 (c'_{l-1}) and d0, d1 (d_{l-1}): its factors m and values
        // d_l = (y_l - a_l d_{l-1}) m_l go to keep(u, m0, m1, d0, d1)
        auto forward = [&](auto edge, int blk, float2& c0, float2& c1, float2& d0, float2& d1, auto keep) {
            float4 y[ZU2];
#pragma unroll
            for (int u = 0; u < ZU2; ++u) y[u] = zwiden<H>(*slot(blk, u));
#pragma unroll
            for (int u = 0; u < ZU2; ++u) {
                const int l = blk * ZU2 + u;
                if (!edge || l < nz) {
                    const bool end = edge && (l == 0 || l == nz - 1);
                    const float a = !edge ? 1.f : (l == 0 ? 0.f : (l == nz - 1 ? zz : 1.f));
                    const float sup = !edge ? 1.f : (l == nz - 1 ? 0.f : (l == 0 ? zz : 1.f));
                    const float2 czl = scz[l];
                    const float2 m0 = zpivot(s0, czl, end, gz, a, sup, c0), m1 = zpivot(s1, czl, end, gz, a, sup, c1);
                    d0 = zfwd(f2(y[u].x, y[u].y), d0, a, m0);
                    d1 = zfwd(f2(y[u].z, y[u].w), d1, a, m1);
                    keep(u, m0, m1, d0, d1);
                }
            }
        };
        auto save = [&](int b, const float4& c, const float4& d) {
            float4* o = ALL ? sck + (size_t)(2 * b) * ZRT + tid : ck + (size_t)(2 * b) * nall + prb;
            o[0] = c;
            o[ALL ? ZRT : nall] = d;
        };
        auto state = [&](int b, float4& c, float4& d) {
            const float4* o = ALL ? sck + (size_t)(2 * b) * ZRT + tid : ck + (size_t)(2 * b) * nall + prb;
            c = o[0];
            d = o[ALL ? ZRT : nall];
        };
        // ---- forward: the checkpoints (the last block's values are formed by the backward sweep alone)
        float2 d0 = f2(0.f, 0.f), d1 = d0, c0 = d0, c1 = d0;
        if (ALL) zwait_all();
        for (int b = 0; b < nblk; ++b) {
            if (!ALL) {
                fetch(b + ZPB - 1);
                zwait_piv();   // block b has landed
            }
            save(b, make_float4(c0.x, c0.y, c1.x, c1.y), make_float4(d0.x, d0.y, d1.x, d1.y));
            if (b == nblk - 1) break;
            auto none = [](int, float2, float2, float2, float2) {};
            if (interior(b)) forward(BoolC<false>(), b, c0, c1, d0, d1, none);
            else forward(BoolC<true>(), b, c0, c1, d0, d1, none);
        }
        // ---- backward: x_l = d_l - sup_l m_l x_{l+1}, blocks in decreasing order
        float2 x0 = f2(0.f, 0.f), x1 = x0;
        float4 cn, dn;
        state(nblk - 1, cn, dn);
        auto bwd = [&](auto edge, int blk, const float4& cv, const float4& dv) {
            float2 e0 = f2(cv.x, cv.y), e1 = f2(cv.z, cv.w), g0 = f2(dv.x, dv.y), g1 = f2(dv.z, dv.w);
            float2 m0[ZU2], m1[ZU2], v0[ZU2], v1[ZU2];
            forward(edge, blk, e0, e1, g0, g1, [&](int u, float2 a, float2 b, float2 p, float2 q) {
                m0[u] = a;
                m1[u] = b;
                v0[u] = p;
                v1[u] = q;
            });
            Y* o = out + base + (size_t)(blk * ZU2) * plane;
#pragma unroll
            for (int uu = 0; uu < ZU2; ++uu) {
                const int u = ZU2 - 1 - uu, l = blk * ZU2 + u;
                if (!edge || l < nz) {
                    const float sup = !edge ? 1.f : (l == nz - 1 ? 0.f : (l == 0 ? zz : 1.f));
                    x0 = zbwd(v0[u], m0[u], x0, sup);
                    x1 = zbwd(v1[u], m1[u], x1, sup);
                    if constexpr (BF) {
                        const float a = oscale * x0.x, b2 = oscale * x0.y, c2 = oscale * x1.x, d2 = oscale * x1.y;
                        o[(size_t)u * plane] = make_uint2(zpack16<H>(a, b2), zpack16<H>(c2, d2));
                        nacc = fmaf(a, a, fmaf(b2, b2, fmaf(c2, c2, fmaf(d2, d2, nacc))));
                    } else {
                        o[(size_t)u * plane] = make_float4(x0.x, x0.y, x1.x, x1.y);
                    }
                }
            }
        };
        for (int b = 0; b < nblk; ++b) {
            const int blk = nblk - 1 - b;
            if (!ALL) {
                // the last ZPB blocks are still in their slots; slot of block blk + 1 is free for blk - (ZPB - 1)
                if (b > 0) fetch(blk - (ZPB - 1));
                else zcommit();
                zwait_piv();   // block blk has landed
            }
            const float4 cv = cn, dv = dn;
            if (blk > 0) state(blk - 1, cn, dn);   // the next block's checkpoint, early
            if (interior(blk)) bwd(BoolC<false>(), blk, cv, dv);
            else bwd(BoolC<true>(), blk, cv, dv);
        }
        zwait_all();
    }
    if (BF && h16d) {
        double d = (double)nacc;
        for (int o = 16; o > 0; o >>= 1) d += __shfl_down_sync(0xffffffffu, d, o);
        if ((threadIdx.x & 31) == 0) atomicAdd(h16d + 2, d);
    }
}

}  // namespace

// Set-up: the Thomas factors of the z-systems with lateral eigenvalue shifts dxs_i + dys_j (one complex64
// per point) into *m (allocated here if NULL).
helm_status zsolve_factor_with(helm_ctx* c, const float2* dxs, const float2* dys, float2** m, cudaStream_t s) {
    if (!*m) {
        if (cudaMalloc(m, c->npts * sizeof(float2)) != cudaSuccess) { cudaGetLastError(); return HELM_ERR_NOMEM; }
    }
    if (!c->zring_sms) {   // the ring kernel of the factorised solve: shared memory and grid size
        HELM_CUDA_TRY(cudaFuncSetAttribute(zsolve_ring_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)zring_bytes(0)));
        HELM_CUDA_TRY(cudaFuncSetAttribute(zsolve_ring_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)zring_bytes(1)));
        HELM_CUDA_TRY(cudaFuncSetAttribute(zsolve_ring_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)zring_bytes(2)));
        HELM_CUDA_TRY(cudaDeviceGetAttribute(&c->zring_sms, cudaDevAttrMultiProcessorCount, c->device));
    }
    ZParams p;
    p.nx = c->nx; p.ny = c->ny; p.nz = c->nz;
    p.dxs = dxs; p.dys = dys; p.cz = c->cz;
    p.gz = make_float2((float)c->gam[2].x, (float)c->gam[2].y);
    p.zz = (float)c->zeta[2];
    dim3 grid((c->nx + 127) / 128, c->ny);
    zfactor_kernel<<<grid, 128, 0, s>>>(p, *m, c->status_d);
    HELM_CUDA_TRY(cudaGetLastError());
    return HELM_OK;
}

helm_status zsolve_factor(helm_ctx* c, cudaStream_t s) { return zsolve_factor_with(c, c->dxs, c->dys, &c->zfac, s); }

// factorised solve with factors m
helm_status launch_zsolve_fact(helm_ctx* c, const float2* m, const float2* in, float2* out, cudaStream_t s, int nb) {
    prof_begin(c, s, PROF_ZSOLVE);
    if (c->nx % 2 == 0 && c->tune_zring && c->zring_sms > 0) {
        const int sms = c->zring_sms;
        const int npairs = c->nx / 2 * c->ny * nb;
        const int need = (npairs + ZRT - 1) / ZRT;
        const int grid = need < sms * c->tune_zring ? need : sms * c->tune_zring;
        zsolve_ring_kernel<0><<<grid, ZRT, zring_bytes(0), s>>>(c->nx, c->ny, c->nz, (float)c->zeta[2],
                                                                reinterpret_cast<const float4*>(m),
                                                                reinterpret_cast<const float4*>(in),
                                                                reinterpret_cast<float4*>(out), nb, ZGen());
        prof_end(c, s);
        HELM_CUDA_TRY(cudaGetLastError());
        return HELM_OK;
    }
    dim3 grid((c->nx + 127) / 128, c->ny * nb);
    zsolve_fact_kernel<<<grid, 128, 0, s>>>(c->nx, c->ny, c->nz, (float)c->zeta[2], m, in, out);
    prof_end(c, s);
    HELM_CUDA_TRY(cudaGetLastError());
    return HELM_OK;
}

helm_status launch_zsolve_gen(helm_ctx* c, const float2* m, const float2* in, float2* out, const ZGen& g, cudaStream_t s) {
    if (c->nx % 2 != 0 || c->zring_sms <= 0) return HELM_ERR_UNSUPPORTED;
    const int need = (c->nx / 2 * c->ny + ZRT - 1) / ZRT, cap = 2 * c->zring_sms;   // two CTAs per SM (shared memory)
    const int grid = need < cap ? need : cap;
    prof_begin(c, s, PROF_ZSOLVE);
    if (in)
        zsolve_ring_kernel<1><<<grid, ZRT, zring_bytes(1), s>>>(c->nx, c->ny, c->nz, (float)c->zeta[2],
                                                                reinterpret_cast<const float4*>(m),
                                                                reinterpret_cast<const float4*>(in),
                                                                reinterpret_cast<float4*>(out), 1, g);
    else
        zsolve_ring_kernel<2><<<grid, ZRT, zring_bytes(2), s>>>(c->nx, c->ny, c->nz, (float)c->zeta[2],
                                                                reinterpret_cast<const float4*>(m), nullptr,
                                                                reinterpret_cast<float4*>(out), 1, g);
    prof_end(c, s);
    HELM_CUDA_TRY(cudaGetLastError());
    return HELM_OK;
}

size_t zsolve_ck_bytes(const helm_ctx* c, int nb) {
    return (size_t)((c->nz + ZU2 - 1) / ZU2) * 2 * (size_t)(c->nx / 2) * c->ny * nb * sizeof(float4);
}

// The context's own pivot checkpoints, for nb right-hand sides per z-solve launch.  Growing frees the old block, so
// launches that are captured to run again later must not hold it: a batch plan brings its own (c->zck swapped while it
// captures).
helm_status zsolve_reserve(helm_ctx* c, int nb) {
    const size_t bytes = zsolve_ck_bytes(c, nb);
    if (bytes <= c->zck_bytes) return HELM_OK;
    cudaFree(c->zck);
    c->zck = nullptr;
    c->zck_bytes = 0;
    if (cudaMalloc(&c->zck, bytes) != cudaSuccess) { cudaGetLastError(); return HELM_ERR_NOMEM; }
    c->zck_bytes = bytes;
    return HELM_OK;
}

// the pivot-recomputing kernel on the checkpoints c->zck
template <int H>
static helm_status run_zpiv(helm_ctx* c, const void* in, void* out, int nb, float oscale, double* h16d, float gain,
                            cudaStream_t s) {
    const int need = (c->nx / 2 * c->ny * nb + ZRT - 1) / ZRT;
    const int cap = c->zring_sms * 2 * (c->tune_zring > 0 ? c->tune_zring : 1);   // tune_zring 1..3: 2, 4 or 6 CTAs per SM
    // lines held whole where all CTAs fit the SMs that way, two on each
    const size_t all = zpiv_smem(c->nz, H != 0, true), ring = zpiv_smem(c->nz, H != 0, false);
    const bool whole = all <= ZPIV_ALL_MAX && need <= 2 * c->zring_sms;
    float4* ck = reinterpret_cast<float4*>(c->zck);
    const float2 gz = make_float2((float)c->gam[2].x, (float)c->gam[2].y);
    if (!(c->zpiv_ready & (1 << H))) {
        HELM_CUDA_TRY(cudaFuncSetAttribute(zsolve_piv_kernel<H, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)zpiv_smem(512, H != 0, false)));
        HELM_CUDA_TRY(cudaFuncSetAttribute(zsolve_piv_kernel<H, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)ZPIV_ALL_MAX));
        c->zpiv_ready |= 1 << H;
    }
    if (whole)
        launch_after(c->follows, zsolve_piv_kernel<H, true>, need, ZRT, all, s, c->nx, c->ny, c->nz, (float)c->zeta[2], gz, c->dxs,
                     c->dys, c->cz, in, out, ck, nb, oscale, h16d, gain);
    else
        launch_after(c->follows, zsolve_piv_kernel<H, false>, need < cap ? need : cap, ZRT, ring, s, c->nx, c->ny, c->nz,
                     (float)c->zeta[2], gz, c->dxs, c->dys, c->cz, in, out, ck, nb, oscale, h16d, gain);
    HELM_CUDA_TRY(cudaGetLastError());
    return HELM_OK;
}

helm_status launch_zsolve(helm_ctx* c, const float2* in, float2* out, cudaStream_t s, int nb) {
    if (!c->zfac) return HELM_ERR_UNSUPPORTED;   // a context without a preconditioner
    if (in && c->nx % 2 == 0 && c->tune_zring && c->zring_sms > 0 && !c->zpiv_off) {
        // EigT: pivots recomputed from the shifts (the set-up factors' operations), checkpoints in a scratch
        // of the context (grown here outside stream capture; a capturing caller provides it beforehand)
        if (zsolve_ck_bytes(c, nb) > c->zck_bytes) {
            cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
            HELM_CUDA_TRY(cudaStreamIsCapturing(s, &cap));
            if (cap != cudaStreamCaptureStatusNone) return launch_zsolve_fact(c, c->zfac, in, out, s, nb);
            helm_status st;
            if ((st = zsolve_reserve(c, nb)) != HELM_OK) return st;
        }
        prof_begin(c, s, PROF_ZSOLVE);
        const helm_status st = run_zpiv<0>(c, in, out, nb, 1.f, nullptr, 1.f, s);
        prof_end(c, s);
        return st;
    }
    return launch_zsolve_fact(c, c->zfac, in, out, s, nb);
}

// The z-solves of the 16-bit transform chain (HELM_PREC_BF16, HELM_PREC_FP16): the pivot-recomputing kernel
// with 16-bit y and x (in may equal out; x scaled by oscale).  No fallback: a launch under stream capture without
// reserved checkpoints returns HELM_ERR_UNSUPPORTED.
helm_status launch_zsolve_h16(helm_ctx* c, const void* in, void* out, float oscale, cudaStream_t s, int nb,
                              double* h16d, float gain) {
    const int H = c->opt.precision == HELM_PREC_FP16 ? 2 : 1;
    if (c->nx % 2 != 0 || c->zring_sms <= 0) return HELM_ERR_UNSUPPORTED;
    if (zsolve_ck_bytes(c, nb) > c->zck_bytes) {
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        HELM_CUDA_TRY(cudaStreamIsCapturing(s, &cap));
        if (cap != cudaStreamCaptureStatusNone) return HELM_ERR_UNSUPPORTED;
        helm_status st;
        if ((st = zsolve_reserve(c, nb)) != HELM_OK) return st;
    }
    prof_begin(c, s, PROF_ZSOLVE);
    const helm_status st = H == 2 ? run_zpiv<2>(c, in, out, nb, oscale, h16d, gain, s)
                                  : run_zpiv<1>(c, in, out, nb, oscale, nullptr, 1.f, s);
    prof_end(c, s);
    return st;
}
