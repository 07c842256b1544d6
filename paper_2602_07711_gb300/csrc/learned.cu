// Learned correction (an extension of the method, not in the paper): a small 3D U-Net N applied after
// the EigT preconditioner inside flexible GMRES,
//     c = s * N( v/RMS(v), M^-1 v/s, Re(k^2/k0^2) - 1 ),    s = RMS(M^-1 v),
//     z = M^-1 v + alpha c,   alpha = <A c, v - A M^-1 v> / <A c, A c>  (complex, minimises |v - A z|_2),
// trained on (residual, error) pairs of the solver's own solves.  The minimal-residual step makes plain
// EigT the fallback: |v - A z| <= |v - A M^-1 v| for any network output, alpha -> 0 for a useless one,
// and the correction is dropped (z = M^-1 v) when A c vanishes or any of the sums is not finite.
//
// Network (width c):  a1 = relu(conv(x, 5->c)), a2 = relu(conv(a1, c->c)), p = avgpool2(a2),
// b1 = relu(conv(p, c->2c)), b2 = relu(conv(b1, 2c->2c)), u = [upsample2(b2), a2],
// d1 = relu(conv(u, 3c->c)), y = conv(d1, c->2).  3x3x3 convolutions, zero padding, stride 1.
// Activations and weights are stored in BF16, every product is accumulated in FP32; training keeps FP32
// master weights and Adam moments.  The caller's tensors are channel-first [B][C][Z][Y][X]; inside, activations
// are cells of 8 channels on halo grids (cells.cuh).  The gradient of a layer's output is an MMA operand twice
// (data and weight gradient), which rounds it to BF16, so it is stored that way; whatever is summed from it in
// FP32 (the bias gradient) is summed before the rounding, by the kernel that produces it, and the gradients that
// are summed further (those of u and p) stay FP32.
//
// Kernels: the 3x3x3 convolutions run on the tcgen05 tensor cores as implicit GEMMs (conv_tc.cu: forward
// and data gradient through flipped/transposed weights with the ReLU mask fused, weight gradient with the
// taps' accumulators in tensor memory).  Here: packing of the caller's tensors into cells, pooling/upsampling
// and their adjoints, MSE, Adam, feature assembly and the correction step.
#include "cells.cuh"
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

namespace {
// a device buffer that grows on demand
struct Buf {
    void* p = nullptr;
    size_t cap = 0;
};
}  // namespace

struct helm_net {
    int c = 0;
    size_t nparam = 0;
    float *W = nullptr, *G = nullptr, *Mom = nullptr, *Vel = nullptr;   // fp32 master weights, grads, Adam
    bf16* Wb = nullptr;                                                 // bf16 copy
    size_t woff[6], boff[6];
    int co[6], ci[6];
    // workspace of the last forward's shape (full-resolution and half-resolution grids); grown on demand, never
    // shrunk.  `fresh`: the cells that no kernel writes have to be zeroed before use (new shape or new memory).
    // `recorded`: a call was recorded into a CUDA graph, whose replays may use the memory in another shape unseen
    int B = 0, Z = 0, Y = 0, X = 0;
    CellGrid gf, gh;
    bool fresh = false, gfresh = false, recorded = false;
    int gB_ = 0, gZ_ = 0, gY_ = 0, gX_ = 0;                 // shape of the gradient workspace
    Buf xp, y;                                              // channel-first features (BF16) and output (FP32)
    Buf x, a1, u, d1, p, b1, b2;                            // BF16 cells; u holds [up(b2), a2]; p, b1, b2 half resolution
    Buf gy, gC, gD, gH1, gH2;                                   // gradients, BF16 cells (gH1, gH2 half resolution)
    Buf gU, gP;                                             // gradients of u and p, FP32 cells
    // statistics and reduction scratch (16 doubles): 0 sum|v|^2, 1 sum|M^-1 v|^2, 2 |alpha| of the last
    // correction, 3 corrections dropped, 4 corrections applied, 5 sum over applied corrections of
    // |v - A z|^2/|v - A M^-1 v|^2, 6-7 <Ac, rho>, 8 |Ac|^2, 9 |rho|^2, 15 scratch of helm_net_target
    double* stats = nullptr;
    // solver-side fields (complex64, one grid): v = sigma r, c, A M^-1 v, A c
    float2 *vbuf = nullptr, *cbuf = nullptr, *az0 = nullptr, *ac = nullptr;
    size_t fcap = 0;
    bf16* wscr = nullptr;          // weights arranged for the tensor-core convolutions (one layer at a time)
    unsigned* status = nullptr;    // device status word of the network's own calls (bounded waits)
};

namespace {

bf16* cells(const Buf& b) { return reinterpret_cast<bf16*>(b.p); }
float* floats(const Buf& b) { return reinterpret_cast<float*>(b.p); }

// ---- element kernels on cells: one thread per point (of the coarse grid where there are two) and group of 8
// channels, 16-byte cells; blockIdx.y = batch * groups + group.  The channels of a2 start at channel 2c of u: where
// that is inside a cell (width not a multiple of 4), cells are assembled channel by channel. ----
struct Pt { int z, y, x; };
__device__ __forceinline__ Pt point_of(long id, const CellGrid& g) {
    const int x = (int)(id % g.X);
    const long r = id / g.X;
    return {(int)(r / g.Y), (int)(r % g.Y), x};
}
__device__ __forceinline__ long cell_of(const CellGrid& g, int z, int y, int x) {
    return (long)(z + 1) * g.plane + (long)(y + 1) * g.pitch + x + 1;
}
// channels c0 .. c0 + 7 (below C) of a BF16 tensor of G groups at cell q
__device__ __forceinline__ uint4 read_cell(const bf16* t, int G, int b, long vol, long q, int c0, int C) {
    if (c0 % 8 == 0) return *reinterpret_cast<const uint4*>(t + 8 * (((long)b * G + c0 / 8) * vol + q));
    float v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j)
        v[j] = c0 + j < C ? __bfloat162float(t[8 * (((long)b * G + (c0 + j) / 8) * vol + q) + (c0 + j) % 8]) : 0.f;
    return pack_cell(v);
}
__device__ __forceinline__ void read_cell_f32(const float* t, int G, int b, long vol, long q, int c0, int C, float* v) {
    if (c0 % 8 == 0) {
        const float4* p = reinterpret_cast<const float4*>(t) + 2 * (((long)b * G + c0 / 8) * vol + q);
        const float4 lo = p[0], hi = p[1];
        v[0] = lo.x; v[1] = lo.y; v[2] = lo.z; v[3] = lo.w;
        v[4] = hi.x; v[5] = hi.y; v[6] = hi.z; v[7] = hi.w;
        return;
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = c0 + j < C ? t[8 * (((long)b * G + (c0 + j) / 8) * vol + q) + (c0 + j) % 8] : 0.f;
}
// gb[c0 + k] += the block's sums of s[k] (channels below C)
__device__ __forceinline__ void add_channel_sums(const float* s, float* gb, int c0, int C) {
    __shared__ float red[8];
    const int lane = threadIdx.x & 31;
    if (threadIdx.x < 8) red[threadIdx.x] = 0.f;
    __syncthreads();
    const float f = lane_fold8(s, lane);
    if (!(lane & 3)) atomicAdd(&red[lane_fold8_channel(lane)], f);
    __syncthreads();
    if (threadIdx.x < 8 && c0 + threadIdx.x < C) atomicAdd(&gb[c0 + threadIdx.x], red[threadIdx.x]);
}

// The cells of up to seven tensors that the kernels read but never write are zeroed: the halos, the slack behind each
// tensor and the groups from Gw on, whose last channels nobody writes.  One warp per row of a padded plane.  Bound by its
// short scattered writes: 160^3, width 28, 145 us (of a forward pass of 2.1 ms) where a fill of the whole workspace took 480;
// 96^3 33 us, 16^3 12 us, where the fill took what the largest shape's takes.
struct Rest {
    bf16* t;
    int half, G, Gw;   // a half-resolution tensor; its groups; those that are written whole
};
struct Rests { Rest r[7]; };
__global__ void __launch_bounds__(256) zero_rest_kernel(CellGrid gf, CellGrid gh, const __grid_constant__ Rests rests) {
    const Rest R = rests.r[blockIdx.y];
    const CellGrid& g = R.half ? gh : gf;
    uint4* t = reinterpret_cast<uint4*>(R.t);
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // the rows of every channel group in `parts` shares of a CTA
    const int rows = (g.Z + 2) * (g.Y + 2), groups = g.B * R.G, parts = max(1, (int)gridDim.x / groups);
    for (int c = blockIdx.x; c < groups * parts; c += gridDim.x) {
        const int group = c / parts;
        const bool written = group % R.G < R.Gw;
        for (int q = (c % parts) * 8 + warp; q < rows; q += parts * 8) {
            const int z = q / (g.Y + 2), y = q - z * (g.Y + 2);
            uint4* row = t + ((long)group * rows + q) * g.pitch;
            if (written && z >= 1 && z <= g.Z && y >= 1 && y <= g.Y) {
                for (int x = lane ? g.X + lane : 0; x < g.pitch; x += 32) row[x] = zero;
            } else {
                for (int x = lane; x < g.pitch; x += 32) row[x] = zero;
            }
        }
    }
    const long end = (long)groups * g.vol;
    for (long x = blockIdx.x * 256L + threadIdx.x; x < CELL_SLACK; x += gridDim.x * 256L) t[end + x] = zero;
}

// channel-first features (5 channels) -> cells of group 0 (channels 5-7 zero)
__global__ void pack_x_kernel(CellGrid g, const bf16* __restrict__ in, int G, bf16* __restrict__ out) {
    const long n = (long)g.Z * g.Y * g.X;
    const int b = blockIdx.y;
    const uint16_t* s = reinterpret_cast<const uint16_t*>(in) + (size_t)b * 5 * n;
    for (long id = blockIdx.x * (long)blockDim.x + threadIdx.x; id < n; id += (long)gridDim.x * blockDim.x) {
        const Pt p = point_of(id, g);
        const uint32_t c0 = s[id], c1 = s[id + n], c2 = s[id + 2 * n], c3 = s[id + 3 * n], c4 = s[id + 4 * n];
        *reinterpret_cast<uint4*>(out + 8 * ((long)b * G * g.vol + cell_of(g, p.z, p.y, p.x))) =
            make_uint4(c0 | c1 << 16, c2 | c3 << 16, c4, 0u);
    }
}

// channel-first gradient of the output (2 channels, FP32) -> cells of group 0; gb += its sums
__global__ void __launch_bounds__(256) pack_gy_kernel(CellGrid g, const float* __restrict__ in, int G, bf16* __restrict__ out,
                                                      float* __restrict__ gb) {
    const long n = (long)g.Z * g.Y * g.X;
    const int b = blockIdx.y;
    const float* s = in + (size_t)b * 2 * n;
    float sum[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (long id = blockIdx.x * (long)blockDim.x + threadIdx.x; id < n; id += (long)gridDim.x * blockDim.x) {
        const Pt p = point_of(id, g);
        const float c0 = s[id], c1 = s[id + n];
        sum[0] += c0;
        sum[1] += c1;
        *reinterpret_cast<uint4*>(out + 8 * ((long)b * G * g.vol + cell_of(g, p.z, p.y, p.x))) =
            make_uint4(pack2(c0, c1), 0u, 0u, 0u);
    }
    add_channel_sums(sum, gb, 0, 2);
}

// out (coarse, C channels) = mean of the 8 children of a2 (channels ca .. ca + C - 1 of u)
__global__ void avgpool2_kernel(CellGrid gf, CellGrid gh, const bf16* __restrict__ u, int Gu, int ca, int C,
                                bf16* __restrict__ out, int G) {
    const long n = (long)gh.Z * gh.Y * gh.X;
    const int ng = (C + 7) / 8, b = blockIdx.y / ng, cg = blockIdx.y % ng;
    for (long id = blockIdx.x * (long)blockDim.x + threadIdx.x; id < n; id += (long)gridDim.x * blockDim.x) {
        const Pt p = point_of(id, gh);
        float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint4 v = read_cell(u, Gu, b, gf.vol, cell_of(gf, 2 * p.z + (k >> 2), 2 * p.y + ((k >> 1) & 1), 2 * p.x + (k & 1)),
                                      ca + 8 * cg, ca + C);
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[j] += cell_value(v, j);
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[j] *= 0.125f;
        *reinterpret_cast<uint4*>(out + 8 * (((long)b * G + cg) * gh.vol + cell_of(gh, p.z, p.y, p.x))) = pack_cell(acc);
    }
}

// channels 0 .. C - 1 of u (fine) = upsample2(in) (coarse): a thread writes the 8 children of a cell
__global__ void upsample2_kernel(CellGrid gf, CellGrid gh, const bf16* __restrict__ in, int G, int C, bf16* __restrict__ u,
                                 int Gu) {
    const long n = (long)gh.Z * gh.Y * gh.X;
    const int ng = (C + 7) / 8, b = blockIdx.y / ng, cg = blockIdx.y % ng;
    const bool whole = 8 * cg + 8 <= C;   // else a2's channels follow in the same cell
    for (long id = blockIdx.x * (long)blockDim.x + threadIdx.x; id < n; id += (long)gridDim.x * blockDim.x) {
        const Pt p = point_of(id, gh);
        const uint4 v = *reinterpret_cast<const uint4*>(in + 8 * (((long)b * G + cg) * gh.vol + cell_of(gh, p.z, p.y, p.x)));
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            bf16* o = u + 8 * (((long)b * Gu + cg) * gf.vol +
                               cell_of(gf, 2 * p.z + (k >> 2), 2 * p.y + ((k >> 1) & 1), 2 * p.x + (k & 1)));
            if (whole) *reinterpret_cast<uint4*>(o) = v;
            else
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (8 * cg + j < C) o[j] = __float2bfloat16(cell_value(v, j));
        }
    }
}

// gh (coarse cells, C channels) = mask(b2 > 0) * sum of the 8 children of gu (adjoint of upsample2); gb += its sums
__global__ void __launch_bounds__(256) upsample2_adj_kernel(CellGrid gf, CellGrid gh, const float* __restrict__ gu, int Gu,
                                                            const bf16* __restrict__ mask, bf16* __restrict__ out, int G, int C,
                                                            float* __restrict__ gb) {
    const long n = (long)gh.Z * gh.Y * gh.X;
    const int ng = (C + 7) / 8, b = blockIdx.y / ng, cg = blockIdx.y % ng;
    float sum[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (long id = blockIdx.x * (long)blockDim.x + threadIdx.x; id < n; id += (long)gridDim.x * blockDim.x) {
        const Pt p = point_of(id, gh);
        float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            float v[8];
            read_cell_f32(gu, Gu, b, gf.vol, cell_of(gf, 2 * p.z + (k >> 2), 2 * p.y + ((k >> 1) & 1), 2 * p.x + (k & 1)), 8 * cg,
                          C, v);
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[j] += v[j];
        }
        const long q = ((long)b * G + cg) * gh.vol + cell_of(gh, p.z, p.y, p.x);
        const uint4 m = *reinterpret_cast<const uint4*>(mask + 8 * q);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            if (!(cell_value(m, j) > 0.f)) acc[j] = 0.f;
            sum[j] += acc[j];
        }
        *reinterpret_cast<uint4*>(out + 8 * q) = pack_cell(acc);
    }
    add_channel_sums(sum, gb, 8 * cg, C);
}

// ga2 (cells, C channels) = mask(a2 > 0) * (gu_a2 + upsample2(gp)/8) (adjoint of avgpool2 added to the skip
// gradient; a2 and its gradient are channels ca .. ca + C - 1 of u and gu); gb += its sums
__global__ void __launch_bounds__(256) skip_grad_kernel(CellGrid gf, CellGrid gh, const float* __restrict__ gu,
                                                        const float* __restrict__ gp, int Gp, const bf16* __restrict__ u, int Gu,
                                                        int ca, int C, bf16* __restrict__ out, int G, float* __restrict__ gb) {
    const long n = (long)gf.Z * gf.Y * gf.X;
    const int ng = (C + 7) / 8, b = blockIdx.y / ng, cg = blockIdx.y % ng;
    float sum[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (long id = blockIdx.x * (long)blockDim.x + threadIdx.x; id < n; id += (long)gridDim.x * blockDim.x) {
        const Pt p = point_of(id, gf);
        const long q = cell_of(gf, p.z, p.y, p.x);
        float v[8], c[8];
        read_cell_f32(gu, Gu, b, gf.vol, q, ca + 8 * cg, ca + C, v);
        read_cell_f32(gp, Gp, b, gh.vol, cell_of(gh, p.z / 2, p.y / 2, p.x / 2), 8 * cg, C, c);
        const uint4 m = read_cell(u, Gu, b, gf.vol, q, ca + 8 * cg, ca + C);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            v[j] += 0.125f * c[j];
            if (8 * cg + j >= C || !(cell_value(m, j) > 0.f)) v[j] = 0.f;
            sum[j] += v[j];
        }
        *reinterpret_cast<uint4*>(out + 8 * (((long)b * G + cg) * gf.vol + q)) = pack_cell(v);
    }
    add_channel_sums(sum, gb, 8 * cg, C);
}

__global__ void mse_kernel(const float* __restrict__ y, const float* __restrict__ t, float* __restrict__ g, size_t n,
                           double* __restrict__ loss) {
    __shared__ double red[8];
    double s = 0;
    const float inv = 1.f / (float)n;
    for (size_t id = blockIdx.x * (size_t)blockDim.x + threadIdx.x; id < n; id += (size_t)gridDim.x * blockDim.x) {
        const float d = y[id] - t[id];
        g[id] = d * inv;
        s += (double)d * d;
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += red[w];
        atomicAdd(loss, 0.5 * tot / (double)n);
    }
}

__global__ void adam_kernel(float* W, const float* G, float* M, float* V, bf16* Wb, size_t n, float lr, float b1,
                            float b2, float eps, float c1, float c2) {
    const size_t id = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (id >= n) return;
    const float g = G[id];
    const float m = b1 * M[id] + (1.f - b1) * g;
    const float v = b2 * V[id] + (1.f - b2) * g * g;
    M[id] = m;
    V[id] = v;
    const float w = W[id] - lr * (m / c1) / (sqrtf(v / c2) + eps);
    W[id] = w;
    Wb[id] = __float2bfloat16(w);
}

__global__ void to_bf16_kernel(const float* a, bf16* b, size_t n) {
    const size_t id = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (id < n) b[id] = __float2bfloat16(a[id]);
}

// acc[slot] += sum |v|^2 (FP64 partials)
__global__ void sumsq_kernel(const float2* __restrict__ v, size_t n, double* acc) {
    __shared__ double r[8];
    double s = 0;
    for (size_t id = blockIdx.x * (size_t)blockDim.x + threadIdx.x; id < n; id += (size_t)gridDim.x * blockDim.x) {
        const float2 a = v[id];
        s += (double)a.x * a.x + (double)a.y * a.y;
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) r[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += r[w];
        atomicAdd(acc, t);
    }
}

// x[c0] = Re(v)/rms(v), x[c0+1] = Im(v)/rms(v)  (rms from the sum of squares in *acc); bf16 planes of n
__global__ void feat_pair_kernel(const float2* __restrict__ v, const double* __restrict__ acc, size_t n,
                                 bf16* __restrict__ x0, bf16* __restrict__ x1) {
    const float iv = acc[0] > 0 ? (float)(1.0 / sqrt(acc[0] / (double)n)) : 0.f;
    for (size_t id = blockIdx.x * (size_t)blockDim.x + threadIdx.x; id < n; id += (size_t)gridDim.x * blockDim.x) {
        const float2 a = v[id];
        x0[id] = __float2bfloat16(a.x * iv);
        x1[id] = __float2bfloat16(a.y * iv);
    }
}

// x = Re(k^2)/k0^2 - 1
__global__ void feat_contrast_kernel(const float2* __restrict__ k2, float ik02, size_t n, bf16* __restrict__ x) {
    for (size_t id = blockIdx.x * (size_t)blockDim.x + threadIdx.x; id < n; id += (size_t)gridDim.x * blockDim.x)
        x[id] = __float2bfloat16(k2[id].x * ik02 - 1.f);
}

// x0 = Re(r)/rms(r), x1 = Im(r)/rms(r) (bf16) and v = sigma[sidx] r (the vector M^-1 is applied to)
__global__ void feat_v_kernel(const float2* __restrict__ r, const double* __restrict__ acc, size_t n,
                              bf16* __restrict__ x0, bf16* __restrict__ x1, const double* __restrict__ sigma, int sidx,
                              float2* __restrict__ v) {
    const float iv = acc[0] > 0 ? (float)(1.0 / sqrt(acc[0] / (double)n)) : 0.f;
    const float sg = sigma ? (float)sigma[sidx] : 1.f;
    for (size_t id = blockIdx.x * (size_t)blockDim.x + threadIdx.x; id < n; id += (size_t)gridDim.x * blockDim.x) {
        const float2 a = r[id];
        x0[id] = __float2bfloat16(a.x * iv);
        x1[id] = __float2bfloat16(a.y * iv);
        v[id] = make_float2(a.x * sg, a.y * sg);
    }
}

// c = s (y_re + i y_im), s = sqrt(acc[1]/n) = RMS(M^-1 v)
__global__ void make_c_kernel(const float* __restrict__ y, const double* __restrict__ acc, size_t n,
                              float2* __restrict__ c) {
    const float s = (float)sqrt(acc[1] / (double)n);
    for (size_t id = blockIdx.x * (size_t)blockDim.x + threadIdx.x; id < n; id += (size_t)gridDim.x * blockDim.x)
        c[id] = make_float2(s * y[id], s * y[n + id]);
}

// rho = v - A z0:  acc[6..7] += <Ac, rho> = sum conj(Ac) rho,  acc[8] += |Ac|^2,  acc[9] += |rho|^2
__global__ void mr_dots_kernel(const float2* __restrict__ v, const float2* __restrict__ az0,
                               const float2* __restrict__ ac, size_t n, double* __restrict__ acc) {
    __shared__ double red[4][8];
    double pr = 0, pi = 0, q = 0, rr = 0;
    for (size_t id = blockIdx.x * (size_t)blockDim.x + threadIdx.x; id < n; id += (size_t)gridDim.x * blockDim.x) {
        const float2 a = ac[id], b = v[id], z = az0[id];
        const double rx = (double)b.x - z.x, ry = (double)b.y - z.y;
        pr += (double)a.x * rx + (double)a.y * ry;
        pi += (double)a.x * ry - (double)a.y * rx;
        q += (double)a.x * a.x + (double)a.y * a.y;
        rr += rx * rx + ry * ry;
    }
    for (int o = 16; o > 0; o >>= 1) {
        pr += __shfl_down_sync(0xffffffffu, pr, o);
        pi += __shfl_down_sync(0xffffffffu, pi, o);
        q += __shfl_down_sync(0xffffffffu, q, o);
        rr += __shfl_down_sync(0xffffffffu, rr, o);
    }
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) { red[0][w] = pr; red[1][w] = pi; red[2][w] = q; red[3][w] = rr; }
    __syncthreads();
    if (threadIdx.x < 4) {
        double t = 0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += red[threadIdx.x][k];
        atomicAdd(&acc[6 + threadIdx.x], t);
    }
}

// z += alpha c with alpha = acc[6..7]/acc[8]; dropped when |Ac| = 0 or a sum is not finite
__global__ void mr_apply_kernel(const float2* __restrict__ c, double* __restrict__ acc, size_t n,
                                float2* __restrict__ z) {
    const double pr = acc[6], pi = acc[7], q = acc[8], rr = acc[9];
    const bool ok = q > 0 && isfinite(q) && isfinite(pr) && isfinite(pi) && isfinite(rr);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (ok) {
            acc[2] = sqrt(pr * pr + pi * pi) / q;
            acc[4] += 1.0;
            acc[5] += rr > 0 ? fmax(0.0, rr - (pr * pr + pi * pi) / q) / rr : 1.0;
        } else {
            acc[2] = 0.0;
            acc[3] += 1.0;
        }
    }
    if (!ok) return;
    const float ar = (float)(pr / q), ai = (float)(pi / q);
    for (size_t id = blockIdx.x * (size_t)blockDim.x + threadIdx.x; id < n; id += (size_t)gridDim.x * blockDim.x) {
        const float2 a = c[id];
        float2 b = z[id];
        b.x += ar * a.x - ai * a.y;
        b.y += ar * a.y + ai * a.x;
        z[id] = b;
    }
}

// t = (xs - xk - mv)/rms(mv): the training target of the network for v = b - A xk, whose exact
// preconditioned image is A^-1 v = xs - xk (xs the converged solution); complex128 xs, xk
__global__ void target_kernel(const double2* __restrict__ xs, const double2* __restrict__ xk,
                              const float2* __restrict__ mv, const double* __restrict__ acc, size_t n,
                              float* __restrict__ t) {
    const double is = acc[0] > 0 ? 1.0 / sqrt(acc[0] / (double)n) : 0.0;
    for (size_t id = blockIdx.x * (size_t)blockDim.x + threadIdx.x; id < n; id += (size_t)gridDim.x * blockDim.x) {
        const double2 a = xs[id], b = xk[id];
        const float2 m = mv[id];
        t[id] = (float)((a.x - b.x - (double)m.x) * is);
        t[n + id] = (float)((a.y - b.y - (double)m.y) * is);
    }
}

unsigned nblk(size_t n) { const size_t b = (n + 255) / 256; return (unsigned)(b > 4096 ? 4096 : b); }

void free_bufs(void** ps, int n) {
    for (int i = 0; i < n; ++i) {
        if (ps[i]) cudaFree(ps[i]);
    }
}
bool grow(Buf& b, size_t bytes) {
    if (bytes <= b.cap) return true;
    cudaFree(b.p);
    b = Buf();
    if (cudaMalloc(&b.p, bytes) != cudaSuccess) { cudaGetLastError(); return false; }
    b.cap = bytes;
    return true;
}

// inference workspace for B x Z x Y x X (grown on demand, never shrunk); when the shape or the memory is new, the next
// forward zeroes the cells that it does not write
helm_status ensure_ws(helm_net* n, int B, int Z, int Y, int X) {
    if (B < 1 || Z < 2 || Y < 2 || X < 2 || Z % 2 || Y % 2 || X % 2) return HELM_ERR_ARG;
    if (B == n->B && Z == n->Z && Y == n->Y && X == n->X) return HELM_OK;
    n->B = 0;
    n->gf = cell_grid(B, Z, Y, X);
    n->gh = cell_grid(B, Z / 2, Y / 2, X / 2);
    const int c = n->c;
    const size_t pts = (size_t)B * Z * Y * X;
    if (!grow(n->xp, 5 * pts * 2) || !grow(n->y, 2 * pts * 4) || !grow(n->x, cell_bytes(n->gf, 5)) ||
        !grow(n->a1, cell_bytes(n->gf, c)) || !grow(n->u, cell_bytes(n->gf, 3 * c)) || !grow(n->d1, cell_bytes(n->gf, c)) ||
        !grow(n->p, cell_bytes(n->gh, c)) || !grow(n->b1, cell_bytes(n->gh, 2 * c)) || !grow(n->b2, cell_bytes(n->gh, 2 * c)))
        return HELM_ERR_NOMEM;
    n->fresh = true;
    n->B = B; n->Z = Z; n->Y = Y; n->X = X;
    return HELM_OK;
}

// gradient workspace for the current B x Z x Y x X (training only)
helm_status ensure_grad_ws(helm_net* n) {
    if (n->B == n->gB_ && n->Z == n->gZ_ && n->Y == n->gY_ && n->X == n->gX_) return HELM_OK;
    n->gB_ = 0;
    const int c = n->c;
    if (!grow(n->gy, cell_bytes(n->gf, 2)) || !grow(n->gC, cell_bytes(n->gf, c)) || !grow(n->gD, cell_bytes(n->gf, c)) || !grow(n->gU, cell_bytes(n->gf, 3 * c, 4)) ||
        !grow(n->gP, cell_bytes(n->gh, c, 4)) || !grow(n->gH1, cell_bytes(n->gh, 2 * c)) || !grow(n->gH2, cell_bytes(n->gh, 2 * c)))
        return HELM_ERR_NOMEM;
    n->gfresh = true;
    n->gB_ = n->B; n->gZ_ = n->Z; n->gY_ = n->Y; n->gX_ = n->X;
    return HELM_OK;
}

dim3 cell_blocks(const CellGrid& g, int C) {
    const long pts = (long)g.Z * g.Y * g.X, b = (pts + 255) / 256;
    return dim3((unsigned)(b > 1024 ? 1024 : b), (unsigned)(g.B * ((C + 7) / 8)));
}

// Zeroes what a forward or backward reads and does not write, where that may hold anything else: in new memory or a new
// shape (`fresh`, cleared), and always in a graph and once a call was recorded into one, since its replays may lie
// between any two calls and nothing here sees them.
helm_status zero_rest(helm_net* n, bool& fresh, cudaStream_t s, const Rests& rests, int count) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    HELM_CUDA_TRY(cudaStreamIsCapturing(s, &cap));
    const bool recording = cap != cudaStreamCaptureStatusNone;
    n->recorded |= recording;
    if (!fresh && !n->recorded) return HELM_OK;
    zero_rest_kernel<<<dim3(1216, count), 256, 0, s>>>(n->gf, n->gh, rests);
    HELM_CUDA_TRY(cudaGetLastError());
    if (!recording) fresh = false;
    return HELM_OK;
}

// forward of channel-first features xp into y (channel-first FP32); bounded-wait failures OR-ed into *status
helm_status forward(helm_net* n, const bf16* xp, float* y, unsigned* status, cudaStream_t s) {
    const int c = n->c;
    const CellGrid &gf = n->gf, &gh = n->gh;
    const bf16* W = n->Wb;
    const float* F = n->W;
    helm_status st;
    // (u: where its parts do not meet between cells, its last cell's channels are written one by one)
    if ((st = zero_rest(n, n->fresh, s, Rests{{{cells(n->x), 0, cell_groups(5), 1}, {cells(n->a1), 0, cell_groups(c), (c + 7) / 8},
                                              {cells(n->u), 0, cell_groups(3 * c), c % 4 ? 3 * c / 8 : (3 * c + 7) / 8},
                                              {cells(n->d1), 0, cell_groups(c), (c + 7) / 8}, {cells(n->p), 1, cell_groups(c), (c + 7) / 8},
                                              {cells(n->b1), 1, cell_groups(2 * c), (2 * c + 7) / 8},
                                              {cells(n->b2), 1, cell_groups(2 * c), (2 * c + 7) / 8}}}, 7)) != HELM_OK)
        return st;
    auto conv = [&](const CellGrid& g, int mode, int l, const Buf& in, void* out, int Cout_total, int ooff, int relu) {
        return conv_cells(g, mode, cells(in), n->ci[l], W + n->woff[l], 0, F + n->boff[l], out, n->co[l], Cout_total, ooff, relu,
                          nullptr, nullptr, n->wscr, status, s);
    };
    pack_x_kernel<<<cell_blocks(gf, 8), 256, 0, s>>>(gf, xp, cell_groups(5), cells(n->x));
    if ((st = conv(gf, CONV_CELLS, 0, n->x, cells(n->a1), c, 0, 1)) != HELM_OK) return st;
    if ((st = conv(gf, CONV_CELLS, 1, n->a1, cells(n->u), 3 * c, 2 * c, 1)) != HELM_OK) return st;   // a2 lives in u
    avgpool2_kernel<<<cell_blocks(gh, c), 256, 0, s>>>(gf, gh, cells(n->u), cell_groups(3 * c), 2 * c, c, cells(n->p),
                                                       cell_groups(c));
    if ((st = conv(gh, CONV_CELLS, 2, n->p, cells(n->b1), 2 * c, 0, 1)) != HELM_OK) return st;
    if ((st = conv(gh, CONV_CELLS, 3, n->b1, cells(n->b2), 2 * c, 0, 1)) != HELM_OK) return st;
    upsample2_kernel<<<cell_blocks(gh, 2 * c), 256, 0, s>>>(gf, gh, cells(n->b2), cell_groups(2 * c), 2 * c, cells(n->u),
                                                            cell_groups(3 * c));
    if ((st = conv(gf, CONV_CELLS, 4, n->u, cells(n->d1), c, 0, 1)) != HELM_OK) return st;
    return conv(gf, CONV_PLANAR, 5, n->d1, y, 2, 0, 0);
}

}  // namespace

helm_status ensure_field_ws(helm_net* n, size_t npts);

extern "C" {

size_t helm_net_num_params(const helm_net* n) { return n ? n->nparam : 0; }

helm_status helm_net_create(int width, unsigned long long seed, helm_net** out) {
    if (!out) return HELM_ERR_ARG;
    *out = nullptr;   // on every error return
    if (width < 1 || width > 64) return HELM_ERR_ARG;
    helm_net* n = new helm_net();
    n->c = width;
    const int c = width;
    const int co[6] = {c, c, 2 * c, 2 * c, c, 2}, ci[6] = {5, c, c, 2 * c, 3 * c, c};
    size_t off = 0;
    for (int l = 0; l < 6; ++l) {
        n->co[l] = co[l]; n->ci[l] = ci[l];
        n->woff[l] = off; off += (size_t)co[l] * ci[l] * 27;
        n->boff[l] = off; off += co[l];
    }
    n->nparam = off;
    std::vector<float> h(off, 0.f);
    unsigned long long st = seed * 2862933555777941757ull + 3037000493ull;
    auto rnd = [&]() {   // splitmix64 -> uniform (0,1)
        st += 0x9E3779B97F4A7C15ull;
        unsigned long long z = st;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        z ^= z >> 31;
        return ((z >> 11) + 0.5) * (1.0 / 9007199254740992.0);
    };
    for (int l = 0; l < 6; ++l) {
        const double std = sqrt(2.0 / (27.0 * ci[l])) * (l == 5 ? 0.1 : 1.0);
        for (size_t k = 0; k < (size_t)co[l] * ci[l] * 27; ++k) {
            const double u1 = rnd(), u2 = rnd();
            h[n->woff[l] + k] = (float)(std * sqrt(-2.0 * log(u1)) * cos(2 * M_PI * u2));
        }
    }
    size_t scr = 0;   // arranged weights of the largest layer, in either direction
    for (int l = 0; l < 6; ++l) {
        scr = std::max(scr, conv_scratch_bytes(ci[l], co[l]));
        scr = std::max(scr, conv_scratch_bytes(co[l], ci[l]));
    }
    bool ok = cudaMalloc(&n->W, off * 4) == cudaSuccess && cudaMalloc(&n->G, off * 4) == cudaSuccess &&
              cudaMalloc(&n->Mom, off * 4) == cudaSuccess && cudaMalloc(&n->Vel, off * 4) == cudaSuccess &&
              cudaMalloc(&n->Wb, off * 2) == cudaSuccess && cudaMalloc(&n->stats, 16 * sizeof(double)) == cudaSuccess &&
              cudaMalloc(&n->wscr, scr) == cudaSuccess && cudaMalloc(&n->status, sizeof(unsigned)) == cudaSuccess;
    if (!ok) { cudaGetLastError(); helm_net_destroy(n); return HELM_ERR_NOMEM; }
    cudaMemcpy(n->W, h.data(), off * 4, cudaMemcpyHostToDevice);
    cudaMemset(n->G, 0, off * 4);
    cudaMemset(n->Mom, 0, off * 4);
    cudaMemset(n->Vel, 0, off * 4);
    cudaMemset(n->stats, 0, 16 * sizeof(double));
    cudaMemset(n->status, 0, sizeof(unsigned));
    if (conv_prepare() != HELM_OK) { cudaGetLastError(); helm_net_destroy(n); return HELM_ERR_CUDA; }
    to_bf16_kernel<<<(unsigned)((off + 255) / 256), 256>>>(n->W, n->Wb, off);
    if (cudaDeviceSynchronize() != cudaSuccess) { cudaGetLastError(); helm_net_destroy(n); return HELM_ERR_CUDA; }
    *out = n;
    return HELM_OK;
}

void helm_net_destroy(helm_net* n) {
    if (!n) return;
    void* ps[] = {n->W, n->G, n->Mom, n->Vel, n->Wb, n->stats, n->vbuf, n->cbuf, n->az0, n->ac, n->wscr, n->status,
                  n->xp.p, n->y.p, n->x.p, n->a1.p, n->u.p, n->d1.p, n->p.p, n->b1.p, n->b2.p, n->gy.p, n->gC.p, n->gD.p, n->gH1.p,
                  n->gH2.p, n->gU.p, n->gP.p};
    for (void* p : ps) if (p) cudaFree(p);
    delete n;
}

helm_status helm_net_set_params(helm_net* n, const float* host, size_t count) {
    if (!n || !host || count != n->nparam) return HELM_ERR_ARG;
    HELM_CUDA_TRY(cudaMemcpy(n->W, host, count * 4, cudaMemcpyHostToDevice));
    to_bf16_kernel<<<(unsigned)((count + 255) / 256), 256>>>(n->W, n->Wb, count);
    HELM_CUDA_TRY(cudaDeviceSynchronize());
    return HELM_OK;
}

helm_status helm_net_get_params(helm_net* n, float* host, size_t count) {
    if (!n || !host || count != n->nparam) return HELM_ERR_ARG;
    HELM_CUDA_TRY(cudaMemcpy(host, n->W, count * 4, cudaMemcpyDeviceToHost));
    return HELM_OK;
}

helm_status helm_net_get_grads(helm_net* n, float* host, size_t count) {
    if (!n || !host || count != n->nparam) return HELM_ERR_ARG;
    HELM_CUDA_TRY(cudaMemcpy(host, n->G, count * 4, cudaMemcpyDeviceToHost));
    unsigned st = 0;
    HELM_CUDA_TRY(cudaMemcpy(&st, n->status, sizeof(unsigned), cudaMemcpyDeviceToHost));
    if (st & HELM_DEV_WAIT) return HELM_ERR_ITER_LIMIT;
    return HELM_OK;
}

helm_status helm_net_zero_grad(helm_net* n, void* stream) {
    if (!n) return HELM_ERR_ARG;
    HELM_CUDA_TRY(cudaMemsetAsync(n->G, 0, n->nparam * 4, (cudaStream_t)stream));
    return HELM_OK;
}

helm_status helm_net_forward(helm_net* n, const void* x, float* y, int B, int Z, int Y, int X, void* stream) {
    if (!n || !x || !y || B < 1) return HELM_ERR_ARG;
    helm_status st = ensure_ws(n, B, Z, Y, X);
    if (st != HELM_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    if ((st = forward(n, (const bf16*)x, y, n->status, s)) != HELM_OK) return st;
    HELM_CUDA_TRY(cudaGetLastError());
    return HELM_OK;
}

helm_status helm_net_backward(helm_net* n, const float* gy, void* stream) {
    if (!n || !gy || !n->B) return HELM_ERR_ARG;
    helm_status st = ensure_grad_ws(n);
    if (st != HELM_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    const int c = n->c;
    const CellGrid &gf = n->gf, &gh = n->gh;
    const bf16* W = n->Wb;
    float* G = n->G;
    if ((st = zero_rest(n, n->gfresh, s, Rests{{{cells(n->gy), 0, cell_groups(2), 1}, {cells(n->gC), 0, cell_groups(c), (c + 7) / 8},
                                               {cells(n->gD), 0, cell_groups(c), (c + 7) / 8},
                                               {cells(n->gH1), 1, cell_groups(2 * c), (2 * c + 7) / 8},
                                               {cells(n->gH2), 1, cell_groups(2 * c), (2 * c + 7) / 8}}}, 5)) != HELM_OK)
        return st;
    auto wgrad = [&](const CellGrid& g, int l, const Buf& in, const Buf& gr) {
        return wgrad_cells(g, cells(in), n->ci[l], cells(gr), n->co[l], G + n->woff[l], n->status, s);
    };
    // data gradient of layer l (flipped, transposed weights): CONV_GRAD masks by the layer input's ReLU and sums
    // the bias gradient of the layer that produced it, bl
    auto dgrad = [&](const CellGrid& g, int mode, int l, const Buf& gr, const Buf& out, const Buf* mask, int bl) {
        return conv_cells(g, mode, cells(gr), n->co[l], W + n->woff[l], 1, nullptr, out.p, n->ci[l], n->ci[l], 0, 0,
                          mask ? cells(*mask) : nullptr, mask ? G + n->boff[bl] : nullptr, n->wscr, n->status, s);
    };
    // layer 6 (linear): d1 gradient with the ReLU mask of d1
    pack_gy_kernel<<<cell_blocks(gf, 2), 256, 0, s>>>(gf, gy, cell_groups(2), cells(n->gy), G + n->boff[5]);
    if ((st = wgrad(gf, 5, n->d1, n->gy)) != HELM_OK) return st;
    if ((st = dgrad(gf, CONV_GRAD, 5, n->gy, n->gC, &n->d1, 4)) != HELM_OK) return st;
    // layer 5: u gradient (no mask: u mixes up(b2) and a2, masks applied below)
    if ((st = wgrad(gf, 4, n->u, n->gC)) != HELM_OK) return st;
    if ((st = dgrad(gf, CONV_F32CELLS, 4, n->gC, n->gU, nullptr, 0)) != HELM_OK) return st;
    // up branch: adjoint of upsample2 with the ReLU mask of b2
    upsample2_adj_kernel<<<cell_blocks(gh, 2 * c), 256, 0, s>>>(gf, gh, floats(n->gU), cell_groups(3 * c), cells(n->b2),
                                                                cells(n->gH1), cell_groups(2 * c), 2 * c, G + n->boff[3]);
    // layer 4: b1 gradient with mask(b1)
    if ((st = wgrad(gh, 3, n->b1, n->gH1)) != HELM_OK) return st;
    if ((st = dgrad(gh, CONV_GRAD, 3, n->gH1, n->gH2, &n->b1, 2)) != HELM_OK) return st;
    // layer 3: p gradient (no ReLU on p)
    if ((st = wgrad(gh, 2, n->p, n->gH2)) != HELM_OK) return st;
    if ((st = dgrad(gh, CONV_F32CELLS, 2, n->gH2, n->gP, nullptr, 0)) != HELM_OK) return st;
    // a2 gradient: skip part + adjoint of avgpool2, masked by a2
    skip_grad_kernel<<<cell_blocks(gf, c), 256, 0, s>>>(gf, gh, floats(n->gU), floats(n->gP), cell_groups(c), cells(n->u),
                                                        cell_groups(3 * c), 2 * c, c, cells(n->gC), cell_groups(c),
                                                        G + n->boff[1]);
    // layer 2: a1 gradient with mask(a1)
    if ((st = wgrad(gf, 1, n->a1, n->gC)) != HELM_OK) return st;
    if ((st = dgrad(gf, CONV_GRAD, 1, n->gC, n->gD, &n->a1, 0)) != HELM_OK) return st;
    // layer 1
    if ((st = wgrad(gf, 0, n->x, n->gD)) != HELM_OK) return st;
    HELM_CUDA_TRY(cudaGetLastError());
    return HELM_OK;
}

helm_status helm_net_adam(helm_net* n, float lr, float b1, float b2, float eps, int step, void* stream) {
    if (!n || step < 1) return HELM_ERR_ARG;
    const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
    adam_kernel<<<(unsigned)((n->nparam + 255) / 256), 256, 0, (cudaStream_t)stream>>>(n->W, n->G, n->Mom, n->Vel, n->Wb,
                                                                                      n->nparam, lr, b1, b2, eps, c1, c2);
    HELM_CUDA_TRY(cudaGetLastError());
    return HELM_OK;
}

helm_status helm_net_mse(const float* y, const float* t, float* gy, size_t count, double* loss_dev, void* stream) {
    if (!y || !t || !gy || !loss_dev || !count) return HELM_ERR_ARG;
    mse_kernel<<<nblk(count), 256, 0, (cudaStream_t)stream>>>(y, t, gy, count, loss_dev);
    HELM_CUDA_TRY(cudaGetLastError());
    return HELM_OK;
}

helm_status helm_net_features(helm_ctx* c, helm_net* n, const void* v, const void* mv, void* x, void* stream) {
    if (!c || !n || !v || !mv || !x) return HELM_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const size_t N = c->npts;
    double* acc = n->stats;
    bf16* X = (bf16*)x;
    HELM_CUDA_TRY(cudaMemsetAsync(acc, 0, 2 * sizeof(double), s));
    sumsq_kernel<<<nblk(N), 256, 0, s>>>((const float2*)v, N, acc);
    sumsq_kernel<<<nblk(N), 256, 0, s>>>((const float2*)mv, N, acc + 1);
    feat_pair_kernel<<<nblk(N), 256, 0, s>>>((const float2*)v, acc, N, X, X + N);
    feat_pair_kernel<<<nblk(N), 256, 0, s>>>((const float2*)mv, acc + 1, N, X + 2 * N, X + 3 * N);
    feat_contrast_kernel<<<nblk(N), 256, 0, s>>>(c->k2_f, (float)(1.0 / (c->k0 * c->k0)), N, X + 4 * N);
    HELM_CUDA_TRY(cudaGetLastError());
    return HELM_OK;
}

helm_status helm_net_target(helm_ctx* c, helm_net* n, const void* xs, const void* xk, const void* mv, float* t,
                            void* stream) {
    if (!c || !n || !xs || !xk || !mv || !t) return HELM_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const size_t N = c->npts;
    double* acc = n->stats + 15;
    HELM_CUDA_TRY(cudaMemsetAsync(acc, 0, sizeof(double), s));
    sumsq_kernel<<<nblk(N), 256, 0, s>>>((const float2*)mv, N, acc);
    target_kernel<<<nblk(N), 256, 0, s>>>((const double2*)xs, (const double2*)xk, (const float2*)mv, acc, N, t);
    HELM_CUDA_TRY(cudaGetLastError());
    return HELM_OK;
}

helm_status helm_attach_net(helm_ctx* c, helm_net* n) {
    if (!c) return HELM_ERR_ARG;
    if (n) {
        if (!c->opt.flexible || c->nx % 2 || c->ny % 2 || c->nz % 2) return HELM_ERR_ARG;
        helm_status st = ensure_ws(n, 1, c->nz, c->ny, c->nx);
        if (st != HELM_OK) return st;
        if ((st = ensure_field_ws(n, c->npts)) != HELM_OK) return st;
    }
    c->net = n;
    return HELM_OK;
}

helm_status helm_net_stats(helm_net* n, double* host6) {
    if (!n || !host6) return HELM_ERR_ARG;
    HELM_CUDA_TRY(cudaMemcpy(host6, n->stats, 6 * sizeof(double), cudaMemcpyDeviceToHost));
    return HELM_OK;
}

}  // extern "C"

// solver-side field buffers for npts points
helm_status ensure_field_ws(helm_net* n, size_t npts) {
    if (npts <= n->fcap) return HELM_OK;
    void* ps[] = {n->vbuf, n->cbuf, n->az0, n->ac};
    free_bufs(ps, 4);
    n->vbuf = n->cbuf = n->az0 = n->ac = nullptr;
    n->fcap = 0;
    const size_t b = npts * sizeof(float2);
    const bool ok = cudaMalloc(&n->vbuf, b) == cudaSuccess && cudaMalloc(&n->cbuf, b) == cudaSuccess &&
                    cudaMalloc(&n->az0, b) == cudaSuccess && cudaMalloc(&n->ac, b) == cudaSuccess;
    if (!ok) { cudaGetLastError(); return HELM_ERR_NOMEM; }
    n->fcap = npts;
    return HELM_OK;
}

// Before M^-1: the per-call sums are reset, the r features written and v = sigma[sidx] r kept (r may be
// overwritten by M^-1 afterwards).
helm_status learned_pre(helm_ctx* c, const float2* r, const double* sigma, int sidx, cudaStream_t s) {
    helm_net* n = c->net;
    helm_status st = ensure_ws(n, 1, c->nz, c->ny, c->nx);
    if (st != HELM_OK) return st;
    if ((st = ensure_field_ws(n, c->npts)) != HELM_OK) return st;
    const size_t N = c->npts;
    double* acc = n->stats;
    prof_begin(c, s, PROF_LEARNED);
    HELM_CUDA_TRY(cudaMemsetAsync(acc, 0, 2 * sizeof(double), s));
    HELM_CUDA_TRY(cudaMemsetAsync(acc + 6, 0, 4 * sizeof(double), s));
    sumsq_kernel<<<nblk(N), 256, 0, s>>>(r, N, acc);
    feat_v_kernel<<<nblk(N), 256, 0, s>>>(r, acc, N, cells(n->xp), cells(n->xp) + N, sigma, sidx, n->vbuf);
    feat_contrast_kernel<<<nblk(N), 256, 0, s>>>(c->k2_f, (float)(1.0 / (c->k0 * c->k0)), N, cells(n->xp) + 4 * N);
    prof_end(c, s);
    HELM_CUDA_TRY(cudaGetLastError());
    return HELM_OK;
}

// After M^-1 (z = z0 = M^-1 v): c = s N(features), then the minimal-residual step z = z0 + alpha c.
helm_status learned_post(helm_ctx* c, float2* z, cudaStream_t s) {
    helm_net* n = c->net;
    const size_t N = c->npts;
    double* acc = n->stats;
    helm_status st;
    prof_begin(c, s, PROF_LEARNED);
    sumsq_kernel<<<nblk(N), 256, 0, s>>>(z, N, acc + 1);
    feat_pair_kernel<<<nblk(N), 256, 0, s>>>(z, acc + 1, N, cells(n->xp) + 2 * N, cells(n->xp) + 3 * N);
    if ((st = forward(n, cells(n->xp), floats(n->y), c->status_d, s)) != HELM_OK) return st;
    make_c_kernel<<<nblk(N), 256, 0, s>>>(floats(n->y), acc, N, n->cbuf);
    prof_end(c, s);
    if ((st = launch_stencil_f32_cls(c, z, n->az0, nullptr, 0, PROF_LEARNED, s)) != HELM_OK) return st;
    if ((st = launch_stencil_f32_cls(c, n->cbuf, n->ac, nullptr, 0, PROF_LEARNED, s)) != HELM_OK) return st;
    prof_begin(c, s, PROF_LEARNED);
    mr_dots_kernel<<<nblk(N), 256, 0, s>>>(n->vbuf, n->az0, n->ac, N, acc);
    mr_apply_kernel<<<nblk(N), 256, 0, s>>>(n->cbuf, acc, N, z);
    prof_end(c, s);
    HELM_CUDA_TRY(cudaGetLastError());
    return HELM_OK;
}
