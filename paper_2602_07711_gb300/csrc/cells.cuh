// Activation layout of the learned correction: cells of 8 channels (BF16, 16 bytes) on a grid with a zero halo
// of one point, [batch][channel group][Z + 2][Y + 2][pitch] cells, point (z, y, x) at (z + 1, y + 1, x + 1).  Channels
// of the last group beyond the tensor's are zero; where an odd number of groups leaves half of a 16-channel chunk, the
// kernels stage the zeros that follow the tensor (rounding the groups up to even ones instead took 1.6 times the
// workspace at width 4).  Halo cells are zeroed when the workspace takes a new shape (zero_rest_kernel) and never written, so a plane can be walked along its flattened index:
// the points (y, x) sit at pitch + 1 + y pitch + x, and what lies between rows is zero.  The pitch is at least 16,
// so that 15 points beyond the last one (a K step of the weight gradient) are halo too.  Tiles may read past the
// last plane: CELL_SLACK zeroed cells follow every tensor.  FP32 cells (gradients that are summed further) are 8
// floats on the same grid; their halo is never read.
#pragma once
#include "common.cuh"
#include <cuda_bf16.h>

typedef __nv_bfloat16 bf16;

constexpr long CELL_SLACK = 4096;

struct CellGrid {
    int B, Z, Y, X, pitch, span;   // span: flattened points from the first to the last of a plane
    long plane, vol;               // cells of a padded plane and of a channel group
};
inline CellGrid cell_grid(int B, int Z, int Y, int X) {
    CellGrid g;
    g.B = B; g.Z = Z; g.Y = Y; g.X = X;
    g.pitch = X + 2 < 16 ? 16 : X + 2;
    g.span = (Y - 1) * g.pitch + X;
    g.plane = (long)(Y + 2) * g.pitch;
    g.vol = (Z + 2) * g.plane;
    return g;
}
__host__ __device__ inline int cell_groups(int C) { return (C + 7) / 8; }
inline size_t cell_bytes(const CellGrid& g, int C, int elem = 2) {
    return ((size_t)g.B * cell_groups(C) * g.vol + CELL_SLACK) * 8 * elem;
}

__device__ __forceinline__ uint32_t pack2(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ uint4 pack_cell(const float* v) {
    return make_uint4(pack2(v[0], v[1]), pack2(v[2], v[3]), pack2(v[4], v[5]), pack2(v[6], v[7]));
}
// channel j (a constant after unrolling) of a cell
__device__ __forceinline__ float cell_value(const uint4& q, int j) {
    const uint32_t w = j < 2 ? q.x : (j < 4 ? q.y : (j < 6 ? q.z : q.w));
    return __uint_as_float(j & 1 ? w & 0xFFFF0000u : w << 16);
}

// Sums over the 32 lanes of 16 (8) values each: at every step a lane keeps half of the values and adds the other
// half's share from its partner.  The result of value lane_fold16_channel(lane) (lane_fold8_channel) is returned
// to that lane (the same to both lanes of a pair; to four lanes for 8 values).
__device__ __forceinline__ float lane_fold16(const float* v, int lane) {
    float f[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) f[i] = v[i];
#pragma unroll
    for (int h = 8, o = 16; h >= 1; h >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const float keep = up ? f[i + h] : f[i], send = up ? f[i] : f[i + h];
            f[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    return f[0] + __shfl_xor_sync(0xffffffffu, f[0], 1);
}
__device__ __forceinline__ int lane_fold16_channel(int lane) {
    return (lane & 16 ? 8 : 0) + (lane & 8 ? 4 : 0) + (lane & 4 ? 2 : 0) + (lane & 2 ? 1 : 0);
}
__device__ __forceinline__ float lane_fold8(const float* v, int lane) {
    float f[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) f[i] = v[i];
#pragma unroll
    for (int h = 4, o = 16; h >= 1; h >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const float keep = up ? f[i + h] : f[i], send = up ? f[i] : f[i + h];
            f[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    f[0] += __shfl_xor_sync(0xffffffffu, f[0], 2);
    return f[0] + __shfl_xor_sync(0xffffffffu, f[0], 1);
}
__device__ __forceinline__ int lane_fold8_channel(int lane) {
    return (lane & 16 ? 4 : 0) + (lane & 8 ? 2 : 0) + (lane & 4 ? 1 : 0);
}

// conv_tc.cu.  Output of conv_cells: BF16 cells at channel ooff of a tensor of Cout_total channels; FP32
// channel-first [B][Cout][Z][Y][X]; FP32 cells; BF16 cells zeroed where mask <= 0, with gb[o] += the FP32 sum
// over points
enum { CONV_CELLS = 0, CONV_PLANAR = 1, CONV_F32CELLS = 2, CONV_GRAD = 3 };
size_t conv_scratch_bytes(int Cin, int Cout);
helm_status conv_prepare();
helm_status conv_cells(const CellGrid& g, int mode, const bf16* in, int Cin, const bf16* w, int wmode, const float* bias,
                       void* out, int Cout, int Cout_total, int ooff, int relu, const bf16* mask, float* gb, bf16* wscr,
                       unsigned* status, cudaStream_t s);
helm_status wgrad_cells(const CellGrid& g, const bf16* in, int Cin, const bf16* gr, int Cout, float* gw, unsigned* status,
                        cudaStream_t s);
