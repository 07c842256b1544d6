// High-order closure of the Sommerfeld condition on collocated grids (the constant-k test problems of
// Sec. 2.1 close the fourth- and sixth-order schemes with a high-order three-point approximation of the
// ABC; the paper gives no formula, this is our reading).
//
// Per face, with B the boundary node, I its interior neighbour, G the ghost and h the normal step:
//     U_G = U_I + i k0 sum_{m=0..2} c_m (-1)^m L^m U_B,      c_m = 2 h^(2m+1) / (2m+1)!,
// L = k0^2 + (tangential second derivatives), from the Taylor series of u about B in the normal
// direction with every odd normal derivative reduced by the ABC and the equation (k = k0 on the face).
// m = 0 alone is the three-point rule of the preconditioner.  The tangential derivatives are sixth-order
// differences along the face: seven centred points where they fit, the eight nearest points otherwise.
// The faces are filled x, then y, then z; a face covers the ghost columns of the directions filled before
// it, so edge and corner ghosts come from the rule applied along an already-filled ghost line.
// The closure's f part (U-independent) belongs to the right-hand side the caller supplies.
//
// Layout: the ghosts go into a padded array (nx+2) x (ny+2) x (nz+2), x fastest.  The complex64 matvec reads the
// interior from the operand itself and only the shell from there; for the general kernels (complex128,
// double-float) the operand is copied into the interior too.  Per face two launches: V1 = L U_B into a scratch face,
// then the ghost from U_I, U_B, V1 and L V1 (formed on the fly).  The arithmetic is FP64 for complex128 and
// double-float operands and double-float (about 44 bits) for complex64 ones, whose ghosts are rounded to FP32: the
// faces are O(N^2) work, so a launch is a chain of latencies, and on GB300 the 34 conversions and 32 products of a
// point in FP64 were the longest part of it.  The loads of a point are independent (eight per direction).
// Double-float has FP32's exponent range, and L U and L^2 U carry 1/h^2 and 1/h^4: there L is scaled by a power of two
// that brings its row sums to one at most (make_face_consts), and the Taylor weights undo it.  No intermediate is then
// larger than the operand, none that matters is lost below it, and no other bit changes.
// With FP64 faces instead, the matvec of thirteen grids (36 to 198 points a side, 14 to 55 points per wavelength) has the
// same error against 64 bits to five digits, at 100^3 the same bits, and takes 64.5 us instead of 50.7.
// Measured at 100^3, complex64: 8 and 7 us per launch in FP64 with loops over the rows -> 5.1-5.8 us; the whole
// matvec (its stencil kernel in stencil_fast.cu) 142 -> 64 us.
#include "common.cuh"
#include "dfloat.cuh"
#include <cmath>
#include <cstring>

namespace {

constexpr int HO_NT = 64;   // small blocks: a face has tens of thousands of points for 152 SMs

// ---- arithmetic of the faces: FP64, or double-float for complex64 operands -------------------------------
struct A64 {
    typedef double2 V;    // value
    typedef double S;     // real scalar
    typedef double2 St;   // stored value (scratch faces)
    static constexpr double row = 1.0;   // scale of the difference rows
    static double scale_of(double) { return 1.0; }   // scale of L, from a bound of its row sums
    static S cst(double v) { return v; }
    static __device__ __forceinline__ S minus_one() { return -1.0; }
    static __device__ __forceinline__ V zero() { return make_double2(0.0, 0.0); }
    static __device__ __forceinline__ V add(V a, V b) { return make_double2(a.x + b.x, a.y + b.y); }
    static __device__ __forceinline__ V mul(V a, S s) { return make_double2(a.x * s, a.y * s); }
    static __device__ __forceinline__ V times_i(V a) { return make_double2(-a.y, a.x); }
    static __device__ __forceinline__ V ld(const double2* p, long long i) { return p[i]; }
    static __device__ __forceinline__ V ld(const float4* p, long long i) {
        const float4 v = p[i];
        return make_double2((double)v.x + (double)v.z, (double)v.y + (double)v.w);
    }
    static __device__ __forceinline__ void st(double2* p, long long i, V v) { p[i] = v; }
    static __device__ __forceinline__ void st(float4* p, long long i, V v) {
        const float rh = (float)v.x, ih = (float)v.y;
        p[i] = make_float4(rh, ih, (float)(v.x - (double)rh), (float)(v.y - (double)ih));
    }
};
struct ADF {
    typedef cdf V;
    typedef df S;
    typedef float4 St;
    static constexpr double row = 1.0 / 256;   // the one-sided rows sum to 194 in magnitude
    static double scale_of(double bound) { return ldexp(1.0, -(int)ceil(log2(bound))); }
    static S cst(double v) {
        const float h = (float)v;
        return df{h, (float)(v - (double)h)};
    }
    static __device__ __forceinline__ S minus_one() { return df{-1.f, 0.f}; }
    static __device__ __forceinline__ V zero() { return cdf_zero(); }
    static __device__ __forceinline__ V add(V a, V b) { return cdf_add(a, b); }
    static __device__ __forceinline__ V mul(V a, S s) { return cdf_scale(a, s); }
    static __device__ __forceinline__ V times_i(V a) {
        return cdf{make_float2(-a.hi.y, a.hi.x), make_float2(-a.lo.y, a.lo.x)};
    }
    static __device__ __forceinline__ V ld(const float2* p, long long i) { return cdf_from_f2(p[i]); }
    static __device__ __forceinline__ V ld(const float4* p, long long i) { return cdf_from4(p[i]); }
    static __device__ __forceinline__ void st(float2* p, long long i, V v) { p[i] = cdf_round(v); }
    static __device__ __forceinline__ void st(float4* p, long long i, V v) { p[i] = cdf_to4(v); }
};
template <class M> struct ArithOf { typedef A64 T; };
template <> struct ArithOf<float2> { typedef ADF T; };

// Rows of the second-derivative stencils (times h^2 and A::row) over eight consecutive nodes: nodes 0, 1, 2 of a line
// (one-sided), inner nodes (seven centred weights and a zero), node n - 4 (a zero and the seven), nodes n - 3 .. n - 1
template <class A>
struct Wts {
    typename A::S w[8][8];
};

struct Face {
    int axis;            // 0 x, 1 y, 2 z
    int la, lb;          // face extents along the tangential axes ta, tb (array order: ta slower)
    int sa0, sb0;        // first padded coordinate along ta, tb
    long long sn, sa, sb;  // padded strides along the normal and the tangential axes
    int nb_lo, nb_hi;    // padded normal index of the two boundary planes (1 and n)
};
template <class A>
struct FaceC {
    // L and L^2 are formed as f L and f^2 L^2
    typename A::S iha2, ihb2;      // f / (A::row h_ta^2), f / (A::row h_tb^2)
    typename A::S c0, mc1, c2;     // Taylor weights of the normal step: c_0, -c_1 / f, c_2 / f^2
    typename A::S c1, k0, kk, mkk; // c_1, k0, f k0^2, -k0^2 (c_1, c_2 and -k0^2 of the closure's f part: FP64, f = 1)
};

// the row of node i on a line of n nodes, and its first node
__device__ __forceinline__ int lap_row(int i, int n, int& first) {
    first = min(max(i - 3, 0), n - 8);
    return i < 3 ? i : (i <= n - 5 ? 3 : i - (n - 8));
}

// L V at face point (ia, ib): at(ia, ib) gives V
template <class A, class At>
__device__ __forceinline__ typename A::V apply_L(const Face& f, const FaceC<A>& k, const Wts<A>& W, const At& at, int ia, int ib) {
    int sa, sb;
    const int ra = lap_row(ia, f.la, sa), rb = lap_row(ib, f.lb, sb);
    typename A::V ua[8], ub[8];
    const typename A::V v = at(ia, ib);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        ua[q] = at(sa + q, ib);
        ub[q] = at(ia, sb + q);
    }
    typename A::V s = A::zero(), t = s;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        s = A::add(s, A::mul(ua[q], W.w[ra][q]));
        t = A::add(t, A::mul(ub[q], W.w[rb][q]));
    }
    return A::add(A::mul(v, k.kk), A::add(A::mul(s, k.iha2), A::mul(t, k.ihb2)));
}

// The operand with its ghosts: the interior from U (from P where U is NULL), the shell from the padded P
template <class M>
struct Operand {
    const M* U;
    const M* P;
    int nx, ny, nz;
    typedef typename ArithOf<M>::T A;
    // padded coordinates
    __device__ __forceinline__ typename A::V at(int X, int Y, int Z) const {
        if (U && X >= 1 && X <= nx && Y >= 1 && Y <= ny && Z >= 1 && Z <= nz)
            return A::ld(U, ((long long)(Z - 1) * ny + (Y - 1)) * nx + (X - 1));
        return A::ld(P, ((long long)Z * (ny + 2) + Y) * (nx + 2) + X);
    }
    // point (ia, ib) of the face's plane with normal index n
    __device__ __forceinline__ typename A::V face(const Face& f, int n, int ia, int ib) const {
        const int a = ia + f.sa0, b = ib + f.sb0;
        return f.axis == 0 ? at(n, b, a) : (f.axis == 1 ? at(b, n, a) : at(b, a, n));
    }
};

// copy the operand into the interior of the padded array
template <class M>
__global__ void ho_copy_kernel(int nx, int ny, int nz, const M* __restrict__ U, M* __restrict__ P) {
    const long long n = (long long)nx * ny * nz;
    for (long long id = blockIdx.x * (long long)blockDim.x + threadIdx.x; id < n; id += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(id % nx);
        const long long r = id / nx;
        const int j = (int)(r % ny), l = (int)(r / ny);
        P[((long long)(l + 1) * (ny + 2) + (j + 1)) * (nx + 2) + (i + 1)] = U[id];
    }
}

// S[side][ia][ib] = (f) L U_B on both boundary planes of one direction
template <class M, class A>
__global__ void __launch_bounds__(HO_NT) ho_lap_kernel(const __grid_constant__ Face f, const __grid_constant__ FaceC<A> k,
                                                       const __grid_constant__ Wts<A> W, const Operand<M> op,
                                                       typename A::St* S) {
    grid_wait();
    grid_trigger();
    const int per = f.la * f.lb;
    const int id = blockIdx.x * HO_NT + threadIdx.x;
    if (id >= 2 * per) return;
    const int side = id >= per, q = id - side * per;
    const int n = side ? f.nb_hi : f.nb_lo;
    A::st(S, id, apply_L<A>(f, k, W, [&](int ia, int ib) { return op.face(f, n, ia, ib); }, q / f.lb, q % f.lb));
}

// U_G = U_I + i k0 (c0 U_B - c1 L U_B + c2 L^2 U_B) on both ghost planes of one direction, plus (when fd
// is given; FP64 only) the f part s [c1 f_n + c2 (f_nnn - k0^2 f_n - lap_T f_n)], s = -1 near face, +1 far face;
// fd holds [side][field][ia][ib] with the fields f_n, f_nnn, lap_T f_n (derivatives along the axis).
template <class M, class A>
__global__ void __launch_bounds__(HO_NT) ho_ghost_kernel(const __grid_constant__ Face f, const __grid_constant__ FaceC<A> k,
                                                         const __grid_constant__ Wts<A> W, const Operand<M> op, M* P,
                                                         const typename A::St* S, const double2* __restrict__ fd) {
    typedef typename A::V V;
    grid_wait();
    grid_trigger();
    const int per = f.la * f.lb;
    const int id = blockIdx.x * HO_NT + threadIdx.x;
    if (id >= 2 * per) return;
    const int side = id >= per, q = id - side * per;
    const int ia = q / f.lb, ib = q % f.lb;
    const int pb = side ? f.nb_hi : f.nb_lo;
    const int pi = side ? pb - 1 : pb + 1;
    const int pg = side ? pb + 1 : pb - 1;
    const typename A::St* L1 = S + (long long)side * per;
    const V ub = op.face(f, pb, ia, ib), ui = op.face(f, pi, ia, ib);
    const V v1 = A::ld(L1, q);
    const V v2 = apply_L<A>(f, k, W, [&](int a, int b) { return A::ld(L1, a * f.lb + b); }, ia, ib);
    const V t = A::add(A::mul(ub, k.c0), A::add(A::mul(v1, k.mc1), A::mul(v2, k.c2)));
    V g = A::add(ui, A::times_i(A::mul(t, k.k0)));
    if constexpr (sizeof(typename A::S) == sizeof(double) && sizeof(M) == sizeof(double2)) {
        if (fd) {
            const long long fb = (long long)side * 3 * per + q;
            const V fn = A::ld(fd, fb), fnnn = A::ld(fd, fb + per), flt = A::ld(fd, fb + 2 * per);
            const V part = A::add(A::mul(fn, k.c1), A::mul(A::add(fnnn, A::add(A::mul(fn, k.mkk), A::mul(flt, A::minus_one()))), k.c2));
            g = A::add(g, side ? part : A::mul(part, A::minus_one()));
        }
    }
    A::st(P, pg * f.sn + (ia + f.sa0) * f.sa + (ib + f.sb0) * f.sb, g);
}

// Second-derivative weights on offsets o_k (Taylor conditions sum_k w_k o_k^q / q! = [q == 2]), FP64
// Gaussian elimination with partial pivoting on the small Vandermonde system.
void fd_weights(const double* o, int n, double* w) {
    double A[8][9];
    for (int q = 0; q < n; ++q) {
        double fact = 1.0;
        for (int t = 2; t <= q; ++t) fact *= t;
        for (int k = 0; k < n; ++k) A[q][k] = std::pow(o[k], q) / fact;
        A[q][n] = q == 2 ? 1.0 : 0.0;
    }
    for (int col = 0; col < n; ++col) {
        int piv = col;
        for (int r = col + 1; r < n; ++r) if (std::fabs(A[r][col]) > std::fabs(A[piv][col])) piv = r;
        if (piv != col) for (int k = 0; k <= n; ++k) std::swap(A[col][k], A[piv][k]);
        for (int r = col + 1; r < n; ++r) {
            const double m = A[r][col] / A[col][col];
            for (int k = col; k <= n; ++k) A[r][k] -= m * A[col][k];
        }
    }
    for (int r = n - 1; r >= 0; --r) {
        double s = A[r][n];
        for (int k = r + 1; k < n; ++k) s -= A[r][k] * w[k];
        w[r] = s / A[r][r];
    }
}

template <class A>
Wts<A> make_weights() {
    Wts<A> W;
    double o[8], wc[7], w[8][8] = {};
    for (int k = 0; k < 7; ++k) o[k] = k - 3;
    fd_weights(o, 7, wc);
    for (int k = 0; k < 7; ++k) w[3][k] = w[4][k + 1] = wc[k];
    for (int i = 0; i < 3; ++i) {
        double wl[8];
        for (int k = 0; k < 8; ++k) o[k] = k - i;
        fd_weights(o, 8, wl);
        for (int k = 0; k < 8; ++k) w[i][k] = w[7 - i][7 - k] = wl[k];   // the right rows mirror the left ones
    }
    for (int r = 0; r < 8; ++r)
        for (int k = 0; k < 8; ++k) W.w[r][k] = A::cst(A::row * w[r][k]);
    return W;
}

template <class A>
FaceC<A> make_face_consts(const helm_ctx* c, int axis) {
    const int ta = axis == 2 ? 1 : 2, tb = axis == 0 ? 1 : 0;
    const double h = c->h[axis], c1 = 2.0 * h * h * h / 6.0, c2 = 2.0 * h * h * h * h * h / 120.0;
    const double iha2 = 1.0 / (c->h[ta] * c->h[ta]), ihb2 = 1.0 / (c->h[tb] * c->h[tb]);
    const double f = A::scale_of(c->k0 * c->k0 + 256.0 * (iha2 + ihb2));   // L's row sums (rows of at most 256)
    FaceC<A> k;
    k.iha2 = A::cst(f / A::row * iha2);
    k.ihb2 = A::cst(f / A::row * ihb2);
    k.c0 = A::cst(2.0 * h);
    k.c1 = A::cst(c1);
    k.mc1 = A::cst(-c1 / f);
    k.c2 = A::cst(c2 / f / f);
    k.k0 = A::cst(c->k0);
    k.kk = A::cst(f * c->k0 * c->k0);
    k.mkk = A::cst(-c->k0 * c->k0);
    return k;
}

Face make_face(const helm_ctx* c, int axis) {
    const int n[3] = {c->nx, c->ny, c->nz};
    const long long st[3] = {1, (long long)(c->nx + 2), (long long)(c->nx + 2) * (c->ny + 2)};
    // tangential axes in array order: x-face (z, y), y-face (z, x), z-face (y, x)
    const int ta = axis == 2 ? 1 : 2, tb = axis == 0 ? 1 : 0;
    Face f;
    f.axis = axis;
    // a face covers the ghost columns of the directions filled before it
    f.la = ta < axis ? n[ta] + 2 : n[ta];
    f.lb = tb < axis ? n[tb] + 2 : n[tb];
    f.sa0 = ta < axis ? 0 : 1;
    f.sb0 = tb < axis ? 0 : 1;
    f.sn = st[axis]; f.sa = st[ta]; f.sb = st[tb];
    f.nb_lo = 1; f.nb_hi = n[axis];
    return f;
}

// The ghost shell of P.  copy: also U into the interior of P (which then holds the whole operand); U = nullptr: the
// interior is zero (the f part of the closure alone); faces = nullptr: no f part.
template <class M>
helm_status fill(helm_ctx* c, const M* U, M* P, const double2* faces, bool copy, cudaStream_t s) {
    if (!U) {
        HELM_CUDA_TRY(cudaMemsetAsync(P, 0, (size_t)(c->nx + 2) * (c->ny + 2) * (c->nz + 2) * sizeof(M), s));
    } else if (copy) {
        ho_copy_kernel<M><<<1024, 256, 0, s>>>(c->nx, c->ny, c->nz, U, P);
        HELM_CUDA_TRY(cudaGetLastError());
    }
    typedef typename ArithOf<M>::T A;
    static const Wts<A> W = make_weights<A>();   // the same for every grid (weights times 1/h^2 per face)
    typename A::St* S = reinterpret_cast<typename A::St*>(c->ho_S);   // 16 bytes a value either way
    const Operand<M> op = {U, P, c->nx, c->ny, c->nz};
    long long foff = 0;
    LaunchChain chain(c, s, 0);   // timed as one launch, if at all
    for (int axis = 0; axis < 3; ++axis) {
        const Face f = make_face(c, axis);
        const int tot = 2 * f.la * f.lb;
        const unsigned blocks = (unsigned)((tot + HO_NT - 1) / HO_NT);
        const FaceC<A> k = make_face_consts<A>(c, axis);
        launch_after(c->follows, ho_lap_kernel<M, A>, blocks, HO_NT, 0, s, f, k, W, op, S);
        chain.first_done();
        HELM_CUDA_TRY(cudaGetLastError());
        launch_after(c->follows, ho_ghost_kernel<M, A>, blocks, HO_NT, 0, s, f, k, W, op, P, S, faces ? faces + foff : nullptr);
        HELM_CUDA_TRY(cudaGetLastError());
        foff += 3LL * tot;
    }
    return HELM_OK;
}

__global__ void sub_kernel(const double2* __restrict__ a, const double2* __restrict__ b, double2* __restrict__ out,
                           size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        out[i] = make_double2(a[i].x - b[i].x, a[i].y - b[i].y);
}

}  // namespace

size_t closure_face_points(const helm_ctx* c) {
    size_t tot = 0;
    for (int axis = 0; axis < 3; ++axis) {
        const Face f = make_face(c, axis);
        tot += 2 * 3 * (size_t)f.la * f.lb;
    }
    return tot;
}

helm_status closure_fill_f32(helm_ctx* c, const float2* U, bool copy, cudaStream_t s) { return fill(c, U, c->ho_P32, nullptr, copy, s); }
helm_status closure_fill_f64(helm_ctx* c, const double2* U, cudaStream_t s) { return fill(c, U, c->ho_P64, nullptr, true, s); }
helm_status closure_fill_df(helm_ctx* c, const float4* U, cudaStream_t s) { return fill(c, U, c->ho_Pdf, nullptr, true, s); }

// F_out = F_in - A(G_f), G_f the ghosts of the closure's f part with a zero interior (FP64)
helm_status closure_rhs(helm_ctx* c, const double2* faces, const double2* Fin, double2* Fout, cudaStream_t s) {
    double2* y = nullptr;
    if (cudaMalloc(&y, c->npts * sizeof(double2)) != cudaSuccess) { cudaGetLastError(); return HELM_ERR_NOMEM; }
    helm_status st = fill<double2>(c, nullptr, c->ho_P64, faces, false, s);
    if (st == HELM_OK) st = launch_stencil_f64_padded(c, c->ho_P64, y, s);
    if (st == HELM_OK) {
        sub_kernel<<<1024, 256, 0, s>>>(Fin, y, Fout, c->npts);
        if (cudaGetLastError() != cudaSuccess) st = HELM_ERR_CUDA;
    }
    cudaStreamSynchronize(s);
    cudaFree(y);
    return st;
}

void closure_release(helm_ctx* c) {
    void* ps[] = {c->ho_P32, c->ho_P64, c->ho_Pdf, c->ho_S};
    for (void* p : ps) if (p) cudaFree(p);
    c->ho_P32 = nullptr; c->ho_P64 = nullptr; c->ho_Pdf = nullptr; c->ho_S = nullptr;
    if (c->ho) stencil_real_release(c);
    c->ho = 0;
}

extern "C" helm_status helm_set_closure(helm_ctx* c, int closure) {
    if (!c || (closure != HELM_CLOSURE_THREE_POINT && closure != HELM_CLOSURE_HIGH_ORDER)) return HELM_ERR_ARG;
    if (closure == HELM_CLOSURE_THREE_POINT) { closure_release(c); return HELM_OK; }
    // the one-sided rows need eight nodes on every face line
    if (!c->colloc || c->nx < 8 || c->ny < 8 || c->nz < 8) return HELM_ERR_UNSUPPORTED;
    if (c->ho) return HELM_OK;
    const size_t np = (size_t)(c->nx + 2) * (c->ny + 2) * (c->nz + 2);
    const int nmax = c->nx > c->ny ? (c->nx > c->nz ? c->nx : c->nz) : (c->ny > c->nz ? c->ny : c->nz);
    const size_t ns = 2 * (size_t)(nmax + 2) * (nmax + 2);
    if (cudaMalloc(&c->ho_P32, np * sizeof(float2)) != cudaSuccess ||
        cudaMalloc(&c->ho_P64, np * sizeof(double2)) != cudaSuccess ||
        cudaMalloc(&c->ho_Pdf, np * sizeof(float4)) != cudaSuccess ||
        cudaMalloc(&c->ho_S, ns * sizeof(double2)) != cudaSuccess) {
        cudaGetLastError();
        closure_release(c);
        return HELM_ERR_NOMEM;
    }
    // ghost planes are rewritten by every fill; zero once so that no word is ever undefined
    HELM_CUDA_TRY(cudaMemset(c->ho_P32, 0, np * sizeof(float2)));
    HELM_CUDA_TRY(cudaMemset(c->ho_P64, 0, np * sizeof(double2)));
    HELM_CUDA_TRY(cudaMemset(c->ho_Pdf, 0, np * sizeof(float4)));
    c->ho = 1;
    // the real fields of a medium without attenuation; without room for them the matvec reads the complex ones
    const helm_status st = stencil_real_prepare(c, nullptr);
    if (st == HELM_OK || st == HELM_ERR_NOMEM) return HELM_OK;
    closure_release(c);
    return st;
}
