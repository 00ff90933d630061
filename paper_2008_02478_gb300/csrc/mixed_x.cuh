// Mixed-radix x passes (kernels; instantiated per precision in mixed_x_f32.cu and
// mixed_x_f64.cu).
//
// x_fwd: a CTA transforms 2 HL rows of one (component, plane): two rows are the
// real and imaginary part of one complex line (HL = 2^lhl lines in shared
// memory), whose spectrum untangles as A_k = (Z_k + conj Z_-k)/2,
// B_k = (Z_k - conj Z_-k)/(2i); it writes X[kx][c][z][y], 2 HL consecutive y per
// kx.  x_inv packs Z_k = A_k + i B_k from those columns and runs the passes
// backwards.  Latency-bound on small meshes (256 x 64 x 1: 3.6 us a pass against
// 7.1 and 8.2 for the two-rows-per-warp kernels of fft512.cu, which have 6 CTAs
// there), bound by the shared-memory pipe on large ones (256 x 256 x 8: 7.9 us
// against 11.1; 1500 x 700 x 4, 3072 instead of 4096 points: 69 and 85 against
// 87 and 106).
#pragma once
#include "mixed_demag.cuh"

namespace boris {

template <typename T>
struct XArgs {
    using C = typename Cx<T>::t;
    int nx, ny, nz, lhl;
    const T* M;       // x_fwd: field, and its scale (map or uniform)
    const T* ms_map;
    T ms;
    T* Hf;            // x_inv: field
    C* X;
    const C* tw;
    const unsigned short* pos;
};

// CTAs per SM the register budget is fitted to
template <typename T, typename L>
constexpr int x_ctas()
{
    return L::R1 > 8 ? (sizeof(T) == 4 ? 2 : 1) : sizeof(T) == 4 ? 4 : 2;
}

template <typename T, typename L>
__global__ void __launch_bounds__(256, x_ctas<T, L>()) x_fwd_kernel(const __grid_constant__ XArgs<T> g)
{
    using C = typename Cx<T>::t;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* buf = reinterpret_cast<C*>(smem_raw);  // [HL][LS]
    const int HL = 1 << g.lhl;
    const int y0 = blockIdx.x << (g.lhl + 1), z = blockIdx.y, c = blockIdx.z;
    const int nx = g.nx, ny = g.ny, nz = g.nz;
    constexpr int H = L::H, LS = L::template LS<C>;
    const size_t row0 = ((size_t)z * ny + y0) * nx;
    const T* Mb = g.M + (size_t)c * nx * ny * nz + row0;
    const int rows = ny - y0;
    if (g.ms_map) {
        const T* mb = g.ms_map + row0;
        line_fwd1<L>(HL, buf, g.tw, [&](int t, int n, bool) {
            const int i = t * nx + n, j = i + HL * nx;
            const bool a = n < nx && t < rows, b = n < nx && t + HL < rows;
            const T va = a ? Mb[i] : T(0), vb = b ? Mb[j] : T(0), sa = a ? mb[i] : T(0), sb = b ? mb[j] : T(0);
            return C{va * sa, vb * sb};
        });
    } else {
        line_fwd1<L>(HL, buf, g.tw, [&](int t, int n, bool) {
            const int i = t * nx + n, j = i + HL * nx;
            const T va = n < nx && t < rows ? Mb[i] : T(0), vb = n < nx && t + HL < rows ? Mb[j] : T(0);
            return C{va * g.ms, vb * g.ms};
        });
    }
    line_fwd_rest<L>(HL, buf, g.tw);
    const size_t plane = (size_t)3 * nz * ny;
    C* Xb = g.X + ((size_t)c * nz + z) * ny + y0;
    for (int i = threadIdx.x; i < (H + 1) << g.lhl; i += blockDim.x) {
        const int t = i & (HL - 1), k = i >> g.lhl;
        const C* line = buf + t * LS;
        const C zk = line[g.pos[k]], zm = line[g.pos[k == 0 ? 0 : 2 * H - k]];
        C* d = Xb + (size_t)k * plane + t;
        if (t < rows) d[0] = C{T(0.5) * (zk.x + zm.x), T(0.5) * (zk.y - zm.y)};
        if (t + HL < rows) d[HL] = C{T(0.5) * (zk.y + zm.y), T(-0.5) * (zk.x - zm.x)};
    }
}

template <typename T, typename L>
__global__ void __launch_bounds__(256, x_ctas<T, L>()) x_inv_kernel(const __grid_constant__ XArgs<T> g)
{
    using C = typename Cx<T>::t;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* buf = reinterpret_cast<C*>(smem_raw);
    const int HL = 1 << g.lhl;
    const int y0 = blockIdx.x << (g.lhl + 1), z = blockIdx.y, c = blockIdx.z;
    const int nx = g.nx, ny = g.ny, nz = g.nz;
    constexpr int H = L::H, LS = L::template LS<C>;
    const int rows = ny - y0;
    const size_t plane = (size_t)3 * nz * ny;
    const C* Xb = g.X + ((size_t)c * nz + z) * ny + y0;
    const int total = (H + 1) << g.lhl;
    constexpr int U = 4;  // loads in flight per thread
    for (int b = threadIdx.x; b < total; b += blockDim.x * U) {
        C va[U], vb[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int i = b + u * (int)blockDim.x;
            const int t = i & (HL - 1), k = i >> g.lhl;
            const C* s = Xb + (size_t)k * plane + t;
            va[u] = i < total && t < rows ? s[0] : C{T(0), T(0)};
            vb[u] = i < total && t + HL < rows ? s[HL] : C{T(0), T(0)};
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int i = b + u * (int)blockDim.x;
            if (i >= total) break;
            const int t = i & (HL - 1), k = i >> g.lhl;
            C* line = buf + t * LS;
            if (k == 0 || k == H) {
                line[g.pos[k]] = C{va[u].x, vb[u].x};  // DC and Nyquist bins of a real row are real
            } else {
                line[g.pos[k]] = C{va[u].x - vb[u].y, va[u].y + vb[u].x};
                line[g.pos[2 * H - k]] = C{va[u].x + vb[u].y, vb[u].x - va[u].y};
            }
        }
    }
    __syncthreads();
    line_inv_rest<L>(HL, buf, g.tw);
    T* Hb = g.Hf + (size_t)c * nx * ny * nz + ((size_t)z * ny + y0) * nx;
    line_inv1<L>(HL, buf, g.tw, [&](int t, int n, C v) {
        if (n < nx) {
            if (t < rows) Hb[t * nx + n] = v.x;
            if (t + HL < rows) Hb[(t + HL) * nx + n] = v.y;
        }
    });
}

template <typename T>
struct XLaunch {
    XArgs<T> a;
    dim3 grid;
    int threads;
    size_t smem;
};
template <typename T>
XLaunch<T> x_launch(const MixedPlan& m)
{
    using C = typename Cx<T>::t;
    const int hl = x_lines(m, sizeof(C));
    XLaunch<T> l = {};
    l.a.nx = m.x.n;
    l.a.ny = m.y.n;
    l.a.nz = m.nz;
    l.a.lhl = ilog2(hl);
    l.a.tw = (const C*)m.twx;
    l.a.pos = m.posx;
    l.grid = dim3((m.y.n + 2 * hl - 1) / (2 * hl), m.nz, 3);
    const int items = hl * m.x.r2 * m.x.r3;
    l.threads = items >= 256 ? 256 : items <= 64 ? 64 : (items + 31) / 32 * 32;
    l.smem = (size_t)hl * m.x.LS * sizeof(C);
    return l;
}

template <typename T>
cudaError_t x_set_attr(const MixedPlan& m)
{
    cudaError_t e = cudaErrorInvalidValue;
    switch (m.x.id) {
#define X(i, r1, r2, r3, ...)                                                                                              \
    case i:                                                                                                           \
        e = cudaFuncSetAttribute(x_fwd_kernel<T, Len<r1, r2, r3, __VA_ARGS__>>, cudaFuncAttributeMaxDynamicSharedMemorySize,       \
                                 227 * 1024);                                                                         \
        if (e == cudaSuccess)                                                                                         \
            e = cudaFuncSetAttribute(x_inv_kernel<T, Len<r1, r2, r3, __VA_ARGS__>>, cudaFuncAttributeMaxDynamicSharedMemorySize,   \
                                     227 * 1024);                                                                     \
        break;
        BORIS_LENGTHS_FINE(X)
#undef X
    }
    return e;
}

template <typename T>
cudaError_t launch_mixed_x_fwd(const MixedPlan& m, const T* M, const T* ms_map, T ms, typename Cx<T>::t* X_, cudaStream_t st)
{
    XLaunch<T> l = x_launch<T>(m);
    l.a.M = M;
    l.a.ms_map = ms_map;
    l.a.ms = ms;
    l.a.X = X_;
    switch (m.x.id) {
#define X(i, r1, r2, r3, ...) \
    case i: x_fwd_kernel<T, Len<r1, r2, r3, __VA_ARGS__>><<<l.grid, l.threads, l.smem, st>>>(l.a); break;
        BORIS_LENGTHS_FINE(X)
#undef X
    }
    return cudaGetLastError();
}
template <typename T>
cudaError_t launch_mixed_x_inv(const MixedPlan& m, const typename Cx<T>::t* X_, T* H, cudaStream_t st)
{
    XLaunch<T> l = x_launch<T>(m);
    l.a.X = const_cast<typename Cx<T>::t*>(X_);
    l.a.Hf = H;
    switch (m.x.id) {
#define X(i, r1, r2, r3, ...) \
    case i: x_inv_kernel<T, Len<r1, r2, r3, __VA_ARGS__>><<<l.grid, l.threads, l.smem, st>>>(l.a); break;
        BORIS_LENGTHS_FINE(X)
#undef X
    }
    return cudaGetLastError();
}

#define MIXED_X_INST(T)                                                                                             \
    template cudaError_t x_set_attr<T>(const MixedPlan&);                                                           \
    template cudaError_t launch_mixed_x_fwd<T>(const MixedPlan&, const T*, const T*, T, Cx<T>::t*, cudaStream_t);   \
    template cudaError_t launch_mixed_x_inv<T>(const MixedPlan&, const Cx<T>::t*, T*, cudaStream_t);

}  // namespace boris
