// Multi-mesh x and y passes on mixed-radix lengths (ml_mixed.cuh).
//
// Before, the layers were copied into a zero frame [3][Z][NY][NX], the whole
// frame was transformed and the field copied out again: on the six-layer 512 x
// 512 stack (34 planes, 46 % of the frame's rows exist) the copies took 151 + 54
// us of a 1690 us evaluation and the x passes 134.  The x passes here read the
// layers and transform their rows only, and the y passes load and store only
// rows that exist.  Those of this file take 72 + 60 (x) and 132 + 200 us (y) on
// that frame; its 1024-point axes go to the warp-held transforms of
// demag_fast.cu with the same windows, 41 + 37 and 103 + 123.
#include "ml_mixed.cuh"

#include <algorithm>
#include <type_traits>

namespace boris {

namespace {

template <typename L>
__global__ void __launch_bounds__(256, 4) ml_x_fwd_kernel(const MLPlane* __restrict__ planes, int NY, int Z, int lhl,
                                                          const float* __restrict__ M, const float* __restrict__ ms_map,
                                                          float ms, float2* __restrict__ X, const float2* __restrict__ tw,
                                                          const unsigned short* __restrict__ pos)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* buf = reinterpret_cast<float2*>(smem_raw);  // [HL][LS]
    const int HL = 1 << lhl, z = blockIdx.y, c = blockIdx.z;
    const MLPlane q = planes[z];
    const int r0 = blockIdx.x << (lhl + 1), rows = q.ny - r0;
    if (rows <= 0) return;
    constexpr int H = L::H, LS = L::template LS<float2>;
    const int nx = q.nx, ox = q.ox;
    const float* Mb = M + q.off + c * q.comp + (size_t)r0 * nx;
    const float* mb = ms_map + (ms_map ? q.moff + (size_t)r0 * nx : 0);
    auto load = [&](int t, int n, auto map) {
        const int x = n - ox, i = t * nx + x, j = i + HL * nx;
        const bool in = x >= 0 && x < nx, a = in && t < rows, b = in && t + HL < rows;
        const float va = a ? Mb[i] : 0.f, vb = b ? Mb[j] : 0.f;
        if constexpr (decltype(map)::value) {
            const float sa = a ? mb[i] : 0.f, sb = b ? mb[j] : 0.f;
            return float2{va * sa, vb * sb};
        } else {
            return float2{va * ms, vb * ms};
        }
    };
    if (ms_map) line_fwd1<L>(HL, buf, tw, [&](int t, int n, bool) { return load(t, n, std::true_type{}); });
    else line_fwd1<L>(HL, buf, tw, [&](int t, int n, bool) { return load(t, n, std::false_type{}); });
    line_fwd_rest<L>(HL, buf, tw);
    const size_t plane = (size_t)3 * Z * NY;
    float2* Xb = X + ((size_t)c * Z + z) * NY + q.oy + r0;
    for (int i = threadIdx.x; i < (H + 1) << lhl; i += blockDim.x) {
        const int t = i & (HL - 1), k = i >> lhl;
        const float2* line = buf + t * LS;
        const float2 zk = line[pos[k]], zm = line[pos[k == 0 ? 0 : 2 * H - k]];
        float2* d = Xb + (size_t)k * plane + t;
        if (t < rows) d[0] = float2{0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y)};
        if (t + HL < rows) d[HL] = float2{0.5f * (zk.y + zm.y), -0.5f * (zk.x - zm.x)};
    }
}

template <typename L>
__global__ void __launch_bounds__(256, 4) ml_x_inv_kernel(const MLPlane* __restrict__ planes, int NY, int Z, int lhl,
                                                          const float2* __restrict__ X, float* __restrict__ Hf,
                                                          const float2* __restrict__ tw,
                                                          const unsigned short* __restrict__ pos)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* buf = reinterpret_cast<float2*>(smem_raw);
    const int HL = 1 << lhl, z = blockIdx.y, c = blockIdx.z;
    const MLPlane q = planes[z];
    const int r0 = blockIdx.x << (lhl + 1), rows = q.ny - r0;
    if (rows <= 0) return;
    constexpr int H = L::H, LS = L::template LS<float2>;
    const int nx = q.nx, ox = q.ox;
    const size_t plane = (size_t)3 * Z * NY;
    const float2* Xb = X + ((size_t)c * Z + z) * NY + q.oy + r0;
    const int total = (H + 1) << lhl;
    constexpr int U = 4;  // loads in flight per thread
    for (int b = threadIdx.x; b < total; b += blockDim.x * U) {
        float2 va[U], vb[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int i = b + u * (int)blockDim.x;
            const int t = i & (HL - 1), k = i >> lhl;
            const float2* s = Xb + (size_t)k * plane + t;
            va[u] = i < total && t < rows ? s[0] : float2{0.f, 0.f};
            vb[u] = i < total && t + HL < rows ? s[HL] : float2{0.f, 0.f};
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int i = b + u * (int)blockDim.x;
            if (i >= total) break;
            const int t = i & (HL - 1), k = i >> lhl;
            float2* line = buf + t * LS;
            if (k == 0 || k == H) {
                line[pos[k]] = float2{va[u].x, vb[u].x};  // DC and Nyquist bins of a real row are real
            } else {
                line[pos[k]] = float2{va[u].x - vb[u].y, va[u].y + vb[u].x};
                line[pos[2 * H - k]] = float2{va[u].x + vb[u].y, vb[u].x - va[u].y};
            }
        }
    }
    __syncthreads();
    line_inv_rest<L>(HL, buf, tw);
    float* Hb = Hf + q.off + c * q.comp + (size_t)r0 * nx;
    line_inv1<L>(HL, buf, tw, [&](int t, int n, float2 v) {
        const int x = n - ox;
        if (x >= 0 && x < nx) {
            if (t < rows) Hb[t * nx + x] = v.x;
            if (t + HL < rows) Hb[(t + HL) * nx + x] = v.y;
        }
    });
}

}  // namespace

bool ml_mixed_shape(int NX, int NY, int Z, int max_smem, MLMixed* p)
{
    if (NX < 2 || NY < 2) return false;
    p->Z = Z;
    p->m.nz = Z;
    if (!make_line_fft(NX, sizeof(float2), false, &p->m.x) || !make_line_fft(NY, sizeof(float2), true, &p->m.y)) return false;
    return (size_t)p->m.y.LS * sizeof(float2) <= (size_t)max_smem && (size_t)2 * p->m.x.LS * sizeof(float2) <= (size_t)max_smem;
}

// f(Len) for an axis plan
template <typename F>
static cudaError_t fine_length(int id, F f)
{
    switch (id) {
#define X(i, r1, r2, r3, ...) \
    case i: return f(Len<r1, r2, r3, __VA_ARGS__>{});
        BORIS_LENGTHS_FINE(X)
#undef X
    }
    return cudaErrorInvalidValue;
}
cudaError_t ml_mixed_prepare(const MLMixed& p)
{
    constexpr int most = 227 * 1024;
    cudaError_t e = fine_length(p.m.x.id, [&](auto L) {
        cudaError_t r = cudaFuncSetAttribute(ml_x_fwd_kernel<decltype(L)>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        if (r != cudaSuccess) return r;
        return cudaFuncSetAttribute(ml_x_inv_kernel<decltype(L)>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    });
    return e == cudaSuccess ? line_y_prepare(p.m) : e;
}

cudaError_t launch_ml_x_fwd(const MLMixed& p, const float* M, const float* ms_map, float ms, float2* X, cudaStream_t st)
{
    int hl = 8;
    while (hl > 2 && (size_t)hl * p.m.x.LS * sizeof(float2) > 100 * 1024) hl /= 2;
    const dim3 grid((p.rows + 2 * hl - 1) / (2 * hl), p.Z, 3);
    return fine_length(p.m.x.id, [&](auto L) {
        ml_x_fwd_kernel<decltype(L)><<<grid, 256, (size_t)hl * p.m.x.LS * sizeof(float2), st>>>(
            p.planes, p.m.y.n, p.Z, ilog2(hl), M, ms_map, ms, X, (const float2*)p.m.twx, p.m.posx);
        return cudaGetLastError();
    });
}

cudaError_t launch_ml_x_inv(const MLMixed& p, const float2* X, float* H, cudaStream_t st)
{
    int hl = 8;
    while (hl > 2 && (size_t)hl * p.m.x.LS * sizeof(float2) > 100 * 1024) hl /= 2;
    const dim3 grid((p.rows + 2 * hl - 1) / (2 * hl), p.Z, 3);
    return fine_length(p.m.x.id, [&](auto L) {
        ml_x_inv_kernel<decltype(L)><<<grid, 256, (size_t)hl * p.m.x.LS * sizeof(float2), st>>>(
            p.planes, p.m.y.n, p.Z, ilog2(hl), X, H, (const float2*)p.m.twx, p.m.posx);
        return cudaGetLastError();
    });
}

}  // namespace boris
