// y passes on mixed-radix lengths (ml_mixed.cuh, mixed_split.cu): G lines of one kx
// per CTA of 128 threads, coarse radices; small CTAs, so that several per SM are
// in different phases (load, passes, store) at any time.
#include "ml_mixed.cuh"

#include <algorithm>

namespace boris {

namespace {

template <typename L>
__global__ void __launch_bounds__(128, 4)
    line_y_fwd_kernel(const MLPlane* __restrict__ planes, int ny, int nlines, int Z, int G, const float2* __restrict__ X,
                    float2* __restrict__ Y, const float2* __restrict__ tw, const unsigned short* __restrict__ pos)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* buf = reinterpret_cast<float2*>(smem_raw);
    __shared__ int lo[16], hi[16];
    const int l0 = blockIdx.x * G, n = min(G, nlines - l0);
    if ((int)threadIdx.x < n) {
        const MLPlane* q = planes ? planes + (l0 + threadIdx.x) % Z : nullptr;
        lo[threadIdx.x] = q ? q->oy : 0;
        hi[threadIdx.x] = q ? q->oy + q->ny : ny;
    }
    __syncthreads();
    const float2* src = X + ((size_t)blockIdx.y * nlines + l0) * ny;
    line_fwd1<L>(n, buf, tw, [&](int l, int y, bool) {
        return y >= lo[l] && y < hi[l] ? src[l * ny + y] : float2{0.f, 0.f};
    });
    line_fwd_rest<L>(n, buf, tw);
    constexpr int P = 2 * L::H;
    float2* dst = Y + ((size_t)blockIdx.y * nlines + l0) * P;
    for (int i = threadIdx.x; i < n * P; i += blockDim.x) {
        const int l = i / P, k = i % P;
        dst[i] = buf[l * L::template LS<float2> + pos[k]];
    }
}

template <typename L>
__global__ void __launch_bounds__(128, 4)
    line_y_inv_kernel(const MLPlane* __restrict__ planes, int ny, int nlines, int Z, int G, const float2* __restrict__ Y,
                    float2* __restrict__ X, const float2* __restrict__ tw, const unsigned short* __restrict__ pos)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* buf = reinterpret_cast<float2*>(smem_raw);
    __shared__ int lo[16], hi[16];
    const int l0 = blockIdx.x * G, n = min(G, nlines - l0);
    if ((int)threadIdx.x < n) {
        const MLPlane* q = planes ? planes + (l0 + threadIdx.x) % Z : nullptr;
        lo[threadIdx.x] = q ? q->oy : 0;
        hi[threadIdx.x] = q ? q->oy + q->ny : ny;
    }
    constexpr int P = 2 * L::H;
    const float2* src = Y + ((size_t)blockIdx.y * nlines + l0) * P;
    staged_loop<128, float2>(n * P, [&](int i) { return src[i]; },
                             [&](int i, float2 v) { buf[i / P * L::template LS<float2> + pos[i % P]] = v; });
    __syncthreads();
    line_inv_rest<L>(n, buf, tw);
    float2* dst = X + ((size_t)blockIdx.y * nlines + l0) * ny;
    line_inv1<L>(n, buf, tw, [&](int l, int y, float2 v) {
        if (y >= lo[l] && y < hi[l]) dst[l * ny + y] = v;
    });
}

int y_lines(const MixedPlan& m, int nlines)
{
    int g = 4;
    while (g > 1 && (size_t)g * m.y.LS * sizeof(float2) > 50 * 1024) g--;
    return std::min(g, nlines);
}

template <typename F>
cudaError_t coarse_length(int id, F f)
{
    switch (id) {
#define X(i, r1, r2, r3, ...) \
    case i:                   \
        if constexpr (i >= N_FINE || !has_coarse(r1 * r2 * r3)) return f(Len<r1, r2, r3, __VA_ARGS__>{}); \
        break;
        BORIS_LENGTHS(X)
#undef X
    }
    return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t line_y_prepare(const MixedPlan& m)
{
    return coarse_length(m.y.id, [&](auto L) {
        constexpr int most = 226 * 1024;  // beside the row windows
        cudaError_t r = cudaFuncSetAttribute(line_y_fwd_kernel<decltype(L)>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        if (r != cudaSuccess) return r;
        return cudaFuncSetAttribute(line_y_inv_kernel<decltype(L)>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    });
}

cudaError_t launch_line_y(const MixedPlan& m, const MLPlane* planes, int nlines, int Z, float2* X, float2* Y, cudaStream_t st,
                          bool forward)
{
    const int G = y_lines(m, nlines);
    const dim3 grid((nlines + G - 1) / G, m.x.H + 1);
    const size_t smem = (size_t)G * m.y.LS * sizeof(float2);
    return coarse_length(m.y.id, [&](auto L) {
        if (forward)
            line_y_fwd_kernel<decltype(L)><<<grid, 128, smem, st>>>(planes, m.y.n, nlines, Z, G, X, Y, (const float2*)m.twy, m.posy);
        else
            line_y_inv_kernel<decltype(L)><<<grid, 128, smem, st>>>(planes, m.y.n, nlines, Z, G, Y, X, (const float2*)m.twy, m.posy);
        return cudaGetLastError();
    });
}

}  // namespace boris
