// The y-z part of the convolution on mixed-radix lengths as three passes over
// the padded spectrum: y transforms X[kx][c][z][y] -> Y[kx][c][z][ky] (those of
// ml_mixed_y.cu), the z stage in place on Y, y inverses.  For meshes whose plane
// does not fit one CTA's shared memory, or whose planes leave SMs idle, where
// the power-of-two lengths pad most (mixed_pays): the z stage, the transforms of
// plane_conv.cuh, reaches a third to a half of the copy rate (loads' latency at
// 8 to 20 warps per SM), the power-of-two one two thirds.  Evaluations, before ->
// now: 160 x 640 x 12 238 -> 131 us, 86 x 705 x 8 87 -> 53, 39 x 143 x 23 56 -> 32,
// 283 x 269 x 24 412 -> 287, 48 x 512 x 32 140 -> 86, 545 x 836 x 6 525 -> 436 (power-of-two
// passes), 160 x 160 x 20 69 -> 62 (planes).
#include "bulk_async.cuh"
#include "ml_mixed.cuh"
#include "plane_conv.cuh"

namespace boris {

namespace {

// Four warps per CTA, the items of all kx side by side (545 x 836 x 6: 126 us with
// those of one kx side by side, now 107).  From HZ 12 on TK bins ky' of one kx,
// their mirrors and their kernel rows go through shared memory in rows of 256
// consecutive bytes, columns as [line][TK | 8 | TK] (the gap keeps a bin and its
// mirror in different banks): read where they are used, the kernel rows were what
// the warps waited for (direct against staged: 160 x 640 x 12 59 and 42 us, 160 x 160
// x 20 25 and 23, 283 x 269 x 24 153 and 122, 55 x 767 x 26 170 and 80).  To HZ 8 each
// warp reads and writes one item's columns in 64-byte pieces (256 x 256 x 8 12.2
// and 15.5, 700 x 700 x 5 89 and 104).
constexpr int TK = 32, ZLS = 2 * TK + 8;
constexpr int KP = 44;  // pitch of a staged kernel row: the rows of four residues start four pairs apart mod 16
constexpr bool z_staged(int HZ) { return HZ >= 12; }

template <int HZ, int RES>
__global__ void __launch_bounds__(128, HZ <= 12 ? 5 : HZ == 32 ? 2 : 3)
    z_conv_kernel(int H, int nz, int kyp, int nkz, float2* __restrict__ Y, const float2* __restrict__ K,
                  const float2* __restrict__ twz)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int KB = 16 / RES;
    const int P = 2 * H, kx = blockIdx.x, k0 = blockIdx.y * TK;
    float2* base = Y + (size_t)kx * 3 * nz * P;
    const float2* Kx = K + (size_t)kx * nkz * 3 * kyp;
    const int warp = threadIdx.x >> 5, items = H / KB + 1;
    if constexpr (z_staged(HZ)) {
        float2* buf = reinterpret_cast<float2*>(smem_raw);
        const int half = (threadIdx.x >> 5) & 1, col = threadIdx.x & 31, k = k0 + col;
        const bool ok = half ? k > 0 && k < H : k <= H;
        const int ky = ok ? (half ? P - k : k) : 0, at = col + half * (TK + 8);
        for (int l = threadIdx.x >> 6; l < 3 * nz; l += 2)
            if (ok)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(buf + l * ZLS + at)),
                             "l"(base + (size_t)l * P + ky)
                             : "memory");
        float2* kbuf = buf + 3 * nz * ZLS;  // [kz'][pair][KP]
        for (int i = threadIdx.x; i < nkz * 3 * (TK / 2); i += 128) {
            const int r = i / (TK / 2), pc = 2 * (i % (TK / 2));
            if (k0 + pc < kyp) cp_async16(kbuf + r * KP + pc, Kx + (size_t)r * kyp + k0 + pc);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        z_columns<float, HZ, RES, true>(H, ZLS, nz * ZLS, nz, KP, kbuf - k0, twz, k0 / KB + warp, min(k0 / KB + TK / KB, items), 4,
                                  [&](int q) { return buf + (q <= H ? q - k0 : P - q - k0 + TK + 8); });
        __syncthreads();
        if (ok)
            for (int l = threadIdx.x >> 6; l < 3 * nz; l += 2) base[(size_t)l * P + ky] = buf[l * ZLS + at];
    } else {
        // one item per warp
        z_columns<float, HZ, RES>(H, P, nz * P, nz, kyp, Kx, twz, blockIdx.y * 4 + warp, items, items, [&](int q) { return base + q; });
    }
}

template <int HZ>
constexpr int z_res = HZ <= 8 ? 2 : 4;

// Shared memory of a CTA for nz planes and nkz kernel rows, 90 KB at most.
constexpr size_t z_smem(int HZ, int nz, int nkz)
{
    return z_staged(HZ) ? ((size_t)3 * nz * ZLS + (size_t)3 * nkz * KP) * sizeof(float2) : 0;
}

// The shared-memory limit belongs to the kernel, which plans of every nz with this
// HZ share: it is set to what the largest nz takes, so no plan lowers it for another.
template <int HZ>
cudaError_t z_prepare()
{
    return cudaFuncSetAttribute(z_conv_kernel<HZ, z_res<HZ>>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)z_smem(HZ, HZ, HZ + 1));
}

template <int HZ>
cudaError_t z_launch(const MixedPlan& m, float2* Y, const float2* K, cudaStream_t st)
{
    constexpr int RES = z_res<HZ>;
    const int tiles = z_staged(HZ) ? m.y.H / TK + 1 : (m.y.H * RES / 16 + 4) / 4;
    z_conv_kernel<HZ, RES><<<dim3(m.x.H + 1, tiles), 128, z_smem(HZ, m.nz, m.nkz), st>>>(m.y.H, m.nz, m.kyp, m.nkz, Y, K,
                                                                                        (const float2*)m.twz);
    return cudaGetLastError();
}

}  // namespace

#define Z_SIZES(Z) Z(2) Z(4) Z(6) Z(8) Z(12) Z(16) Z(20) Z(24) Z(32)

cudaError_t mixed_z_prepare(const MixedPlan& m)
{
    switch (m.HZ) {
#define Z(h) \
    case h: return z_prepare<h>();
        Z_SIZES(Z)
#undef Z
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_mixed_z(const MixedPlan& m, float2* Y, const float2* K, cudaStream_t st)
{
    switch (m.HZ) {
#define Z(h) \
    case h: return z_launch<h>(m, Y, K, st);
        Z_SIZES(Z)
#undef Z
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_mixed_y(const MixedPlan& m, const Geometry& g, float2* X, float2* Y, const float2* tw, cudaStream_t st,
                           bool forward)
{
    // 1024 points: the warp-held transforms (one trip through shared memory)
    if (m.y.H == 512) return launch_ml_y_1024(g, nullptr, X, Y, tw, st, forward);
    return launch_line_y(m, nullptr, 3 * m.nz, m.nz, X, Y, st, forward);
}

}  // namespace boris
