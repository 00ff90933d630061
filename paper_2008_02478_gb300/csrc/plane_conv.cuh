// The y-z part of the convolution for one kx plane per CTA, entirely in shared
// memory: y transforms of all 3 nz lines, the z transforms, the 3 x 3 kernel
// multiply and the inverses (the pipelined convolution of Section 7 over both
// axes).  X[kx][c][z][y] is read once and written once in place, the kernel
// octant is read once: the padded spectrum never leaves the SM.
//
// z stage: a column is the 3 nz values of one ky.  The padded z transform of
// length 2 HZ splits by residue like the y lines do; RES lanes of a warp share
// a column, each holding the residue kz = r mod RES of all three components, so
// the 3 x 3 multiply needs no exchange:
//   RES = 2 (HZ <= 8): u[n] = x[n] w^(r n), DFT of HZ points;
//   RES = 4 (HZ >= 12): u[m] = x[m] w^(r m) + x[m + Q] w^(r (m + Q)), DFT of Q = HZ/2 points.
// The inverse sums the residues' contributions by shuffles that halve what a
// lane keeps (RES = 4: lanes r < 2 keep the rows below Q, then even lanes the
// lower half of those).  Which half a lane keeps must not cost selects: the
// twiddle tables are per lane (a keep row and a send row), and an odd lane
// runs its inverse DFT with every second input negated (folded into the
// kernel's signs), which rotates its outputs by half their count, so that on
// every lane registers 0.. are kept and the upper half is sent.  Only the
// lanes of one warp touch a column, so it is written back in place.
// A half-warp takes bins ky' and the other half py - ky', so both columns of
// a kernel row read it in one instruction.
//
// Bound by the shared-memory pipe (L1 data wavefronts 60-70 % of peak; FMA
// pipe 27-33 %): hence two passes of large radices where registers allow, and
// residues that share a column as few ways as they can.  Measured, y-z part of
// one evaluation, split schedule on power-of-two lengths -> this kernel:
// 512 x 512 x 1 19.2 -> 9.5 us, 256 x 256 x 8 33.4 -> 23.6, 201 x 147 x 5 27.3 -> 13.3,
// 160 x 160 x 20 86 -> 53, 1500 x 700 x 4 522 -> 229 (K and X alone: 62 us at the
// copy rate), FP64 128 x 128 x 16 564 -> 487 us (FP64 units).
#pragma once
#include "mixed_demag.cuh"

namespace boris {

template <typename T>
struct PlaneArgs {
    using C = typename Cx<T>::t;
    int len, ny, nz, HZ, H, LS, kyp;
    C* X;
    const C* K;
    const C* tw;
    const C* twz;
    const unsigned short* pos;
};

__device__ __forceinline__ float2 shfl_x(float2 v, int m)
{
    return make_float2(__shfl_xor_sync(0xffffffffu, v.x, m), __shfl_xor_sync(0xffffffffu, v.y, m));
}
__device__ __forceinline__ double2 shfl_x(double2 v, int m)
{
    return make_double2(__shfl_xor_sync(0xffffffffu, v.x, m), __shfl_xor_sync(0xffffffffu, v.y, m));
}

// (a, b, c) <- K (a, b, c) for kernel pairs (xx, yy) (zz, xy) (xz, yz); s scales all
// entries, sxy, sxz, syz the off-diagonal ones on top
template <typename T, typename C>
__device__ __forceinline__ void kernel_mult(const C d01, const C d23, const C d45, T s, T sxy, T sxz, T syz, C& a, C& b,
                                            C& c)
{
    const T xx = s * d01.x, yy = s * d01.y, zz = s * d23.x, xy = sxy * d23.y, xz = sxz * d45.x, yz = syz * d45.y;
    const C hx{xx * a.x + xy * b.x + xz * c.x, xx * a.y + xy * b.y + xz * c.y};
    const C hy{xy * a.x + yy * b.x + yz * c.x, xy * a.y + yy * b.y + yz * c.y};
    const C hz{xz * a.x + yz * b.x + zz * c.x, xz * a.y + yz * b.y + zz * c.y};
    a = hx;
    b = hy;
    c = hz;
}

// The y passes and the z stage are separate functions (not inlined: one copy
// per length and one per z size instead of one per pair of them).
template <typename T, typename L>
__device__ __noinline__ void y_forward(const typename Cx<T>::t* __restrict__ plane, int lines, int ny,
                                       const typename Cx<T>::t* __restrict__ tw)
{
    using C = typename Cx<T>::t;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* buf = reinterpret_cast<C*>(smem_raw);
    line_fwd1<L>(lines, buf, tw, [&](int line, int n, bool) { return n < ny ? plane[line * ny + n] : C{T(0), T(0)}; });
    line_fwd_rest<L>(lines, buf, tw);
}

template <typename T, typename L>
__device__ __noinline__ void y_inverse(typename Cx<T>::t* __restrict__ plane, int lines, int ny,
                                       const typename Cx<T>::t* __restrict__ tw)
{
    using C = typename Cx<T>::t;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* buf = reinterpret_cast<C*>(smem_raw);
    line_inv_rest<L>(lines, buf, tw);
    line_inv1<L>(lines, buf, tw, [&](int line, int n, C v) {
        if (n < ny) plane[line * ny + n] = v;
    });
}

// The z transforms, kernel multiply and inverses of the columns ky' = KB w .. of
// items w = w0, w0 + wstep, ... < wend: column(ky) is row 0 of component 0, rows LS and
// components cs apart.  KSH: the kernel rows (pitch kyp) are in shared memory.
template <typename T, int HZ, int RES, bool KSH = false, typename Col>
__device__ __forceinline__ void z_columns(int H, int LS, int cs, int nz, int kyp, const typename Cx<T>::t* __restrict__ Kx,
                                          const typename Cx<T>::t* __restrict__ twz, int w0, int wend, int wstep, Col column)
{
    using C = typename Cx<T>::t;
    constexpr int Q = RES == 2 ? HZ : HZ / 2;  // points of a lane's DFT
    constexpr int HQ = Q / 2;
    constexpr int KB = 16 / RES;  // ky' per warp item
    static_assert(Q % 2 == 0, "the halving exchange needs an even number of points");
    const int lane = threadIdx.x & 31;
    const int res = lane & (RES - 1), kl = (lane & 15) / RES;
    const bool mirror = lane & 16, odd = lane & 1, up = RES == 4 && (lane & 2);
    const T sy = mirror ? T(-1) : T(1), so = odd ? T(-1) : T(1), syo = sy * so;
    const C* tz = twz + res * 4 * Q;  // rows: in (x[m]), in (x[m + Q]), keep, send
    const int krow = 3 * kyp;
    for (int w = w0; w < wend; w += wstep) {  // (the same for all lanes of a warp)
        const int k = w * KB + kl;
        const bool ok = k <= H && !(mirror && (k == 0 || k == H));
        const int kc = k <= H ? k : H;  // in range for the loads of idle lanes
        C* col = column(mirror ? (kc == 0 ? 0 : 2 * H - kc) : kc);
        C u[3][Q];
#pragma unroll
        for (int m = 0; m < Q; m++) {
            const C wa = __ldg(tz + m);
#pragma unroll
            for (int c = 0; c < 3; c++)
                u[c][m] = m < nz ? c_mul(col[c * cs + m * LS], wa) : C{T(0), T(0)};
            if (RES == 4) {
                const C wb = __ldg(tz + Q + m);
                if (m + Q < nz) {
#pragma unroll
                    for (int c = 0; c < 3; c++) {
                        const C x = col[c * cs + (m + Q) * LS];
                        u[c][m].x += x.x * wb.x - x.y * wb.y;
                        u[c][m].y += x.x * wb.y + x.y * wb.x;
                    }
                }
            }
        }
#pragma unroll
        for (int c = 0; c < 3; c++) dft<Q, -1>(u[c]);
        // kz = RES j + r; rows past kz = HZ are the mirror image kz' = 2 HZ - kz
        // (odd entries negated; at kz = HZ they are zero, so its sign does not matter)
        const C* Ku = Kx + kc + res * krow;
        const C* Kd = Kx + kc + (2 * HZ - res) * krow;
#pragma unroll
        for (int j = 0; j < Q; j++) {
            const bool fz = j >= Q / 2;
            const C* kp = fz ? Kd - RES * j * krow : Ku + RES * j * krow;
            const C d01 = KSH ? kp[0] : __ldg(kp), d23 = KSH ? kp[kyp] : __ldg(kp + kyp), d45 = KSH ? kp[2 * kyp] : __ldg(kp + 2 * kyp);
            const T s = j & 1 ? so : T(1), t = j & 1 ? syo : sy;
            constexpr auto pm = &Radix<Q>::perm;
            kernel_mult<T>(d01, d23, d45, s, t, fz ? -s : s, fz ? -t : t, u[0][pm(j)], u[1][pm(j)], u[2][pm(j)]);
        }
#pragma unroll
        for (int c = 0; c < 3; c++) dft<Q, 1>(u[c]);
#pragma unroll
        for (int m = 0; m < Q; m++) {
            const C wk = __ldg(tz + 2 * Q + m);
            if (RES == 4) {
                const C ws = __ldg(tz + 3 * Q + m);
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    const C got = shfl_x(c_mul(u[c][m], ws), 2);
                    u[c][m] = c_add(c_mul(u[c][m], wk), got);
                }
            } else {
#pragma unroll
                for (int c = 0; c < 3; c++) u[c][m] = c_mul(u[c][m], wk);
            }
        }
#pragma unroll
        for (int c = 0; c < 3; c++)
#pragma unroll
            for (int m = 0; m < HQ; m++) u[c][m] = c_add(u[c][m], shfl_x(u[c][m + HQ], 1));
        __syncwarp();
        const int row0 = (odd ? HQ : 0) + (up ? Q : 0);
        if (ok) {
#pragma unroll
            for (int m = 0; m < HQ; m++) {
                if (row0 + m < nz) {
#pragma unroll
                    for (int c = 0; c < 3; c++) col[c * cs + (row0 + m) * LS] = u[c][m];
                }
            }
        }
    }
}

template <typename T, int HZ, int RES>
__device__ __noinline__ void z_stage(int H, int LS, int nz, int kyp, const typename Cx<T>::t* __restrict__ Kx,
                                     const typename Cx<T>::t* __restrict__ twz, const unsigned short* __restrict__ pos)
{
    using C = typename Cx<T>::t;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* buf = reinterpret_cast<C*>(smem_raw);  // [3 nz][LS]
    if constexpr (HZ == 1) {
        // one thread per ky': both columns from one kernel row
        for (int k = threadIdx.x; k <= H; k += blockDim.x) {
            const C d01 = __ldg(Kx + k), d23 = __ldg(Kx + kyp + k), d45 = __ldg(Kx + 2 * kyp + k);
            C* p = buf + pos[k];
            kernel_mult<T>(d01, d23, d45, T(1), T(1), T(1), T(1), p[0], p[LS], p[2 * LS]);
            if (k > 0 && k < H) {
                C* q = buf + pos[2 * H - k];
                kernel_mult<T>(d01, d23, d45, T(1), T(-1), T(1), T(-1), q[0], q[LS], q[2 * LS]);
            }
        }
    } else {
        // blockDim is a multiple of 32: a warp's lanes leave the loop together
        z_columns<T, HZ, RES>(H, LS, nz * LS, nz, kyp, Kx, twz, threadIdx.x >> 5, H * RES / 16 + 1, blockDim.x >> 5,
                              [&](int ky) { return buf + pos[ky]; });
    }
    __syncthreads();
}

template <typename T, int CLS, int NT>
__global__ void __launch_bounds__(NT) plane_conv_kernel(const __grid_constant__ PlaneArgs<T> a)
{
    using C = typename Cx<T>::t;
    const int lines = 3 * a.nz, kx = blockIdx.x;
    C* plane = a.X + (size_t)kx * lines * a.ny;
    constexpr auto in_class = [](int id, int H) {
        if (H > plane_h_max(sizeof(T), CLS)) return false;
        if (CLS == 0) return id < N_FINE;
        return id >= N_FINE || !has_coarse(H);
    };
    switch (a.len) {
#define X(i, r1, r2, r3, ...) \
    case i:              \
        if constexpr (in_class(i, r1 * r2 * r3)) y_forward<T, Len<r1, r2, r3, __VA_ARGS__>>(plane, lines, a.ny, a.tw); \
        break;
        BORIS_LENGTHS(X)
#undef X
    }
    const C* Kx = a.K + (size_t)kx * (a.HZ == 1 ? 1 : a.HZ + 1) * 3 * a.kyp;
    switch (a.HZ) {
#define Z(h)  \
    case h:   \
        if constexpr (plane_has(CLS, h)) z_stage<T, h, plane_res(CLS)>(a.H, a.LS, a.nz, a.kyp, Kx, a.twz, a.pos); \
        break;
        Z(1) Z(2) Z(4) Z(6) Z(8) Z(12) Z(16) Z(20) Z(24) Z(32)
#undef Z
    }
    switch (a.len) {
#define X(i, r1, r2, r3, ...) \
    case i:              \
        if constexpr (in_class(i, r1 * r2 * r3)) y_inverse<T, Len<r1, r2, r3, __VA_ARGS__>>(plane, lines, a.ny, a.tw); \
        break;
        BORIS_LENGTHS(X)
#undef X
    }
}

template <typename T, int CLS>
cudaError_t plane_set_attr()
{
    return cudaFuncSetAttribute(plane_conv_kernel<T, CLS, plane_threads_max(sizeof(T), CLS)>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
}

template <typename T, int CLS>
cudaError_t launch_plane_cls(const MixedPlan& m, typename Cx<T>::t* X, const typename Cx<T>::t* K, cudaStream_t st)
{
    using C = typename Cx<T>::t;
    const PlaneArgs<T> a{m.y.id, m.y.n, m.nz, m.HZ, m.y.H, m.y.LS, m.kyp, X, K, (const C*)m.twy, (const C*)m.twz, m.posy};
    plane_conv_kernel<T, CLS, plane_threads_max(sizeof(T), CLS)><<<m.x.H + 1, m.threads, m.smem, st>>>(a);
    return cudaGetLastError();
}

#define PLANE_INST(T, CLS)                              \
    template cudaError_t plane_set_attr<T, CLS>();      \
    template cudaError_t launch_plane_cls<T, CLS>(const MixedPlan&, Cx<T>::t*, const Cx<T>::t*, cudaStream_t);

}  // namespace boris
