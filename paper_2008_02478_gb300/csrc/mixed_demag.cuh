// Convolution on mixed-radix lengths: x passes (mixed_x.cuh), and for the y-z part
// the plane kernel where a padded kx plane fits one CTA's shared memory
// (plane_conv.cuh; FP32 and FP64) or y, z and y passes (mixed_split.cu; FP32).
// Single-mesh plans take them by mixed_pays.
#pragma once
#include "boris_internal.cuh"
#include "mixed_fft.cuh"

namespace boris {

// Device tables and axis plans of one mesh.
struct MixedPlan {
    LineFFT x, y;
    int nz, HZ;       // planes; half the padded z length (HZ = 1 with nz = 1: no z transform)
    int cls;          // class of the plane kernel
    int nkz;          // kernel rows kz' per kx: HZ + 1, or 1
    int kyp;          // ky' entries per kernel row, H_y + 1 rounded up to 16
    size_t smem;      // shared bytes of the plane kernel
    bool split;       // y, z and y passes over the padded spectrum instead of it (FP32)
    int threads;
    const void* twx;  // twiddle tables of the axes, in the plan's precision
    const void* twy;
    const void* twz;  // the z stage's tables (plane_conv.cuh), ZTAB entries
    const unsigned short* posx;  // bin -> position
    const unsigned short* posy;
};

// The plane kernel comes in classes by register need: class 0 runs the fine
// radices with HZ <= 4, class 1 the coarse ones with HZ <= 8, class 2 and 3 the
// coarse ones with the z transform split over four lanes (HZ <= 24, HZ = 32).
constexpr bool plane_has(int cls, int HZ)
{
    return cls == 0 ? HZ <= 4 : cls == 1 ? HZ <= 8 : cls == 2 ? HZ > 8 && HZ <= 24 : HZ > 24;
}
constexpr int plane_res(int cls) { return cls < 2 ? 2 : 4; }  // lanes that share a column
constexpr int plane_threads_max(size_t real_size, int cls)
{
    if (real_size == 8) return cls == 0 ? 512 : 256;
    return cls == 0 ? 1024 : cls < 3 ? 512 : 384;
}
// longest half length of a class: 3 nz lines of 2 H values in 227 KB
constexpr int plane_h_max(size_t real_size, int cls)
{
    const int h = cls < 2 ? 4096 : cls == 2 ? 480 : 160;
    return real_size == 8 ? h / 2 : h;
}
constexpr int ZTAB = 256;

// Whether the mesh runs on this path (host rule); fills the axis plans.
// kind 3 or 4: the plane kernel or the passes wherever possible, 0: the faster one
bool mixed_plan_shape(int nx, int ny, int nz, bool f64, int max_smem, int kind, MixedPlan* m);
// Whether it is the faster path there by the estimates (pow2: the power-of-two geometry of
// the same mesh); *close: they can be wrong by as much as they differ, so time both.
bool mixed_pays(const MixedPlan& m, bool f64, const Geometry& pow2, bool* close);
// Host tables of the plan, concatenated: [twx | twy | twz], positions [posx | posy]
size_t mixed_tw_entries(const MixedPlan& m, size_t* oy, size_t* oz);
void mixed_tw_fill(const MixedPlan& m, double2* out);
size_t mixed_kernel_entries(const MixedPlan& m);  // complex-sized pairs in the kernel spectrum
// Shared-memory limits of the kernels the plan launches (once, at plan creation).
cudaError_t mixed_prepare(const MixedPlan& m, bool f64);

template <typename T>
cudaError_t launch_mixed_x_fwd(const MixedPlan& m, const T* M, const T* ms_map, T ms, typename Cx<T>::t* X,
                               cudaStream_t st);
template <typename T>
cudaError_t launch_mixed_x_inv(const MixedPlan& m, const typename Cx<T>::t* X, T* H, cudaStream_t st);
template <typename T>
cudaError_t launch_plane_conv(const MixedPlan& m, typename Cx<T>::t* X, const typename Cx<T>::t* K, cudaStream_t st);

// The passes (mixed_split.cu); g, tw: the geometry and twiddles of the 1024-point kernels
cudaError_t launch_mixed_y(const MixedPlan& m, const Geometry& g, float2* X, float2* Y, const float2* tw, cudaStream_t st,
                           bool forward);
cudaError_t mixed_z_prepare(const MixedPlan& m);  // (once, at plan creation)
cudaError_t launch_mixed_z(const MixedPlan& m, float2* Y, const float2* K, cudaStream_t st);

// per-type, per-class pieces (one translation unit each)
template <typename T> cudaError_t x_set_attr(const MixedPlan& m);
template <typename T, int CLS> cudaError_t plane_set_attr();
template <typename T, int CLS>
cudaError_t launch_plane_cls(const MixedPlan& m, typename Cx<T>::t* X, const typename Cx<T>::t* K, cudaStream_t st);
// lines (pairs of rows) per CTA of the x passes
int x_lines(const MixedPlan& m, size_t csz);

// Kernel spectrum on the plan's lengths, K[kx][kz'][pair][ky'] with pairs
// (xx, yy), (zz, xy), (xz, yz), scaled by -1/(px py pz) (newell.cu).
cudaError_t build_mixed_spectrum(const Geometry& g, const MixedPlan& m, double dx, double dy, double dz, double rs,
                                 void* K, bool f64, cudaStream_t st, const int* images);

// One FP64 axis pass of the tensor spectra: [ncomp][d2][d1][d0] with the
// transformed axis of length n -> H + 1 bins (components in the order xx yy zz xy xz yz).
cudaError_t run_mixed_axis(const LineFFT& f, const void* in, bool real, double2* out, int axis, int d0, int d1, int d2,
                           int ncomp, const double2* tw, const unsigned short* pos, cudaStream_t st);

}  // namespace boris
