// Passes of the multi-mesh transform on mixed-radix lengths (ml_mixed.cu): the
// x transforms read and write the layers' own arrays, and the y transforms know
// which rows of a plane exist, so the frame around the layers is neither stored
// nor transformed along x.
#pragma once
#include "mixed_demag.cuh"

namespace boris {

// One plane of the frame: its layer's extent and place.
struct MLPlane {
    int nx, ny, ox, oy;
    size_t off;   // row 0 of component 0 of the plane in the concatenated field
    size_t comp;  // component stride of the layer
    size_t moff;  // row 0 of the plane in a concatenated map
};

struct MLMixed {
    MixedPlan m;            // axis plans and tables (z fields unused)
    int Z;
    int rows;               // most rows of any plane
    const MLPlane* planes;  // device [Z]
};

bool ml_mixed_shape(int NX, int NY, int Z, int max_smem, MLMixed* p);
cudaError_t ml_mixed_prepare(const MLMixed& p);
cudaError_t launch_ml_x_fwd(const MLMixed& p, const float* M, const float* ms_map, float ms, float2* X, cudaStream_t st);
cudaError_t launch_ml_x_inv(const MLMixed& p, const float2* X, float* H, cudaStream_t st);
// y transforms of all lines [kx][nlines] between X[..][ny] and Y[..][2 H] (natural
// order); planes: the windows of planes line mod Z, or NULL
cudaError_t line_y_prepare(const MixedPlan& m);
cudaError_t launch_line_y(const MixedPlan& m, const MLPlane* planes, int nlines, int Z, float2* X, float2* Y, cudaStream_t st,
                          bool forward);

// the length-1024 passes of demag_fast.cu on such a frame (y: or, with planes NULL, on full rows)
cudaError_t launch_ml_x_r2c_1024(const Geometry& g, const MLPlane* planes, int rows, const float* M, const float* ms_map,
                                 float ms, float2* X, const float2* tw, cudaStream_t st);
cudaError_t launch_ml_y_1024(const Geometry& g, const MLPlane* planes, float2* X, float2* Y, const float2* tw, cudaStream_t st,
                             bool forward);

}  // namespace boris
