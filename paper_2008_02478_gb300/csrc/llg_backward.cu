// Discrete adjoint of one RK4 step of the LLG equation (the paper has no
// adjoint; this serves gradients of a loss on the final state with respect to
// the initial state and the per-cell Ms and Ku maps).
//
// Forward (recomputed): m1 = m, k_s = f(m_s), m2 = m + dt/2 k1, m3 = m + dt/2 k2,
// m4 = m + dt k3, v = m + dt/6 (k1 + 2k2 + 2k3 + k4), m_out = v/|v|, with
// f(m) = -g' [a + alpha m x a], a = m x H(m), H = Hd(Ms m) + c lap m
// + (2Ku/(mu0 Ms))(m.e)e + Hext, c = 2A/(mu0 Ms).
// Backward: gv = (g - m_out (m_out.g))/|v|; gk_s = w_s dt gv; for s = 4..1 the
// VJP of f at m_s gives gm_s, added to g_m and to gk_{s-1} (times the stage
// coefficient).  The VJP of f splits into a per-cell part (cross products)
// and the field transpose: the demagnetising operator is self-adjoint, so its
// transpose is one more demag application; the Neumann Laplacian is
// symmetric, so its transpose is itself.
//
// Kernels, one between any two demag applications: fwd_stage (stages 1..3),
// bwd_turn (stage 4 of the recompute, the renormalisation's VJP and the
// per-cell VJP at m4) and bwd_field (field transpose at m_s and, s > 1, the
// per-cell VJP at m_{s-1}: gk never goes to memory).  All neighbours load
// unconditionally (llg_cell.cuh), and 1/(mu0 Ms) comes from a map made once per
// call.  Bound by load latency and L2 traffic (256 x 256 x 8: 17 to 28 fields of
// 6.3 MB a kernel, all in L2): bwd_field and bwd_local 24.7 + 5.4 -> 16.8 us (the
// divisions alone 11 us), bwd_start and the last fwd_stage 11.5 + 9.5 -> 14.
#include "boris_internal.cuh"
#include "llg_cell.cuh"
#include "llg_kernels.cuh"

namespace boris {

// Values of the three components of f at a cell's neighbours.
template <typename T>
__device__ __forceinline__ void load_neighbours(const T* __restrict__ f, unsigned n, const Neighbours& q, T nb[3][6])
{
#pragma unroll
    for (int c = 0; c < 3; c++) {
        nb[c][0] = f[c * n + q.xm];
        nb[c][1] = f[c * n + q.xp];
        nb[c][2] = f[c * n + q.ym];
        nb[c][3] = f[c * n + q.yp];
        nb[c][4] = f[c * n + q.zm];
        nb[c][5] = f[c * n + q.zp];
    }
}
template <typename T>
__device__ __forceinline__ T lap_of(const LLGArgs<T>& a, const T nb[6], T m)
{
    T l = a.ihx2 * (nb[0] - m);
    l += a.ihx2 * (nb[1] - m);
    l += a.ihy2 * (nb[2] - m);
    l += a.ihy2 * (nb[3] - m);
    l += a.ihz2 * (nb[4] - m);
    l += a.ihz2 * (nb[5] - m);
    return l;
}

struct Cell {
    unsigned i;
    int x, y, z;
};
template <typename T>
__device__ __forceinline__ Cell cell_of(const LLGArgs<T>& a, unsigned i)
{
    const unsigned nx = a.nx, ny = a.ny, row = i / nx;
    Cell q;
    q.i = i;
    q.x = (int)(i - row * nx);
    q.z = (int)(row / ny);
    q.y = (int)(row - (unsigned)q.z * ny);
    return q;
}

// m, total field H and rate k of a cell at stage state ms
template <typename T>
__device__ __forceinline__ void cell_field(const LLGArgs<T>& a, const T* __restrict__ ms, const T* __restrict__ Hd, Cell q,
                                           T m[3], T H[3], T k[3])
{
    const unsigned n = (unsigned)a.ncell, i = q.i;
    T nb[3][6];
    load_neighbours(ms, n, neighbours(a, i, q.x, q.y, q.z), nb);
#pragma unroll
    for (int c = 0; c < 3; c++) {
        m[c] = ms[c * n + i];
        H[c] = Hd[c * n + i];
    }
    const T Ms = a.ms_map ? a.ms_map[i] : a.Ms;
    const T Ku = a.ku_map ? a.ku_map[i] : a.Ku;
    const T inv = inv_mu0_ms(a, Ms);
    const T me = m[0] * a.e[0] + m[1] * a.e[1] + m[2] * a.e[2];
#pragma unroll
    for (int c = 0; c < 3; c++)
        H[c] = H[c] + T(2) * a.A * inv * lap_of(a, nb[c], m[c]) + T(2) * Ku * inv * me * a.e[c] + a.Hext[c];
    rhs_from_field(a, m, H, k);
}

// Forward stage of the recompute, s in 0..2: stores the stage state's effective
// field H_s and k_s, and the next stage state.  ms = m_s; Hd = demag of Ms m_s.
template <typename T>
__global__ void __launch_bounds__(256) fwd_stage_kernel(LLGArgs<T> a, int s, const T* __restrict__ ms,
                                                        const T* __restrict__ Hd, const T* __restrict__ m0,
                                                        T* __restrict__ Hs, T* __restrict__ ks,
                                                        T* __restrict__ mnext)
{
    const unsigned n = (unsigned)a.ncell;
    const T cdt = s == 2 ? a.dt : T(0.5) * a.dt;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        T b[3], m[3], H[3], k[3];
#pragma unroll
        for (int c = 0; c < 3; c++) b[c] = m0[c * n + i];
        cell_field(a, ms, Hd, cell_of(a, i), m, H, k);
#pragma unroll
        for (int c = 0; c < 3; c++) {
            Hs[c * n + i] = H[c];
            ks[c * n + i] = k[c];
            mnext[c * n + i] = b[c] + cdt * k[c];
        }
    }
}

// Per-cell part of the VJP of f at (m, H) from the cotangent g of its rate:
// gh = ga x m (ga = -g' g + (-g' alpha g) x m) and the local part gml = a x gB + H x ga.
template <typename T>
__device__ __forceinline__ void local_vjp(const LLGArgs<T>& a, const T m[3], const T H[3], const T g[3], T gh[3], T gml[3])
{
    const T A_[3] = {m[1] * H[2] - m[2] * H[1], m[2] * H[0] - m[0] * H[2], m[0] * H[1] - m[1] * H[0]};
    const T gA[3] = {-a.gp * g[0], -a.gp * g[1], -a.gp * g[2]};
    const T gB[3] = {gA[0] * a.alpha, gA[1] * a.alpha, gA[2] * a.alpha};
    // b = m x a: d/dm = a x gB, d/da = gB x m
    const T ga[3] = {gA[0] + gB[1] * m[2] - gB[2] * m[1], gA[1] + gB[2] * m[0] - gB[0] * m[2],
                     gA[2] + gB[0] * m[1] - gB[1] * m[0]};
    const T gm1[3] = {A_[1] * gB[2] - A_[2] * gB[1], A_[2] * gB[0] - A_[0] * gB[2], A_[0] * gB[1] - A_[1] * gB[0]};
    // a = m x H: d/dm = H x ga, d/dH = ga x m
    const T gm2[3] = {H[1] * ga[2] - H[2] * ga[1], H[2] * ga[0] - H[0] * ga[2], H[0] * ga[1] - H[1] * ga[0]};
    gh[0] = ga[1] * m[2] - ga[2] * m[1];
    gh[1] = ga[2] * m[0] - ga[0] * m[2];
    gh[2] = ga[0] * m[1] - ga[1] * m[0];
#pragma unroll
    for (int c = 0; c < 3; c++) gml[c] = gm1[c] + gm2[c];
}

// imap[i] = 1 / (mu0 Ms_i): nine divisions per cell and stage of bwd_field otherwise
template <typename T>
__global__ void __launch_bounds__(256) bwd_inv_ms_kernel(LLGArgs<T> a, T* __restrict__ imap)
{
    const unsigned n = (unsigned)a.ncell;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        imap[i] = inv_mu0_ms(a, a.ms_map[i]);
}

// Where the recompute turns into the backward pass: k4 = f(m4), v from the
// rates, gv = (g - m_out (m_out.g))/|v|, g_m = gv, and the per-cell VJP at m4
// of gk_4 = dt/6 gv.  gv is kept for the other stages' gk.
template <typename T>
__global__ void __launch_bounds__(256) bwd_turn_kernel(LLGArgs<T> a, const T* __restrict__ m4, const T* __restrict__ Hd,
                                                       const T* __restrict__ m0, const T* __restrict__ ks,
                                                       const T* __restrict__ gout, T* __restrict__ gm,
                                                       T* __restrict__ gvb, T* __restrict__ gH, T* __restrict__ gml)
{
    const unsigned n = (unsigned)a.ncell;
    const size_t n3 = 3 * (size_t)n;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        T v[3], g[3], m[3], H[3], k[3];
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const unsigned j = c * n + i;
            v[c] = m0[j];
            g[c] = gout[j];
            k[c] = ks[j] + T(2) * ks[n3 + j] + T(2) * ks[2 * n3 + j];
        }
        T k4[3];
        cell_field(a, m4, Hd, cell_of(a, i), m, H, k4);
#pragma unroll
        for (int c = 0; c < 3; c++) v[c] = v[c] + a.dt / T(6) * (k[c] + k4[c]);
        const T nv = sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
        const T inv = T(1) / nv;
        const T mo[3] = {v[0] * inv, v[1] * inv, v[2] * inv};
        const T mg = mo[0] * g[0] + mo[1] * g[1] + mo[2] * g[2];
        T gk[3], gh[3], gl[3];
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const T gv = (g[c] - mo[c] * mg) * inv;
            gm[c * n + i] = gv;
            gvb[c * n + i] = gv;
            gk[c] = a.dt / T(6) * gv;
        }
        local_vjp(a, m, H, gk, gh, gl);
#pragma unroll
        for (int c = 0; c < 3; c++) {
            gH[c * n + i] = gh[c];
            gml[c * n + i] = gl[c];
        }
    }
}

// Field transpose at stage state m_s: gm_s = gml + Ms D(gH) + L(c gH)
// + (2Ku/(mu0 Ms))(gH.e)e; accumulates gm_s into g_m and the Ms / Ku gradients.
// MORE: then gk_{s-1} = w gv + coef gm_s and the per-cell VJP at m_{s-1} (mp,
// Hp), which writes the next gH and, in place, gml.  DgH = demag of gH; imap:
// 1 / (mu0 Ms) of each cell (with an Ms map).
template <typename T, bool MORE>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 3 : 1) bwd_field_kernel(LLGArgs<T> a, const T* __restrict__ imap,
                                                        const T* __restrict__ ms,
                                                        const T* __restrict__ gH, const T* __restrict__ DgH,
                                                        T* __restrict__ gml, T* __restrict__ gm,
                                                        const T* __restrict__ gvb, T w, T coef,
                                                        const T* __restrict__ mp, const T* __restrict__ Hp,
                                                        T* __restrict__ gHn, T* __restrict__ gMs, T* __restrict__ gKu)
{
    const unsigned n = (unsigned)a.ncell;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const Cell cl = cell_of(a, i);
        const Neighbours q = neighbours(a, i, cl.x, cl.y, cl.z);
        T gb[3][6], mb[3][6], m[3], g[3], D[3], gl[3], gmv[3], gk[3], pm[3], pH[3];
        load_neighbours(gH, n, q, gb);
        load_neighbours(ms, n, q, mb);
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const unsigned j = c * n + i;
            m[c] = ms[j];
            g[c] = gH[j];
            D[c] = DgH[j];
            gl[c] = gml[j];
            gmv[c] = gm[j];
            if (MORE) {
                gk[c] = gvb[j];
                pm[c] = mp[j];
                pH[c] = Hp[j];
            }
        }
        const T Ms = a.ms_map ? a.ms_map[i] : a.Ms;
        const T Ku = a.ku_map ? a.ku_map[i] : a.Ku;
        const T inv = a.ms_map ? imap[i] : a.inv_ms, iMs = T(MU0_D) * inv;
        const T ci = T(2) * a.A * inv;
        // L(c gH) at i: sum_j w (c_j gH_j - c_i gH_i), c = 2A/(mu0 Ms); a missing
        // neighbour is the cell itself and adds nothing
        T cj[6] = {ci, ci, ci, ci, ci, ci};
        if (a.ms_map) {
            const unsigned at[6] = {q.xm, q.xp, q.ym, q.yp, q.zm, q.zp};
#pragma unroll
            for (int d = 0; d < 6; d++) cj[d] = imap[at[d]];
#pragma unroll
            for (int d = 0; d < 6; d++) cj[d] *= T(2) * a.A;
        }
        const T wd[6] = {a.ihx2, a.ihx2, a.ihy2, a.ihy2, a.ihz2, a.ihz2};
        T lcg[3], lm[3];
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const T cg = ci * g[c];
            T l = T(0);
#pragma unroll
            for (int d = 0; d < 6; d++) l += wd[d] * (cj[d] * gb[c][d] - cg);
            lcg[c] = l;
            lm[c] = lap_of(a, mb[c], m[c]);
        }
        const T me = m[0] * a.e[0] + m[1] * a.e[1] + m[2] * a.e[2];
        const T ge = g[0] * a.e[0] + g[1] * a.e[1] + g[2] * a.e[2];
        if (gMs) {
            T gms = m[0] * D[0] + m[1] * D[1] + m[2] * D[2];
            gms -= ci * iMs * (g[0] * lm[0] + g[1] * lm[1] + g[2] * lm[2]);
            gms -= T(2) * Ku * inv * iMs * me * ge;
            gMs[i] += gms;
        }
        if (gKu) gKu[i] += T(2) * inv * me * ge;
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const T v = gl[c] + Ms * D[c] + lcg[c] + T(2) * Ku * inv * ge * a.e[c];
            gm[c * n + i] = gmv[c] + v;
            if (MORE) gk[c] = w * gk[c] + coef * v;
        }
        if (MORE) {
            T gh[3], gn[3];
            local_vjp(a, pm, pH, gk, gh, gn);
#pragma unroll
            for (int c = 0; c < 3; c++) {
                gHn[c * n + i] = gh[c];
                gml[c * n + i] = gn[c];
            }
        }
    }
}

static int grid_for_n(size_t n)
{
    size_t b = (n + 255) / 256;
    if (b > 152 * 16) b = 152 * 16;
    return (int)(b > 0 ? b : 1);
}

template <typename T>
cudaError_t launch_fwd_stage(const LLGArgs<T>& a, int s, const T* ms, const T* Hd, const T* m0, T* Hs, T* ks,
                             T* mnext, cudaStream_t st)
{
    fwd_stage_kernel<T><<<grid_for_n(a.ncell), 256, 0, st>>>(a, s, ms, Hd, m0, Hs, ks, mnext);
    return cudaGetLastError();
}
template <typename T>
cudaError_t launch_bwd_turn(const LLGArgs<T>& a, const T* m4, const T* Hd, const T* m0, const T* ks, const T* gout, T* gm,
                            T* gvb, T* gH, T* gml, cudaStream_t st)
{
    bwd_turn_kernel<T><<<grid_for_n(a.ncell), 256, 0, st>>>(a, m4, Hd, m0, ks, gout, gm, gvb, gH, gml);
    return cudaGetLastError();
}
template <typename T>
cudaError_t launch_bwd_inv_ms(const LLGArgs<T>& a, T* imap, cudaStream_t st)
{
    bwd_inv_ms_kernel<T><<<grid_for_n(a.ncell), 256, 0, st>>>(a, imap);
    return cudaGetLastError();
}
template <typename T>
cudaError_t launch_bwd_field(const LLGArgs<T>& a, const T* imap, const T* ms, const T* gH, const T* DgH, T* gml, T* gm, const T* gvb, T w,
                             T coef, const T* mp, const T* Hp, T* gHn, T* gMs, T* gKu, cudaStream_t st)
{
    if (mp) bwd_field_kernel<T, true><<<grid_for_n(a.ncell), 256, 0, st>>>(a, imap, ms, gH, DgH, gml, gm, gvb, w, coef, mp, Hp, gHn,
                                                                             gMs, gKu);
    else bwd_field_kernel<T, false><<<grid_for_n(a.ncell), 256, 0, st>>>(a, imap, ms, gH, DgH, gml, gm, gvb, w, coef, mp, Hp, gHn,
                                                                             gMs, gKu);
    return cudaGetLastError();
}

#define BWD_INST(T)                                                                                              \
    template cudaError_t launch_fwd_stage<T>(const LLGArgs<T>&, int, const T*, const T*, const T*, T*, T*, T*,    \
                                             cudaStream_t);                                                      \
    template cudaError_t launch_bwd_turn<T>(const LLGArgs<T>&, const T*, const T*, const T*, const T*, const T*,  \
                                            T*, T*, T*, T*, cudaStream_t);                                       \
    template cudaError_t launch_bwd_inv_ms<T>(const LLGArgs<T>&, T*, cudaStream_t);                              \
    template cudaError_t launch_bwd_field<T>(const LLGArgs<T>&, const T*, const T*, const T*, const T*, T*, T*,  \
                                             const T*, T, T, const T*, const T*, T*, T*, T*, cudaStream_t);
BWD_INST(float)
BWD_INST(double)

}  // namespace boris
