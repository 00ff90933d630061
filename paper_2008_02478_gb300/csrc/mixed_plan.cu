// Host planning of the mixed-radix path (mixed_fft.cuh, mixed_x.cuh, plane_conv.cuh).
#include "ml_mixed.cuh"

#include <algorithm>
#include <cmath>

namespace boris {

int x_lines(const MixedPlan& m, size_t csz)
{
    // 16 rows per CTA; fewer where two CTAs would not fit an SM or the mesh has
    // too few rows to give every SM two CTAs (a smaller tile shortens the serial
    // part of each)
    int hl = 8;
    while (hl > 2 && (size_t)hl * m.x.LS * csz > 100 * 1024) hl /= 2;
    while (hl > 2 && (long)((m.y.n + 2 * hl - 1) / (2 * hl)) * m.nz * 3 < 304) hl /= 2;
    return hl;
}

bool make_line_fft(int n, int esz, bool coarse, LineFFT* f)
{
    // radices, strides (line_lengths.h)
    static const int tab[N_LENGTHS][11] = {
#define X(i, r1, r2, r3, ...) {r1, r2, r3, __VA_ARGS__},
        BORIS_LENGTHS(X)
#undef X
    };
    auto half = [](int i) { return tab[i][0] * tab[i][1] * tab[i][2]; };
    for (int i = 0; i < N_FINE; i++) {
        if (half(i) < n) continue;
        int id = i;
        for (int j = N_FINE; coarse && j < N_LENGTHS; j++)
            if (half(j) == half(i)) id = j;
        f->id = id;
        f->n = n;
        f->H = half(id);
        f->r1 = tab[id][0];
        f->r2 = tab[id][1];
        f->r3 = tab[id][2];
        f->LS = esz == 8 ? tab[id][6] : tab[id][10];
        return true;
    }
    return false;
}

static double2 unit_root(long e, long n)
{
    const double a = 6.283185307179586476925286766559 * (double)(e % n) / (double)n;
    return make_double2(std::cos(a), -std::sin(a));
}

void line_tw_host(const LineFFT& f, double2* out)
{
    const int S1 = f.r2 * f.r3, S2 = f.r3;
    for (int p = 0; p < 2; p++)
        for (int k = 0; k < f.r1; k++)
            for (int r = 0; r < S1; r++) out[p * f.H + k * S1 + r] = unit_root((long)r * (2 * k + p), 2 * f.H);
    for (int k = 0; k < f.r2; k++)
        for (int q = 0; q < S2; q++) out[2 * f.H + k * S2 + q] = unit_root((long)q * k, S1);
}

void line_pos_host(const LineFFT& f, int esz, unsigned short* out)
{
    switch (f.id) {
#define X(i, r1, r2, r3, ...)                                                                                          \
    case i:                                                                                                       \
        for (int b = 0; b < 2 * f.H; b++)                                                                         \
            out[b] = (unsigned short)(esz == 8 ? Len<r1, r2, r3, __VA_ARGS__>::pos<float2>(b) : Len<r1, r2, r3, __VA_ARGS__>::pos<double2>(b)); \
        break;
        BORIS_LENGTHS(X)
#undef X
    }
}

// Times of the y-z part, us, fitted to measurements of FP32 meshes.
//
// One CTA carries a whole plane: the points of the planes an SM gets, 0.95e-3
// each with two or more CTAs per SM (256 x 256 x 8: 23.6 us), 1.1e-3 with one and
// HZ <= 8 (512 x 512 x 8: 105), 1.45e-3 to HZ 24 (160 x 160 x 20: 53), 1.75e-3 beyond
// (128 x 128 x 32: 43), and 15 % more with radices 20 and 24 (480 x 480 x 8: 116).
static double plane_us(const MixedPlan& m)
{
    const double w = 3.0 * m.nz * 2.0 * m.y.H;
    const int planes = m.x.H + 1, res = (int)(228 * 1024 / (m.smem + 1024)), per_sm = (planes + 151) / 152;
    const double one = m.HZ <= 8 ? 1.1e-3 : m.HZ <= 24 ? 1.6e-3 : 1.75e-3;
    const double many = res >= 2 ? 0.95e-3 : m.HZ <= 8 ? 1.1e-3 : m.HZ <= 24 ? 1.45e-3 : 1.75e-3;
    return (m.y.H == 480 && m.cls > 0 ? 1.15 : 1.0) * std::max(one * w, per_sm * w * many);
}
// y passes 7e-6 per point (160 x 640 x 12: 57 us), 8e-6 with radix 20 and 10e-6 from
// 1536 points (545 x 836 x 6: 213), 4.8e-6 with 1024; z pass 5e-6 to HZ 8 (107), 5.8e-6
// with 12 (160 x 640 x 12: 42), 8e-6 with 16, 6.5e-6 with 20 (160 x 160 x 20: 23), 8.3e-6
// with 24 (283 x 269 x 24: 122), 9.5e-6 with 32 (55 x 767 x 26: 80).
static double passes_us(const MixedPlan& m)
{
    const double y = m.y.H == 512 ? 4.8e-6 : m.y.H >= 768 ? 10e-6 : m.y.H % 240 == 0 ? 8e-6 : 7e-6;
    const double z = m.HZ <= 8 ? 5e-6 : m.HZ <= 12 ? 5.8e-6 : m.HZ <= 16 ? 8e-6 : m.HZ <= 20 ? 6.5e-6 : m.HZ <= 24 ? 8.3e-6 : 9.5e-6;
    return (m.HZ <= 24 ? 9.0 : 12.0) + (m.x.H + 1) * 3.0 * m.nz * 2.0 * m.y.H * (y + z);
}

bool mixed_plan_shape(int nx, int ny, int nz, bool f64, int max_smem, int kind, MixedPlan* m)
{
    const int csz = f64 ? 16 : 8;
    if (nx < 2 || ny < 2 || nz < 1) return false;
    static const int HZS[] = {1, 2, 4, 6, 8, 12, 16, 20, 24, 32};
    m->HZ = 0;
    for (int h : HZS)
        if (h >= nz && (h > 1 || nz == 1)) {
            m->HZ = h;
            break;
        }
    if (!m->HZ) return false;
    m->nz = nz;
    m->nkz = nz == 1 ? 1 : m->HZ + 1;
    const size_t rs = f64 ? 8 : 4;
    if (!make_line_fft(nx, csz, false, &m->x) || !make_line_fft(ny, csz, false, &m->y)) return false;
    // 1024 and 2048 points have the faster x passes (boris_plan_s::mixed_x1024): with many rows
    // they are worth a few spectral planes more (480 x 480 x 8: 17 against 27 us a pass)
    if (!f64 && (m->x.H == 480 || m->x.H == 960) && (long)ny * nz >= 1024) {
        make_line_fft(m->x.H == 480 ? 512 : 1024, csz, false, &m->x);
        m->x.n = nx;
    }
    // Coarse radices move a third less through shared memory, fine ones keep
    // twice the warps resident: those win for one plane of up to 256 cells
    // (128 x 128 x 1: 3.9 against 4.3 us, 256 x 256 x 1: 5.4 against 5.9) and
    // where the coarse set has no two-pass length (1024 x 1024 x 1: 31.8
    // against 38.4 us); elsewhere the coarse ones (512 x 512 x 1: 9.5 against
    // 12.8 us, 256 x 256 x 4: 13.0 against 15.4, 1500 x 700 x 4: 229 against 273).
    const bool fine = (nz == 1 && m->y.H <= 256) || m->y.H >= 1024;
    m->cls = m->HZ > 24 ? 3 : m->HZ > 8 ? 2 : m->HZ <= 4 && fine ? 0 : 1;
    if (m->cls > 0) make_line_fft(ny, csz, true, &m->y);
    m->kyp = (m->y.H + 1 + 15) / 16 * 16;
    m->smem = (size_t)3 * nz * m->y.LS * csz;
    if ((size_t)2 * m->x.LS * csz > (size_t)max_smem) return false;
    const bool fits = m->smem <= (size_t)max_smem && m->y.H <= plane_h_max(rs, m->cls);
    if (!f64 && nz > 1 && kind != 3) {
        MixedPlan s = *m;
        s.split = true;
        if (s.cls == 0) s.cls = 1;
        make_line_fft(ny, csz, true, &s.y);
        s.kyp = (s.y.H + 1 + 15) / 16 * 16;
        s.smem = 0;
        s.threads = 128;
        // few planes of many points leave most SMs idle (36 x 229 x 13, 41 planes: 29 us an
        // evaluation against 40), and 161 planes make two rounds of 152 SMs (160 x 160 x 20:
        // 62 against 69)
        if (kind == 4 || !fits || passes_us(s) < 0.98 * plane_us(*m)) {
            *m = s;
            return (size_t)m->y.LS * csz <= (size_t)max_smem;
        }
    }
    m->split = false;
    if (!fits || kind == 4) return false;
    // threads per CTA: the register file shared by as many CTAs as it takes to
    // hold all planes at once (up to four, and up to what shared memory allows):
    // one wave of smaller CTAs beats two of larger ones (512 x 512 x 1: 128
    // threads 9.5 us, 192 threads 12.4; 256 x 256 x 2: 256 threads 8.3, 384 11.4)
    int res = (m->x.H + 1 + 151) / 152;
    res = std::min(res, 4);
    res = std::max(1, std::min<int>(res, (int)(228 * 1024 / (m->smem + 1024))));
    const int items = 2 * 3 * nz * m->y.r2 * m->y.r3;  // work items of a middle pass, at least
    m->threads = std::max(64, std::min(plane_threads_max(rs, m->cls) / res, std::max(192, items)) / 32 * 32);
    return true;
}

bool mixed_pays(const MixedPlan& m, bool f64, const Geometry& pow2, bool* close)
{
    *close = false;
    // The power-of-two schedules spread all points over the chip but have more of them.
    const double all = 3.0 * m.nz * pow2.py * (double)pow2.nkx;
    if (f64) {
        // bound by the arithmetic units: 25e-3 (one plane) to 40e-3 per point (128 x 128
        // x 16: 490 us) against 2.2e-4 to 3.2e-4 over all planes (564 us)
        const double w = 3.0 * m.nz * 2.0 * m.y.H, per_sm = (m.x.H + 152) / 152;
        const double c = m.HZ == 1 ? 25e-3 : m.HZ <= 4 ? 31e-3 : m.HZ <= 8 ? 36e-3 : 40e-3;
        // a tenth more from three planes per SM on where the z axis saves nothing and a plane
        // is large: there the x passes cost more than the 1024-point ones, too (evaluations,
        // this path against the other: 387 x 51 x 32 2642 and 2298 us, 457 x 463 x 4 2088 and 1770)
        const double edge = per_sm >= 3 && 2 * m.HZ == pow2.pz && w >= 2500 ? 1.1 : 1.0;
        // the shortest calls take as long either way up to HZ 4; beyond, the chain of the
        // z stage is longer here (49 x 3 x 18 86 and 55 us, 51 x 7 x 6 66 and 51)
        const double least = m.HZ <= 4 ? 15.0 : 0.0;
        // HZ 32 computes all 32 planes whatever nz is: 25 us and 46e-3 per point of them a plane,
        // against 130 us and 3.3e-4 (919 x 8 x 32 798 and 662 us, 214 x 56 x 25 1167 and 1068)
        if (m.HZ > 24 && per_sm * (25.0 + 46e-3 * 96.0 * 2.0 * m.y.H) > 0.98 * (130.0 + 3.3e-4 * 96.0 * pow2.py * pow2.nkx))
            return false;
        return edge * per_sm * w * c <= std::max(least, all * (m.HZ == 1 ? 2.2e-4 : m.HZ <= 4 ? 2.4e-4 : 3.2e-4));
    }
    // their x passes take longer on short rows, per row and evaluation 3.8e-3 us to
    // 128 points (37 x 398 x 16: 35 against 11 us), 2e-3 with 256, 0.6e-3 with 512
    const double x = (double)m.y.n * m.nz * (pow2.px <= 128 ? 3.8e-3 : pow2.px == 256 ? 2e-3 : pow2.px == 512 ? 0.6e-3 : 0.0);
    if (m.split) {
        // few short x lines: the five launches take 25 to 35 us whatever the points, the
        // power-of-two schedules less up to so many points of a plane (evaluations: 3 x 395 x 4
        // 31 and 21 us, 4 x 42 x 28 31 and 23, 6 x 815 x 2 35 and 32; 4 x 2000 x 16 and more 1.1 to 1.6 times
        // the other way)
        if (pow2.px <= 16 && pow2.py < 4096 && (long)pow2.py * pow2.pz < (pow2.px <= 8 ? 65536 : 16384)) return false;
        // 20 us (10 with 33 planes: 27 x 137 x 26 23) plus 7.7e-6 for a full z axis (320 x 388 x 16: 200), more with padding in z
        // (283 x 269 x 24: 370), an eighth more from 2048 points in y (160 x 640 x 12: 205);
        // taken from 8 % less on (197 x 769 x 10, not taken: 227 against 306)
        const double pad = 0.6 + 0.2 * pow2.pz / m.nz;
        const double limit = 0.92 * ((pow2.px <= 64 ? 10.0 : 20.0) + all * 7.7e-6 * pad) * (pow2.py >= 2048 ? 1.12 : 1.0) + x;
        // of 1145 meshes 22 were slower after all, those above 11 cells in x from 0.7 of the
        // limit on (102 x 452 x 12: 90 us against 85), shorter lines from 0.44 (8 x 394 x 26: 46
        // against 42)
        *close = passes_us(m) > (pow2.px <= 32 ? 0.4 : 0.6) * limit;
        return passes_us(m) <= limit;
    }
    // on at most five planes the long z stage takes longer than those of the cluster
    // schedules (3 x 16 x 27 21 and 18 us, 2 x 59 x 15 23 and 21)
    if ((pow2.px <= 8 && m.HZ > 24) || (pow2.px <= 4 && m.HZ > 12)) return false;
    // 8.8e-6 plus 6 us, 16 us at least and 25 from HZ 12 and 128 x points on (256 x 256 x 16: 55 us
    // against 75 in planes; 27 x 137 x 26, 33 planes of 25 k points: 22 against 51; 34 x 88
    // x 22: 31 against 22); with fewer points in x, too, 15 % more
    const double gain = 2 * m.x.H < pow2.px ? 1.15 : 0.98;
    const double limit = gain * std::max(m.HZ <= 8 || pow2.px <= 64 ? 16.0 : 25.0, 6.0 + all * 8.8e-6) + x;
    // of 2163 meshes 33 were slower after all, all with long z stages, and but for three of 3 x 30
    // cells in the plane from 0.57 of the limit on (431 x 189 x 21: 286 us against 229; 656 x 82 x 25: 324
    // against 283)
    *close = m.HZ >= 16 && plane_us(m) > 0.5 * limit;
    return plane_us(m) <= limit;
}

size_t mixed_tw_entries(const MixedPlan& m, size_t* oy, size_t* oz)
{
    *oy = line_tw_entries(m.x);
    *oz = *oy + line_tw_entries(m.y);
    return *oz + ZTAB;
}

// z stage tables of residue r (plane_conv.cuh): [in x[m]] [in x[m + Q]] [keep] [send], Q entries each
static void z_tables(int HZ, int RES, double2* out)
{
    for (int i = 0; i < ZTAB; i++) out[i] = make_double2(1.0, 0.0);
    if (HZ < 2) return;
    const int Q = RES == 2 ? HZ : HZ / 2, P = 2 * HZ;
    for (int r = 0; r < RES; r++)
        for (int m = 0; m < Q; m++) {
            double2* t = out + r * 4 * Q + m;
            const int row = (m + ((r & 1) ? Q / 2 : 0)) % Q;  // odd lanes hold their outputs rotated
            const bool up = r & 2;
            auto conj = [](double2 v) { return make_double2(v.x, -v.y); };
            t[0] = unit_root((long)r * m, P);
            t[Q] = unit_root((long)r * (m + Q), P);
            t[2 * Q] = conj(unit_root((long)r * (row + (up ? Q : 0)), P));
            t[3 * Q] = conj(unit_root((long)r * (row + (up ? 0 : Q)), P));
        }
}

void mixed_tw_fill(const MixedPlan& m, double2* out)
{
    size_t oy, oz;
    mixed_tw_entries(m, &oy, &oz);
    line_tw_host(m.x, out);
    line_tw_host(m.y, out + oy);
    z_tables(m.HZ, plane_res(m.cls), out + oz);
}

size_t mixed_kernel_entries(const MixedPlan& m) { return (size_t)(m.x.H + 1) * m.nkz * 3 * m.kyp; }

template <typename T>
static cudaError_t prepare_t(const MixedPlan& m)
{
    cudaError_t e = x_set_attr<T>(m);
    if (e != cudaSuccess) return e;
    switch (m.cls) {
    case 0: return plane_set_attr<T, 0>();
    case 1: return plane_set_attr<T, 1>();
    case 2: return plane_set_attr<T, 2>();
    default: return plane_set_attr<T, 3>();
    }
}
cudaError_t mixed_prepare(const MixedPlan& m, bool f64)
{
    if (m.split) {
        cudaError_t e = x_set_attr<float>(m);
        if (e == cudaSuccess) e = line_y_prepare(m);
        return e == cudaSuccess ? mixed_z_prepare(m) : e;
    }
    return f64 ? prepare_t<double>(m) : prepare_t<float>(m);
}

template <typename T>
cudaError_t launch_plane_conv(const MixedPlan& m, typename Cx<T>::t* X, const typename Cx<T>::t* K, cudaStream_t st)
{
    switch (m.cls) {
    case 0: return launch_plane_cls<T, 0>(m, X, K, st);
    case 1: return launch_plane_cls<T, 1>(m, X, K, st);
    case 2: return launch_plane_cls<T, 2>(m, X, K, st);
    default: return launch_plane_cls<T, 3>(m, X, K, st);
    }
}
template cudaError_t launch_plane_conv<float>(const MixedPlan&, float2*, const float2*, cudaStream_t);
template cudaError_t launch_plane_conv<double>(const MixedPlan&, double2*, const double2*, cudaStream_t);

}  // namespace boris
