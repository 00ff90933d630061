// Mixed-radix transforms of zero-padded lines in shared memory.
//
// The convolution needs a transform length of at least 2n - 1 along an axis of
// n cells; a power of two wastes up to half of it per axis (n = 160: 512
// points where 320 suffice).  Here the padded length is 2 H with H >= n from a
// fine set of products r1 r2 r3 of the radices 2..16 (from 12 on, a length is at
// most a third above the one before and on average a fifth; below, up to a half),
// so ragged meshes pay for their own size.
//
// The padded line is zero from n on (n <= H), so its even and odd outputs are
// two length-H transforms of the same input: X[2k + p] = DFT_H(x[n] w_2H^(p n)).
// Both are stored side by side (parity blocks) and each runs as up to three
// in-place decimation-in-frequency passes
//   n = a S1 + r      : k1 = DFT_r1 over a, times w_2H^(r (2 k1 + p))
//   r = b S2 + q      : k2 = DFT_r2 over b, times w_S1^(q k2)
//   q                 : k3 = DFT_r3 over q
// with S1 = r2 r3, S2 = r3, so that bin 2 (k1 + r1 k2 + r1 r2 k3) + p sits at
// digit position (p, k1, k2, k3).  The spectrum is never put in order: the
// multiply reads it through a position table, and the inverse runs the passes
// backwards.  A thread holds one DFT of <= 32 points in registers, with
// literal inner twiddles; the twiddles between passes are contiguous rows of a
// table in global memory (read through L1, so no shared copy has to be filled
// before the first pass can start).  The length is a template argument: with
// run-time strides the address arithmetic was a quarter of all instructions
// (256 x 256 x 8 plane kernel: 21.9 M warp instructions, 5.6 M of them integer).
//
// Shared layout of a line: digits (p, k1, k2, k3) at strides OFF, P1, P2, 1,
// chosen per length so that the passes and the multiply meet few bank
// conflicts (gen_lengths.py).
#pragma once
#include "fft_engine.cuh"
#include "line_lengths.h"
#include "twiddle480.h"

namespace boris {

// A half length by its radices and the strides of a stored line
// (line_lengths.h).  The fine set, ascending, has small radices (r1 <= 8: the
// last inverse pass holds both parities of its r1 points), so a thread needs
// 64 registers; the coarse set replaces lengths 120..768 by two passes of
// larger radices (128 registers): a third less shared-memory traffic.
template <int R1_, int R2_, int R3_, int P2f, int P1f, int OFFf, int LSf, int P2d, int P1d, int OFFd, int LSd>
struct Len {
    static constexpr int R1 = R1_, R2 = R2_, R3 = R3_;
    static constexpr int H = R1 * R2 * R3, S1 = R2 * R3, S2 = R3;
    template <typename C> static constexpr int P2 = sizeof(C) == 8 ? P2f : P2d;
    template <typename C> static constexpr int P1 = sizeof(C) == 8 ? P1f : P1d;
    template <typename C> static constexpr int OFF = sizeof(C) == 8 ? OFFf : OFFd;
    template <typename C> static constexpr int LS = sizeof(C) == 8 ? LSf : LSd;
    // place of r = k2 S2 + k3 in a block
    template <typename C> __host__ __device__ static constexpr int at(int r) { return r / S2 * P2<C> + r % S2; }
    // position of bin b in a stored line
    template <typename C> __host__ __device__ static constexpr int pos(int b)
    {
        const int k = b >> 1, k1 = k % R1, k2 = (k / R1) % R2, k3 = k / (R1 * R2);
        return (b & 1) * OFF<C> + k1 * P1<C> + k2 * P2<C> + k3;
    }
};

// whether the coarse set has a half length
__host__ __device__ constexpr bool has_coarse(int H)
{
#define X(i, r1, r2, r3, ...) if (H == r1 * r2 * r3) return true;
    BORIS_LENGTHS_COARSE(X)
#undef X
    return false;
}

// One padded axis on the host.
struct LineFFT {
    int id;             // index in BORIS_LENGTHS
    int n, H;           // cells along the axis (n <= H); padded length 2 H
    int r1, r2, r3;
    int LS;             // line stride in shared memory
};

// The axis plan for n cells; esz = bytes per complex value (8 or 16); coarse
// takes the larger radices where the length has them.
bool make_line_fft(int n, int esz, bool coarse, LineFFT* f);
// entries of the twiddle tables of an axis: [2][H] first-pass, then [S1] second-pass
inline int line_tw_entries(const LineFFT& f) { return 2 * f.H + f.r2 * f.r3; }
void line_tw_host(const LineFFT& f, double2* out);
// position of bin k (0 <= k < 2 H) in a stored line
void line_pos_host(const LineFFT& f, int esz, unsigned short* out);

// w_N^e (N divides 480) for a compile-time e
template <int N> struct WLit {
    template <typename C> static __device__ __forceinline__ C get(int e)
    {
        constexpr int u = 480 / N;
        using R = decltype(C::x);
        return C{(R)w480_re((e % N) * u), (R)w480_im((e % N) * u)};
    }
};

// v * w_N^e (DIR < 0) or v * conj(w_N^e), exact for multiples of a quarter turn
template <int DIR, int N, typename C>
__device__ __forceinline__ C rot(C v, int e)
{
    e %= N;
    if (e == 0) return v;
    if (4 * e == N) return DIR < 0 ? C{v.y, -v.x} : C{-v.y, v.x};
    if (2 * e == N) return C{-v.x, -v.y};
    if (4 * e == 3 * N) return DIR < 0 ? C{-v.y, v.x} : C{v.y, -v.x};
    const C w = WLit<N>::template get<C>(e);
    return DIR < 0 ? c_mul(v, w) : c_mulc(v, w);
}

template <int DIR, typename C>
__device__ __forceinline__ void dft3(C& a, C& b, C& c)
{
    using T = decltype(a.x);
    const C s = c_add(b, c), d = c_sub(b, c);
    const C m{a.x - T(0.5) * s.x, a.y - T(0.5) * s.y};
    constexpr T q = (T)0.86602540378443864676;
    // DIR < 0: X1 = m - i q d, X2 = m + i q d
    const C t = DIR < 0 ? C{q * d.y, -q * d.x} : C{-q * d.y, q * d.x};
    a = c_add(a, s);
    b = c_add(m, t);
    c = c_sub(m, t);
}

template <int DIR, typename C>
__device__ __forceinline__ void dft5(C& a, C& b, C& c, C& d, C& e)
{
    using T = decltype(a.x);
    constexpr T c1 = (T)0.30901699437494742410, c2 = (T)-0.80901699437494742410;
    constexpr T s1 = (T)0.95105651629515357212, s2 = (T)0.58778525229247312917;
    const C t1 = c_add(b, e), t2 = c_add(c, d), t3 = c_sub(b, e), t4 = c_sub(c, d);
    const C m1{a.x + c1 * t1.x + c2 * t2.x, a.y + c1 * t1.y + c2 * t2.y};
    const C m2{a.x + c2 * t1.x + c1 * t2.x, a.y + c2 * t1.y + c1 * t2.y};
    const C n1{s1 * t3.x + s2 * t4.x, s1 * t3.y + s2 * t4.y};
    const C n2{s2 * t3.x - s1 * t4.x, s2 * t3.y - s1 * t4.y};
    // DIR < 0: X1 = m1 - i n1, X4 = m1 + i n1, X2 = m2 - i n2, X3 = m2 + i n2
    const C i1 = DIR < 0 ? C{n1.y, -n1.x} : C{-n1.y, n1.x};
    const C i2 = DIR < 0 ? C{n2.y, -n2.x} : C{-n2.y, n2.x};
    a = c_add(a, c_add(t1, t2));
    b = c_add(m1, i1);
    e = c_sub(m1, i1);
    c = c_add(m2, i2);
    d = c_sub(m2, i2);
}

// Radix R = A 2^m with A in {1, 3, 5}: register DFT, natural order in, output k
// at register perm(k) (DIR < 0); DIR > 0 takes that order back to natural.
template <int R> struct Radix {
    static constexpr int A = R % 5 == 0 ? 5 : R % 3 == 0 ? 3 : 1;
    static constexpr int Q = R / A;  // power of two
    static constexpr int LQ = reg_fft_lg(Q);
    __host__ __device__ static constexpr int brev(int v)
    {
        int r = 0;
        for (int b = 0; b < LQ; b++) r |= ((v >> b) & 1) << (LQ - 1 - b);
        return r;
    }
    __host__ __device__ static constexpr int perm(int k) { return A == 1 ? brev(k) : (k % A) * Q + brev(k / A); }
};

template <int R, int DIR, typename C>
__device__ __forceinline__ void dft(C* v)
{
    constexpr int A = Radix<R>::A, Q = Radix<R>::Q;
    if constexpr (A == 1) {
        reg_fft<R, DIR>(v);
    } else if constexpr (DIR < 0) {
#pragma unroll
        for (int j = 0; j < Q; j++) {
            if constexpr (A == 3) dft3<DIR>(v[j], v[j + Q], v[j + 2 * Q]);
            else dft5<DIR>(v[j], v[j + Q], v[j + 2 * Q], v[j + 3 * Q], v[j + 4 * Q]);
#pragma unroll
            for (int k = 1; k < A; k++) v[j + k * Q] = rot<DIR, R>(v[j + k * Q], j * k);
        }
#pragma unroll
        for (int k = 0; k < A; k++) reg_fft<Q, DIR>(v + k * Q);
    } else {
#pragma unroll
        for (int k = 0; k < A; k++) reg_fft<Q, DIR>(v + k * Q);
#pragma unroll
        for (int j = 0; j < Q; j++) {
#pragma unroll
            for (int k = 1; k < A; k++) v[j + k * Q] = rot<DIR, R>(v[j + k * Q], j * k);
            if constexpr (A == 3) dft3<DIR>(v[j], v[j + Q], v[j + 2 * Q]);
            else dft5<DIR>(v[j], v[j + Q], v[j + 2 * Q], v[j + 3 * Q], v[j + 4 * Q]);
        }
    }
}

// First forward pass of `lines` lines: load(line, n, par) gives the input
// (n < H, zero beyond the axis' cells).  One thread takes both parities of its
// r1 inputs, which are then loaded once (up to 16 of them); FOLD: the caller folds an unpadded
// line, so the inputs differ by parity.  tw: the axis' tables.
template <typename L, bool FOLD = false, typename C, typename Load>
__device__ __forceinline__ void line_fwd1(int lines, C* buf, const C* __restrict__ tw, Load load)
{
    constexpr int R = L::R1, S1 = L::S1;
    constexpr bool AGAIN = FOLD || R > 16;  // above 16 points registers allow one parity at a time
    for (int it = threadIdx.x; it < lines * S1; it += blockDim.x) {
        const int line = it / S1, r = it % S1;
        C* dst = buf + line * L::template LS<C> + L::template at<C>(r);
        const C* t = tw + r;
        C v[R], u[R];
#pragma unroll
        for (int a = 0; a < R; a++) v[a] = load(line, a * S1 + r, false);
        if (!AGAIN) {
#pragma unroll
            for (int a = 0; a < R; a++) u[a] = rot<-1, 2 * R>(v[a], a);
        }
        dft<R, -1>(v);
        dst[0] = v[0];  // its twiddle is 1
#pragma unroll
        for (int k = 1; k < R; k++) dst[k * L::template P1<C>] = c_mul(v[Radix<R>::perm(k)], __ldg(t + k * S1));
        if (AGAIN) {
#pragma unroll
            for (int a = 0; a < R; a++) u[a] = rot<-1, 2 * R>(load(line, a * S1 + r, true), a);
        }
        dft<R, -1>(u);
#pragma unroll
        for (int k = 0; k < R; k++)
            dst[L::template OFF<C> + k * L::template P1<C>] = c_mul(u[Radix<R>::perm(k)], __ldg(t + L::H + k * S1));
    }
}

// Later passes on stored lines, in place; each ends with a block barrier.
template <typename L, int DIR, typename C>
__device__ __forceinline__ void line_pass2(int lines, C* buf, const C* __restrict__ tw)
{
    constexpr int R = L::R2, S2 = L::S2, P2 = L::template P2<C>;
    const C* t2 = tw + 2 * L::H;
    for (int it = threadIdx.x; it < 2 * lines * L::R1 * S2; it += blockDim.x) {
        const int q = it / S2, r = it % S2;
        const int lp = q / L::R1, k1 = q % L::R1;
        C* p = buf + (lp >> 1) * L::template LS<C> + ((lp & 1) ? L::template OFF<C> : 0) + k1 * L::template P1<C> + r;
        C v[R];
        if (DIR < 0) {
#pragma unroll
            for (int a = 0; a < R; a++) v[a] = p[a * P2];
            dft<R, -1>(v);
#pragma unroll
            for (int k = 0; k < R; k++) {
                const C u = v[Radix<R>::perm(k)];
                p[k * P2] = S2 > 1 && k > 0 ? c_mul(u, __ldg(t2 + k * S2 + r)) : u;
            }
        } else {
#pragma unroll
            for (int k = 0; k < R; k++) {
                const C u = p[k * P2];
                v[Radix<R>::perm(k)] = S2 > 1 && k > 0 ? c_mulc(u, __ldg(t2 + k * S2 + r)) : u;
            }
            dft<R, 1>(v);
#pragma unroll
            for (int a = 0; a < R; a++) p[a * P2] = v[a];
        }
    }
    __syncthreads();
}

template <typename L, int DIR, typename C>
__device__ __forceinline__ void line_pass3(int lines, C* buf)
{
    constexpr int R = L::R3;
    for (int it = threadIdx.x; it < 2 * lines * L::R1 * L::R2; it += blockDim.x) {
        const int q = it / L::R2, k2 = it % L::R2;
        const int lp = q / L::R1, k1 = q % L::R1;
        C* p = buf + (lp >> 1) * L::template LS<C> + ((lp & 1) ? L::template OFF<C> : 0) + k1 * L::template P1<C> +
               k2 * L::template P2<C>;
        C v[R];
        if (DIR < 0) {
#pragma unroll
            for (int a = 0; a < R; a++) v[a] = p[a];
            dft<R, -1>(v);
#pragma unroll
            for (int k = 0; k < R; k++) p[k] = v[Radix<R>::perm(k)];
        } else {
#pragma unroll
            for (int k = 0; k < R; k++) v[Radix<R>::perm(k)] = p[k];
            dft<R, 1>(v);
#pragma unroll
            for (int a = 0; a < R; a++) p[a] = v[a];
        }
    }
    __syncthreads();
}

// Last inverse pass: store(line, n, value) receives n < H (the caller crops to
// its cells).  One thread sums both parities of its r1 outputs; above 16
// points the even ones wait in the (consumed) even block meanwhile.
template <typename L, typename C, typename Store>
__device__ __forceinline__ void line_inv1(int lines, C* buf, const C* __restrict__ tw, Store store)
{
    constexpr int R = L::R1, S1 = L::S1, P1 = L::template P1<C>;
    constexpr bool PARK = R > 16;
    for (int it = threadIdx.x; it < lines * S1; it += blockDim.x) {
        const int line = it / S1, r = it % S1;
        C* src = buf + line * L::template LS<C> + L::template at<C>(r);
        const C* t = tw + r;
        C v[R];
        v[0] = src[0];  // its twiddle is 1
#pragma unroll
        for (int k = 1; k < R; k++) v[Radix<R>::perm(k)] = c_mulc(src[k * P1], __ldg(t + k * S1));
        dft<R, 1>(v);
        if (PARK) {
#pragma unroll
            for (int a = 0; a < R; a++) src[a * P1] = v[a];
        }
        C u[R];
#pragma unroll
        for (int k = 0; k < R; k++)
            u[Radix<R>::perm(k)] = c_mulc(src[L::template OFF<C> + k * P1], __ldg(t + L::H + k * S1));
        dft<R, 1>(u);
#pragma unroll
        for (int a = 0; a < R; a++) store(line, a * S1 + r, c_add(PARK ? src[a * P1] : v[a], rot<1, 2 * R>(u[a], a)));
    }
}

// All forward passes after line_fwd1 (barrier included) / all inverse passes before line_inv1.
template <typename L, typename C>
__device__ __forceinline__ void line_fwd_rest(int lines, C* buf, const C* __restrict__ tw)
{
    __syncthreads();
    if constexpr (L::R2 > 1) line_pass2<L, -1>(lines, buf, tw);
    if constexpr (L::R3 > 1) line_pass3<L, -1>(lines, buf);
}
template <typename L, typename C>
__device__ __forceinline__ void line_inv_rest(int lines, C* buf, const C* __restrict__ tw)
{
    if constexpr (L::R3 > 1) line_pass3<L, 1>(lines, buf);
    if constexpr (L::R2 > 1) line_pass2<L, 1>(lines, buf, tw);
}

}  // namespace boris
