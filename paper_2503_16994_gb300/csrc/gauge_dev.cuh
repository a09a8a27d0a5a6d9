// Device helpers on FP64 links (3x3 complex matrices in the even-odd SoA
// layout): products, adjoints, neighbours and the clover field strength.
// Used by the clover construction and by the gauge flow and observables.
#pragma once
#include "kernels.cuh"

namespace lqcd {

using cd = cx<double>;
using m3 = su3<double>;

// acc + a b, acc + conj(a) b and acc + a conj(b) as fma chains: four FP64
// instructions per complex product (separate products and sums take six)
__device__ __forceinline__ void cma(cd &acc, cd a, cd b)
{
    acc.re = fma(a.re, b.re, acc.re);
    acc.re = fma(-a.im, b.im, acc.re);
    acc.im = fma(a.re, b.im, acc.im);
    acc.im = fma(a.im, b.re, acc.im);
}
__device__ __forceinline__ cd cm0(cd a, cd b)  // a b
{
    return cd{fma(-a.im, b.im, a.re * b.re), fma(a.im, b.re, a.re * b.im)};
}

// a b: 108 FP64 instructions.  The gauge kernels run at the FP64 pipe's rate
// (89% busy on GB300), so their time is the number of these instructions.
__device__ __forceinline__ m3 mm(const m3 &a, const m3 &b)
{
    m3 r;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            cd t = cm0(a.m[i][0], b.m[0][j]);
            cma(t, a.m[i][1], b.m[1][j]);
            cma(t, a.m[i][2], b.m[2][j]);
            r.m[i][j] = t;
        }
    return r;
}

__device__ __forceinline__ m3 md(const m3 &a)  // a^dag
{
    m3 r;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) r.m[i][j] = conj(a.m[j][i]);
    return r;
}

// An antihermitian 3x3 matrix by its 9 reals: i d on the diagonal, o = the
// entries (0,1), (0,2), (1,2); the lower triangle is -conj.
struct ah3 {
    double d[3];
    cd o[3];
};

__device__ __forceinline__ ah3 ah_zero()
{
    ah3 r;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        r.d[i] = 0.0;
        r.o[i] = cd{0.0, 0.0};
    }
    return r;
}

// acc += a b - (a b)^dag, formed directly: 90 instructions instead of 108 for
// the product and 9 for the difference
__device__ __forceinline__ void ah_add(ah3 &acc, const m3 &a, const m3 &b)
{
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        double im = 0.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            im = fma(a.m[i][k].re, b.m[k][i].im, im);
            im = fma(a.m[i][k].im, b.m[k][i].re, im);
        }
        acc.d[i] = fma(2.0, im, acc.d[i]);
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const int i = q == 2 ? 1 : 0, j = q == 0 ? 1 : 2;
        cd t = acc.o[q];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            cma(t, a.m[i][k], b.m[k][j]);
            // - conj(a_jk b_ki)
            t.re = fma(-a.m[j][k].re, b.m[k][i].re, t.re);
            t.re = fma(a.m[j][k].im, b.m[k][i].im, t.re);
            t.im = fma(a.m[j][k].re, b.m[k][i].im, t.im);
            t.im = fma(a.m[j][k].im, b.m[k][i].re, t.im);
        }
        acc.o[q] = t;
    }
}

// a A + b B
__device__ __forceinline__ ah3 ah_axpy(double a, const ah3 &A, double b, const ah3 &B)
{
    ah3 r;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        r.d[i] = fma(a, A.d[i], b * B.d[i]);
        r.o[i] = cd{fma(a, A.o[i].re, b * B.o[i].re), fma(a, A.o[i].im, b * B.o[i].im)};
    }
    return r;
}

// c (A - tr A / 3)
__device__ __forceinline__ ah3 ah_traceless(const ah3 &a, double c)
{
    const double tr = (1.0 / 3.0) * (a.d[0] + a.d[1] + a.d[2]);
    ah3 r;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        r.d[i] = c * (a.d[i] - tr);
        r.o[i] = c * a.o[i];
    }
    return r;
}

// tr(A B) of two antihermitian matrices (real)
__device__ __forceinline__ double ah_tr(const ah3 &a, const ah3 &b)
{
    double d = 0.0, o = 0.0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        d = fma(a.d[i], b.d[i], d);
        o = fma(a.o[i].re, b.o[i].re, o);
        o = fma(a.o[i].im, b.o[i].im, o);
    }
    return -fma(2.0, o, d);
}

__device__ __forceinline__ m3 ah_full(const ah3 &a)
{
    m3 r;
#pragma unroll
    for (int i = 0; i < 3; ++i) r.m[i][i] = cd{0.0, a.d[i]};
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const int i = q == 2 ? 1 : 0, j = q == 0 ? 1 : 2;
        r.m[i][j] = a.o[q];
        r.m[j][i] = cd{-a.o[q].re, a.o[q].im};
    }
    return r;
}

// link U_mu(y); with an open time boundary the time links leaving the last
// slice are absent (zero)
__device__ __forceinline__ m3 link_xy(const Geom &g, const LinkField<F64> &U, const int y[4], int mu, bool open)
{
    if (open && mu == 3 && y[3] == g.L[3] - 1) {
        m3 z;
        for (int i = 0; i < 3; ++i)
            for (int j = 0; j < 3; ++j) z.m[i][j] = cd{0.0, 0.0};
        return z;
    }
    int p = (y[0] + y[1] + y[2] + y[3]) & 1;
    return load_link<F64, double>(U, p, mu, cb_index(g, y));
}

__device__ __forceinline__ void shift(const Geom &g, const int x[4], int mu, int d, int y[4])
{
    for (int k = 0; k < 4; ++k) y[k] = x[k];
    y[mu] = (y[mu] + d + g.L[mu]) % g.L[mu];
}

// F_{mu nu}(x) = (Q - Q^dag)/8 made traceless, Q = sum of the four leaves
// around x, each leaf walked mu-direction first; plaq: Re tr of the first
// leaf, the plaquette U_mu(x) U_nu(x+mu) U_mu(x+nu)^dag U_nu(x)^dag.  The sum
// of the leaves stays in its antihermitian form.
__device__ __forceinline__ ah3 field_strength(const Geom &g, const LinkField<F64> &U, const int x[4], int mu, int nu,
                                              bool open, double &plaq)
{
    int xpm[4], xpn[4], xmm[4], xmn[4], a[4], b[4], c[4];
    shift(g, x, mu, +1, xpm);
    shift(g, x, nu, +1, xpn);
    shift(g, x, mu, -1, xmm);
    shift(g, x, nu, -1, xmn);
    shift(g, xmm, nu, +1, a);  // x - mu + nu
    shift(g, xmm, nu, -1, b);  // x - mu - nu
    shift(g, xpm, nu, -1, c);  // x + mu - nu
    const m3 Umx = link_xy(g, U, x, mu, open), Unx = link_xy(g, U, x, nu, open);
    ah3 q = ah_zero();
    {
        const m3 l = mm(Umx, link_xy(g, U, xpm, nu, open)), r = md(mm(Unx, link_xy(g, U, xpn, mu, open)));
        ah_add(q, l, r);
        plaq = 0.0;
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                plaq = fma(l.m[i][k].re, r.m[k][i].re, plaq);
                plaq = fma(-l.m[i][k].im, r.m[k][i].im, plaq);
            }
    }
    const m3 Umm = link_xy(g, U, xmm, mu, open), Unn = link_xy(g, U, xmn, nu, open);
    ah_add(q, mm(Unx, md(link_xy(g, U, a, mu, open))), mm(md(link_xy(g, U, xmm, nu, open)), Umm));
    ah_add(q, mm(md(Umm), md(link_xy(g, U, b, nu, open))), mm(link_xy(g, U, b, mu, open), Unn));
    ah_add(q, mm(md(Unn), link_xy(g, U, xmn, mu, open)), mm(link_xy(g, U, c, nu, open), md(Umx)));
    return ah_traceless(q, 0.125);
}

// Per-slice sums in a fixed order: every block writes its chunk's sum, the
// last block of slice t to arrive adds the chunks in order and writes
// corr[(t - src_t) mod T].  counter[t] is zero between uses.
__device__ __forceinline__ void slice_finish(double v, int t, int c, int nchunk, int T, int src_t, double *partial,
                                             unsigned *counter, double *corr)
{
    __shared__ double sh[32];
    __shared__ int last;
    double s = block_sum(v, sh);
    if (threadIdx.x == 0) {
        partial[(long)t * nchunk + c] = s;
        __threadfence();
        last = atomicAdd(&counter[t], 1u) == unsigned(nchunk - 1);
    }
    __syncthreads();
    if (last) {
        __threadfence();
        double a = 0.0;
        for (int k = threadIdx.x; k < nchunk; k += blockDim.x) a += __ldcg(partial + (long)t * nchunk + k);
        a = block_sum(a, sh);
        if (threadIdx.x == 0) {
            counter[t] = 0;
            corr[((t - src_t) % T + T) % T] = a;
        }
    }
}

}  // namespace lqcd
