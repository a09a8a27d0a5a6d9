// Gauge observables and the Wilson flow (Sec. 3.2) on the resident FP64
// links of a gauge field.  One thread per link (flow) or per site
// (observables); FP64 throughout.
//
// Flow generator (the force of the Wilson action summed over oriented
// plaquettes): Z_mu(x) = -(1/2)(Omega - Omega^dag) + (1/6) tr(Omega - Omega^dag)
// with Omega = U_mu(x) S_mu(x), S_mu(x) the sum of the six staples that close
// the plaquettes through the link.  Third-order Runge-Kutta (wfl_rk3) in
// low-storage form, X accumulating the stage combinations:
//   X = eps Z(W0) / 4;               W1 = exp(X) W0
//   X = 8 eps Z(W1) / 9 - 17 X / 9;  W2 = exp(X) W1
//   X = 3 eps Z(W2) / 4 - X;         W3 = exp(X) W2
// (the stage exponents 8 Z1/9 - 17 Z0/36 and 3 Z2/4 - 8 Z1/9 + 17 Z0/36).
#include "gauge_dev.cuh"
#include "lqcd_impl.h"

namespace lqcd {

__device__ __forceinline__ m3 load_m3(const double2 *base, long stride, long cb)
{
    m3 r;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const double2 w = base[k * stride + cb];
        r.m[k / 3][k % 3] = cd{w.x, w.y};
    }
    return r;
}

__device__ __forceinline__ void store_m3(double2 *base, long stride, long cb, const m3 &m)
{
#pragma unroll
    for (int k = 0; k < 9; ++k) base[k * stride + cb] = make_double2(m.m[k / 3][k % 3].re, m.m[k / 3][k % 3].im);
}

// The antihermitian part of a stored matrix (fields that are antihermitian by
// construction: the flow's accumulator X, the HMC momenta)
__device__ __forceinline__ ah3 load_ah(const double2 *base, long stride, long cb)
{
    ah3 r;
#pragma unroll
    for (int i = 0; i < 3; ++i) r.d[i] = base[4 * i * stride + cb].y;
    const double2 a = base[stride + cb], b = base[2 * stride + cb], c = base[5 * stride + cb];
    r.o[0] = cd{a.x, a.y};
    r.o[1] = cd{b.x, b.y};
    r.o[2] = cd{c.x, c.y};
    return r;
}

// exp(s X) for antihermitian traceless X, as q0 + q1 Y + q2 Y^2 with Y = s X /
// 2^k (Cayley-Hamilton: Y^3 = c1 Y + i c0 with c1 = tr Y^2 / 2 and i c0 =
// det Y, both from Y and Y^2).  The three coefficients come from the Horner
// form of the degree-20 Taylor polynomial, P <- 1/n! + Y P, which costs four
// real operations a step instead of a 3x3 product, and up to four squarings act on
// the coefficients too; the rest, for |s X| above 8, square the matrix: the
// coefficients of large powers are themselves large where eigenvalues nearly
// meet, and their rounding grows as |s X|^2 (1e-11 at 1000, 1e-13 by matrices).
// k is chosen so that |Y|_F <= 1/2, where the terms left out are below 1e-25.  About 200 FP64 instructions; a Taylor polynomial
// with 3x3 products took 2900, and 22.4 ms for the links of 32^4 where
// force_gather_kernel now takes 3.6 ms for the whole update.
constexpr int kExpDegree = 20;
__device__ __forceinline__ m3 exp_ah(const ah3 &X, double s)
{
    ah3 Y;
    double n2 = 0.0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        Y.d[i] = s * X.d[i];
        Y.o[i] = s * X.o[i];
        n2 = fma(Y.d[i], Y.d[i], n2);
        n2 = fma(2.0 * Y.o[i].re, Y.o[i].re, n2);
        n2 = fma(2.0 * Y.o[i].im, Y.o[i].im, n2);
    }
    int k = 0;
    double sc = 1.0;
    while (n2 > 0.25 && k < 60) {
        n2 *= 0.25;
        sc *= 0.5;
        ++k;
    }
    if (k > 0) {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            Y.d[i] *= sc;
            Y.o[i] = sc * Y.o[i];
        }
    }
    // H = Y^2 (Hermitian): with Y = (i d0, a, b; -a*, i d1, c; -b*, -c*, i d2)
    const cd a = Y.o[0], b = Y.o[1], c = Y.o[2];
    const double na = fma(a.re, a.re, a.im * a.im), nb = fma(b.re, b.re, b.im * b.im), nc = fma(c.re, c.re, c.im * c.im);
    const double h0 = -fma(Y.d[0], Y.d[0], na + nb), h1 = -fma(Y.d[1], Y.d[1], na + nc),
                 h2 = -fma(Y.d[2], Y.d[2], nb + nc);
    // H01 = i (d0 + d1) a - b c*, H02 = i (d0 + d2) b + a c, H12 = i (d1 + d2) c - a* b
    const double s01 = Y.d[0] + Y.d[1], s02 = Y.d[0] + Y.d[2], s12 = Y.d[1] + Y.d[2];
    cd ha = cd{-s01 * a.im, s01 * a.re}, hb = cd{-s02 * b.im, s02 * b.re}, hc = cd{-s12 * c.im, s12 * c.re};
    cma(ha, cd{-b.re, -b.im}, cd{c.re, -c.im});
    cma(hb, a, c);
    cma(hc, cd{-a.re, a.im}, b);
    const double c1 = 0.5 * (h0 + h1 + h2);
    // i c0 = tr(Y^3) / 3: tr(H Y) = i (sum_i h_i d_i + 2 sum_(i<j) Im(H_ij* Y_ij))
    double im = 0.0;
    im = fma(ha.re, a.im, im);
    im = fma(-ha.im, a.re, im);
    im = fma(hb.re, b.im, im);
    im = fma(-hb.im, b.re, im);
    im = fma(hc.re, c.im, im);
    im = fma(-hc.im, c.re, im);
    const double c0 = (1.0 / 3.0) * fma(h0, Y.d[0], fma(h1, Y.d[1], fma(h2, Y.d[2], 2.0 * im)));
    // Horner: (q0, q1, q2) <- (1/n! + i c0 q2, q0 + c1 q2, q1)
    double f[kExpDegree + 1];
    f[0] = 1.0;
#pragma unroll
    for (int n = 1; n <= kExpDegree; ++n) f[n] = f[n - 1] / n;
    cd q0 = cd{f[kExpDegree], 0.0}, q1 = cd{0.0, 0.0}, q2 = cd{0.0, 0.0};
#pragma unroll
    for (int n = kExpDegree - 1; n >= 0; --n) {
        const cd t0 = cd{fma(-c0, q2.im, f[n]), c0 * q2.re};
        const cd t1 = cd{fma(c1, q2.re, q0.re), fma(c1, q2.im, q0.im)};
        q2 = q1;
        q1 = t1;
        q0 = t0;
    }
    // squarings: Y^3 = c1 Y + i c0, Y^4 = c1 Y^2 + i c0 Y
    const int kc = min(k, 4);
    for (int n = 0; n < kc; ++n) {
        const cd p12 = 2.0 * cm0(q1, q2), p22 = cm0(q2, q2);
        cd t0 = cd{-c0 * p12.im, c0 * p12.re};
        cma(t0, q0, q0);
        cd t1 = cd{fma(c1, p12.re, -c0 * p22.im), fma(c1, p12.im, c0 * p22.re)};
        cma(t1, 2.0 * q0, q1);
        cd t2 = c1 * p22;
        cma(t2, q1, q1);
        cma(t2, 2.0 * q0, q2);
        q0 = t0;
        q1 = t1;
        q2 = t2;
    }
    m3 E;
    const double h[3] = {h0, h1, h2};
    const cd hh[3] = {ha, hb, hc};
#pragma unroll
    for (int i = 0; i < 3; ++i)
        E.m[i][i] = cd{fma(q2.re, h[i], fma(-q1.im, Y.d[i], q0.re)), fma(q2.im, h[i], fma(q1.re, Y.d[i], q0.im))};
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        const int i = e == 2 ? 1 : 0, j = e == 0 ? 1 : 2;
        cd u = cm0(q1, Y.o[e]);
        cma(u, q2, hh[e]);
        E.m[i][j] = u;
        cd l = cm0(q1, cd{-Y.o[e].re, Y.o[e].im});
        cma(l, q2, cd{hh[e].re, -hh[e].im});
        E.m[j][i] = l;
    }
    for (int n = kc; n < k; ++n) E = mm(E, E);
    return E;
}

__device__ __forceinline__ ah3 ah_sum(const ah3 &a, double s, const ah3 &b)
{
    return ah_axpy(1.0, a, s, b);
}

// ---------------------------------------------------------------------------
// Links and force.  Every plaquette P = B1 B2^dag with B1 = U_mu(x) U_nu(x+mu)
// and B2 = U_nu(x) U_mu(x+nu) serves four links: the two at x take P - P^dag
// (with opposite signs), and B1^dag U_nu(x), B2^dag U_mu(x) are the lower
// staples of U_mu(x+nu) and U_nu(x+mu).  One thread per (site, plane) forms
// them once (6 planes x 522 FP64 instructions a site), and one thread per link
// adds its three upper and three lower terms (about 200 with the link's
// product): 3900 instructions a site against 5700 for the six staples of each
// link formed separately.  The kernels are bound by the FP64 pipe (89% busy),
// so the instructions decide: on 32^4 plaquette_kernel takes 5.5 ms and
// force_gather_kernel, which also updates the link, 3.6 ms, where the staples
// per link and the update took 15.4 and 22.4 ms (six instructions per complex
// product, the exponential by 3x3 products).  It costs scratch (FlowScratch,
// 2160 bytes a site); where the device has no room for that (FlowWork),
// flow_force_kernel forms both terms per link (12.2 ms, and 2.3 ms for the
// update), with the same bits.
// ---------------------------------------------------------------------------
struct FlowScratch {
    double2 *low = nullptr;  // lower staples [parity][mu][slot of nu][9 planes]
    double *up = nullptr;    // P - P^dag [parity][plane][9 planes]: diagonal (imaginary), then the 3 upper entries
    static size_t low_bytes(long stride) { return sizeof(double2) * 2 * 4 * 3 * 9 * (size_t)stride; }
    static size_t up_bytes(long stride) { return sizeof(double) * 2 * 6 * 9 * (size_t)stride; }
};

// planes (0,1) (0,2) (0,3) (1,2) (1,3) (2,3)
__device__ __forceinline__ int plane_of(int mu, int nu)  // mu < nu
{
    return mu == 0 ? nu - 1 : (mu == 1 ? nu + 1 : 5);
}

__global__ void __launch_bounds__(128) plaquette_kernel(Geom g, LinkField<F64> U, double2 *low, double *up)
{
    const int cb = blockIdx.x * blockDim.x + threadIdx.x;
    const int p = blockIdx.y, plane = blockIdx.z;
    if (cb >= g.vh) return;
    const int mu = plane < 3 ? 0 : (plane < 5 ? 1 : 2), nu = plane < 3 ? plane + 1 : (plane < 5 ? plane - 1 : 3);
    int x[4];
    cb_coords(g, p, cb, x);
    const int ym = cb_neighbour(g, x, mu, +1), yn = cb_neighbour(g, x, nu, +1);
    const m3 Um = load_link<F64, double>(U, p, mu, cb), Un = load_link<F64, double>(U, p, nu, cb);
    const m3 B1 = mm(Um, load_link<F64, double>(U, p ^ 1, nu, ym));
    const m3 B2 = md(mm(Un, load_link<F64, double>(U, p ^ 1, mu, yn)));
    ah3 w = ah_zero();
    ah_add(w, B1, B2);
    double *u = up + (long)(p * 6 + plane) * 9 * g.stride + cb;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        u[i * g.stride] = w.d[i];
        u[(3 + 2 * i) * g.stride] = w.o[i].re;
        u[(4 + 2 * i) * g.stride] = w.o[i].im;
    }
    // slot of direction b among the three others of a: b < a ? b : b - 1
    store_m3(low + (long)(((p ^ 1) * 4 + mu) * 3 + nu - 1) * 9 * g.stride, g.stride, yn, mm(md(B1), Un));
    store_m3(low + (long)(((p ^ 1) * 4 + nu) * 3 + mu) * 9 * g.stride, g.stride, ym, mm(B2, Um));
}

// X <- a Z + b X, and the link U <- exp(s X) U when s != 0, for the
// antihermitian om = Omega - Omega^dag (Z = -om / 2 without its trace)
__device__ __forceinline__ void force_finish(const ah3 &om, const m3 &u, double2 *X, double2 *ub, long stride, long cb,
                                             double a, double b, double s)
{
    ah3 x = ah_traceless(om, -0.5 * a);
    if (b != 0.0) x = ah_sum(x, b, load_ah(X, stride, cb));
    store_m3(X, stride, cb, ah_full(x));
    if (s != 0.0) store_m3(ub, stride, cb, mm(exp_ah(x, s), u));
}

__global__ void __launch_bounds__(128) force_gather_kernel(Geom g, double2 *u64, const double2 *low, const double *up,
                                                           double2 *X, double a, double b, double s)
{
    const long cb = long(blockIdx.x) * blockDim.x + threadIdx.x;
    const int p = blockIdx.y, mu = blockIdx.z;
    if (cb >= g.vh) return;
    const long q = p * 4 + mu;
    m3 S = load_m3(low + q * 27 * g.stride, g.stride, cb);
#pragma unroll
    for (int n = 1; n < 3; ++n) {
        const m3 t = load_m3(low + (q * 3 + n) * 9 * g.stride, g.stride, cb);
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) S.m[i][j] = S.m[i][j] + t.m[i][j];
    }
    double2 *ub = u64 + q * 9 * g.stride;
    const m3 u = load_m3(ub, g.stride, cb);
    ah3 om = ah_zero();
    ah_add(om, u, S);
#pragma unroll
    for (int n = 0; n < 3; ++n) {
        const int nu = n < mu ? n : n + 1;
        const double sg = nu > mu ? 1.0 : -1.0;
        const double *w = up + (long)(p * 6 + (nu > mu ? plane_of(mu, nu) : plane_of(nu, mu))) * 9 * g.stride + cb;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            om.d[i] = fma(sg, w[i * g.stride], om.d[i]);
            om.o[i].re = fma(sg, w[(3 + 2 * i) * g.stride], om.o[i].re);
            om.o[i].im = fma(sg, w[(4 + 2 * i) * g.stride], om.o[i].im);
        }
    }
    force_finish(om, u, X + q * 9 * g.stride, ub, g.stride, cb, a, b, s);
}

// X_mu(x) = a Z_mu(x) + b X_mu(x) for every link (b = 0: X not read), the
// terms formed here: no scratch.  Products and sums are those of
// plaquette_kernel and force_gather_kernel, in their order, so that the links
// do not depend on how much memory was free (12.2 ms on 32^4; 10.7 for the
// staples of the link, whose result differs by rounding).
__global__ void __launch_bounds__(64) flow_force_kernel(Geom g, LinkField<F64> U, double2 *X, double a, double b)
{
    const long cb = long(blockIdx.x) * blockDim.x + threadIdx.x;
    const int p = blockIdx.y, mu = blockIdx.z;
    if (cb >= g.vh) return;
    int x[4];
    cb_coords(g, p, int(cb), x);
    m3 S;
#pragma unroll
    for (int n = 0; n < 3; ++n) {  // lower staples, from the plaquettes at x - nu
        const int nu = n < mu ? n : n + 1;
        int y[4], ym[4];
        shift(g, x, nu, -1, y);
        shift(g, y, mu, +1, ym);
        const m3 t = mm(md(mm(link_xy(g, U, y, mu, false), link_xy(g, U, ym, nu, false))), link_xy(g, U, y, nu, false));
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) S.m[i][j] = n == 0 ? t.m[i][j] : S.m[i][j] + t.m[i][j];
    }
    const m3 u = link_xy(g, U, x, mu, false);
    ah3 om = ah_zero();
    ah_add(om, u, S);
#pragma unroll
    for (int n = 0; n < 3; ++n) {  // P - P^dag of the plaquettes at x
        const int nu = n < mu ? n : n + 1, c = min(mu, nu), d = max(mu, nu);
        int xc[4], xd[4];
        shift(g, x, c, +1, xc);
        shift(g, x, d, +1, xd);
        ah3 w = ah_zero();
        ah_add(w, mm(link_xy(g, U, x, c, false), link_xy(g, U, xc, d, false)),
               md(mm(link_xy(g, U, x, d, false), link_xy(g, U, xd, c, false))));
        const double sg = nu > mu ? 1.0 : -1.0;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            om.d[i] = fma(sg, w.d[i], om.d[i]);
            om.o[i].re = fma(sg, w.o[i].re, om.o[i].re);
            om.o[i].im = fma(sg, w.o[i].im, om.o[i].im);
        }
    }
    force_finish(om, u, X + (long)(p * 4 + mu) * 9 * g.stride, nullptr, g.stride, cb, a, b, 0.0);
}

// U_mu(x) <- exp(s X_mu(x)) U_mu(x)
__global__ void __launch_bounds__(128) flow_update_kernel(Geom g, double2 *u64, const double2 *X, double s)
{
    const long cb = long(blockIdx.x) * blockDim.x + threadIdx.x;
    const int p = blockIdx.y, mu = blockIdx.z;
    if (cb >= g.vh) return;
    double2 *ub = u64 + (long)(p * 4 + mu) * 9 * g.stride;
    const ah3 x = load_ah(X + (long)(p * 4 + mu) * 9 * g.stride, g.stride, cb);
    store_m3(ub, g.stride, cb, mm(exp_ah(x, s), load_m3(ub, g.stride, cb)));
}

// HMC momenta: P_mu(x) = sum_a pi_a i lambda_a / 2 from the caller's
// coordinates pi (host layout [site][mu][8], on the device)
__global__ void __launch_bounds__(128) momenta_kernel(Geom g, long V, const double *pi, double2 *P)
{
    const long s = long(blockIdx.x) * blockDim.x + threadIdx.x;
    if (s >= V) return;
    long r = s;
    int x[4];
    x[0] = int(r % g.L[0]);
    r /= g.L[0];
    x[1] = int(r % g.L[1]);
    r /= g.L[1];
    x[2] = int(r % g.L[2]);
    x[3] = int(r / g.L[2]);
    const int p = (x[0] + x[1] + x[2] + x[3]) & 1;
    const long cb = s >> 1;
    const double r3 = 0.57735026918962576451;  // 1 / sqrt 3
    for (int mu = 0; mu < 4; ++mu) {
        const double *a = pi + (s * 4 + mu) * 8;
        m3 M;
        // i lambda_1..8 / 2 weighted by a[0..7]
        M.m[0][0] = cd{0.0, 0.5 * (a[2] + r3 * a[7])};
        M.m[1][1] = cd{0.0, 0.5 * (-a[2] + r3 * a[7])};
        M.m[2][2] = cd{0.0, -r3 * a[7]};
        M.m[0][1] = cd{0.5 * a[1], 0.5 * a[0]};
        M.m[1][0] = cd{-0.5 * a[1], 0.5 * a[0]};
        M.m[0][2] = cd{0.5 * a[4], 0.5 * a[3]};
        M.m[2][0] = cd{-0.5 * a[4], 0.5 * a[3]};
        M.m[1][2] = cd{0.5 * a[6], 0.5 * a[5]};
        M.m[2][1] = cd{-0.5 * a[6], 0.5 * a[5]};
        store_m3(P + (long)(p * 4 + mu) * 9 * g.stride, g.stride, cb, M);
    }
}

// partial[block] = sum over the block's links of -tr P^2 (one thread per link)
__global__ void __launch_bounds__(128) kinetic_kernel(Geom g, const double2 *P, double *partial)
{
    __shared__ double sh[32];
    const long cb = long(blockIdx.x) * blockDim.x + threadIdx.x;
    const int q = blockIdx.y;  // parity * 4 + mu
    double v = 0.0;
    if (cb < g.vh) {
        const m3 M = load_m3(P + (long)q * 9 * g.stride, g.stride, cb);
        const m3 MM = mm(M, M);
        v = -(MM.m[0][0].re + MM.m[1][1].re + MM.m[2][2].re);
    }
    v = block_sum(v, sh);
    if (threadIdx.x == 0) partial[(long)q * gridDim.x + blockIdx.x] = v;
}

// out[0] = sum of the n partials in a fixed order (one block)
__global__ void __launch_bounds__(512) sum_partials_kernel(const double *partial, long n, double *out)
{
    __shared__ double sh[32];
    double t = 0.0;
    for (long k = threadIdx.x; k < n; k += blockDim.x) t += partial[k];
    t = block_sum(t, sh);
    if (threadIdx.x == 0) out[0] = t;
}

// FP32 / FP16 reconstruct-12 copies from the FP64 links (after the flow)
__global__ void __launch_bounds__(128) recon_copies_kernel(Geom g, const double2 *u64, float4 *u32, uint4 *u16,
                                                           uint2 *u16b)
{
    const long cb = long(blockIdx.x) * blockDim.x + threadIdx.x;
    const int q = blockIdx.y;  // parity * 4 + mu
    if (cb >= g.vh) return;
    double m[18];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const double2 w = u64[((long)q * 9 + k) * g.stride + cb];
        m[2 * k] = w.x;
        m[2 * k + 1] = w.y;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k)
        u32[((long)q * 3 + k) * g.stride + cb] =
            make_float4(float(m[4 * k]), float(m[4 * k + 1]), float(m[4 * k + 2]), float(m[4 * k + 3]));
    uint4 w;
    __half2 *h = reinterpret_cast<__half2 *>(&w);
#pragma unroll
    for (int k = 0; k < 4; ++k) h[k] = __floats2half2_rn(float(m[2 * k]), float(m[2 * k + 1]));
    u16[(long)q * g.stride + cb] = w;
    uint2 w2;
    __half2 *h2 = reinterpret_cast<__half2 *>(&w2);
#pragma unroll
    for (int k = 0; k < 2; ++k) h2[k] = __floats2half2_rn(float(m[8 + 2 * k]), float(m[9 + 2 * k]));
    u16b[(long)q * g.stride + cb] = w2;
}

// Gauge observables per time slice (Sec. 3.2; plaquette, Eoft_plaq,
// Eoft_clover, Qtop): thread = site of slice t (lexicographic within the
// slice), sums over the slice by slice_finish into
//   out[0 T + t]: sum Re tr U_p / 3 over the 6 planes,
//   out[1 T + t]: 2 sum_{mu<nu} Re tr (1 - U_p)            (plaquette action density),
//   out[2 T + t]: - sum_{mu<nu} tr F_{mu nu}^2              (clover action density),
//   out[3 T + t]: -(8 / 32 pi^2) [tr F_xy F_zt - tr F_xz F_yt + tr F_xt F_yz]  (clover charge density).
__global__ void __launch_bounds__(128) gauge_obs_kernel(Geom g, LinkField<F64> U, double *partial,
                                                        unsigned *counter, double *out)
{
    const int t = blockIdx.y, c = blockIdx.x, nchunk = gridDim.x;
    const int T = g.L[3];
    const long v3 = long(g.L[0]) * g.L[1] * g.L[2];
    const long k = long(c) * blockDim.x + threadIdx.x;
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    if (k < v3) {
        int x[4];
        long r = k;
        x[0] = int(r % g.L[0]);
        r /= g.L[0];
        x[1] = int(r % g.L[1]);
        x[2] = int(r / g.L[1]);
        x[3] = t;
        ah3 F[6];
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            const int mu = q < 3 ? 0 : (q < 5 ? 1 : 2), nu = q < 3 ? q + 1 : (q < 5 ? q - 1 : 3);
            double re;
            F[q] = field_strength(g, U, x, mu, nu, false, re);
            v[0] += re / 3.0;
            v[1] += 2.0 * (3.0 - re);
            v[2] -= ah_tr(F[q], F[q]);
        }
        const double e = ah_tr(F[0], F[5]) - ah_tr(F[1], F[4]) + ah_tr(F[2], F[3]);
        v[3] = -8.0 * e / (32.0 * 3.14159265358979323846 * 3.14159265358979323846);
    }
    for (int o = 0; o < 4; ++o)
        slice_finish(v[o], t, c, nchunk, T, 0, partial + (long)o * T * nchunk, counter + o * T, out + o * T);
}

// host layout U[site][mu][3][3] from the FP64 SoA links
__global__ void __launch_bounds__(128) gauge_unpack_kernel(Geom g, long V, const double2 *u64, double *U)
{
    const long s = long(blockIdx.x) * blockDim.x + threadIdx.x;
    if (s >= V) return;
    long r = s;
    int x[4];
    x[0] = int(r % g.L[0]);
    r /= g.L[0];
    x[1] = int(r % g.L[1]);
    r /= g.L[1];
    x[2] = int(r % g.L[2]);
    x[3] = int(r / g.L[2]);
    const int p = (x[0] + x[1] + x[2] + x[3]) & 1;
    const long cb = s >> 1;
    for (int mu = 0; mu < 4; ++mu) {
        double *m = U + (s * 4 + mu) * 18;
        for (int k = 0; k < 9; ++k) {
            const double2 w = u64[((long)(p * 4 + mu) * 9 + k) * g.stride + cb];
            m[2 * k] = w.x;
            m[2 * k + 1] = w.y;
        }
    }
}

// scratch of the shared-plaquette force for one call; empty (both pointers
// null) when the device has no room for it, or when it would take more than
// half of what is free: other threads and processes allocate meanwhile, and the
// scratch is a convenience.  Up to kSmallScratch that is not looked at (the
// query takes 4 us, a flow step on 4^4 150).
constexpr size_t kSmallScratch = size_t(64) << 20;
struct FlowWork {
    DevBuf low, up;
    FlowScratch s;
    explicit FlowWork(long stride)
    {
        const size_t need = FlowScratch::low_bytes(stride) + FlowScratch::up_bytes(stride);
        if (need > kSmallScratch) {
            size_t free_b = 0, total_b = 0;
            LQCD_CUDA(cudaMemGetInfo(&free_b, &total_b));
            if (need > free_b / 2) return;
        }
        try {
            low.ensure(FlowScratch::low_bytes(stride));
            up.ensure(FlowScratch::up_bytes(stride));
            s = FlowScratch{low.as<double2>(), up.as<double>()};
        } catch (const Error &e) {
            if (e.code != LQCD_ENOMEM) throw;
            cudaGetLastError();  // the failed allocation is not an error of the call
            low.release();
            up.release();
        }
    }
};

// X <- a Z(u) + b X, then u <- exp(s X) u (s = 0: the force only)
static void force_step(lqcd_lattice_s *lat, double2 *u, double2 *X, const FlowScratch &w, double a, double b, double s,
                       const char *force_name, const char *update_name, cudaStream_t st)
{
    const long S = lat->stride;
    const LinkField<F64> U{u, nullptr, S};
    const unsigned nb = unsigned((lat->vh + 127) / 128);
    if (w.low) {
        {
            // reads the 4 links of a site, writes 12 staples and 6 antihermitian matrices
            ProfScope prof(force_name, double(lat->V) * (4 * 144.0 + 12 * 144.0 + 6 * 72.0), st);
            plaquette_kernel<<<dim3(nb, 2, 6), 128, 0, st>>>(lat->geom, U, w.low, w.up);
            LQCD_CHECK_LAUNCH();
        }
        ProfScope prof(update_name, double(lat->V) * 4 * (3 * 144.0 + 3 * 72.0 + 4 * 144.0), st);
        force_gather_kernel<<<dim3(nb, 2, 4), 128, 0, st>>>(lat->geom, u, w.low, w.up, X, a, b, s);
        LQCD_CHECK_LAUNCH();
        return;
    }
    {
        ProfScope prof("force_no_scratch", double(lat->V) * 4 * (7 * 144.0 + 144.0), st);
        flow_force_kernel<<<dim3(unsigned((lat->vh + 63) / 64), 2, 4), 64, 0, st>>>(lat->geom, U, X, a, b);
        LQCD_CHECK_LAUNCH();
    }
    if (s != 0.0) {
        ProfScope prof(update_name, double(lat->V) * 4 * 3 * 144.0, st);
        flow_update_kernel<<<dim3(nb, 2, 4), 128, 0, st>>>(lat->geom, u, X, s);
        LQCD_CHECK_LAUNCH();
    }
}

// one stage of the low-storage RK3 step (W_stage -> W_stage+1) of the links
// u (FP64 planes), X the stage accumulator
static void flow_stage(lqcd_lattice_s *lat, double2 *u, double2 *X, const FlowScratch &w, int stage, double eps,
                       cudaStream_t st)
{
    const double a[3] = {0.25, 8.0 / 9.0, 0.75}, b[3] = {0.0, -17.0 / 9.0, -1.0};
    force_step(lat, u, X, w, a[stage] * eps, b[stage], 1.0, "flow_force", "flow_update", st);
}

// the FP32/FP16 copies of the flowed links; the clover fields of the old links are dropped
static void flow_finish(lqcd_lattice_s *lat, GaugeSet &g, cudaStream_t st)
{
    const dim3 gr(unsigned((lat->vh + 127) / 128), 8);
    recon_copies_kernel<<<gr, 128, 0, st>>>(lat->geom, g.u64.as<const double2>(), g.u32.as<float4>(),
                                            g.u16.as<uint4>(), g.u16b.as<uint2>());
    LQCD_CHECK_LAUNCH();
    LQCD_CUDA(cudaStreamSynchronize(st));  // scratch buffers are freed on return
    g.clover.clear();
    g.sf_ready = false;  // the SF hopping links belong to the old links
}

void gauge_flow(lqcd_lattice_s *lat, GaugeSet &g, double eps, int nsteps, cudaStream_t st)
{
    const long S = lat->stride;
    DevBuf X;
    X.ensure(sizeof(double2) * 2 * 4 * 9 * S);
    const FlowWork w(S);
    for (int k = 0; k < nsteps; ++k)
        for (int stage = 0; stage < 3; ++stage)
            flow_stage(lat, g.u64.as<double2>(), X.as<double2>(), w.s, stage, eps, st);
    flow_finish(lat, g, st);
}

// ---------------------------------------------------------------------------
// Fermion flow: d chi/dt = Delta chi with the covariant Laplacian
//   (Delta chi)(x) = sum_mu [U~_mu(x) chi(x+mu) + U~_mu(x-mu)^dag chi(x-mu) - 2 chi(x)]
// (colour only; U~ carries the boundary phases theta), the links flowed
// alongside.  Third-order scheme on the gauge stages W0, W1, W2 of a step:
//   lambda1 = chi + eps/4 Delta(W0) chi
//   lambda2 = chi + 8 eps/9 Delta(W1) lambda1 - 2 eps/9 Delta(W0) chi
//   chi'    = lambda1 + 3 eps/4 Delta(W2) lambda2
// With Delta(W0) chi = 4 (lambda1 - chi) / eps and H the hopping sum this is
//   lambda1 = eps/4 H chi + (1 - 2 eps) chi
//   lambda2 = 8 eps/9 H lambda1 - 8/9 (1 + 8 eps) lambda1 + 17/9 chi
//   chi'    = 3 eps/4 H lambda2 - 6 eps lambda2 + lambda1
// so each stage is one pass per parity of
//   out(x) = cH H in (x) + c0 in(x) + c1 a1(x).
// ---------------------------------------------------------------------------
struct Phases {
    double re[4], im[4];
    int mask;  // bit mu set: the phase of direction mu is not 1
};

static Phases phases_of(const lqcd_dirac_params &dp)
{
    Phases th;
    hop_theta(dp, th.re, th.im);
    th.mask = 0;
    for (int mu = 0; mu < 4; ++mu)
        if (th.re[mu] != 1.0 || th.im[mu] != 0.0) th.mask |= 1 << mu;
    return th;
}

// a field by its two parity halves
struct Halves {
    SpinorField<F64> h[2];
};

// acc += W v on the colour index of all four spins, W = U or U^dag, with the
// boundary phase applied to v where the hop wraps: 144 FP64 instructions (the
// sums run inside the products' fma chains)
template <bool DAG>
__device__ __forceinline__ void colour_hop(spinor<double> &acc, const su3<double> &u, spinor<double> v, bool wrap,
                                           double ph_re, double ph_im)
{
    if (wrap) {
#pragma unroll
        for (int s = 0; s < 4; ++s)
#pragma unroll
            for (int a = 0; a < 3; ++a) v.s[s][a] = cm0(cd{ph_re, ph_im}, v.s[s][a]);
    }
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b)
                cma(acc.s[s][a], DAG ? cd{u.m[b][a].re, -u.m[b][a].im} : u.m[a][b], v.s[s][b]);
}

// One thread per (site, right-hand side), both parities in one launch
// (blockIdx.y).  Bound by the FP64 pipe: 1152 instructions for the eight hops
// and 24 to 72 for the sums with in, a1 and a2; phases cost only where a hop
// wraps under a phase other than 1.  3.14 ms for twelve fields on 16^3 x 32,
// against 6.2 ms with separate products and sums and a phase on every hop.
__global__ void __launch_bounds__(128) laplace_kernel(Geom g, LinkField<F64> U, Phases th, Halves in, Halves a1,
                                                      Halves a2, Halves out, int nrhs, double cH, double c0, double c1,
                                                      double c2)
{
    const int p = blockIdx.y;
    const int j = blockIdx.x % nrhs, tile = blockIdx.x / nrhs;
    const int cb = tile * blockDim.x + threadIdx.x;
    if (cb >= g.vh) return;
    int x[4];
    cb_coords(g, p, cb, x);
    const SpinorField<F64> other = p ? in.h[0] : in.h[1];
    spinor<double> acc;
    zero(acc);
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
        const bool ph = (th.mask >> mu) & 1;
        int y = cb_neighbour(g, x, mu, +1);
        colour_hop<false>(acc, load_link<F64, double>(U, p, mu, cb), load_spinor<F64, double>(other, j, y),
                          ph && x[mu] == g.L[mu] - 1, th.re[mu], th.im[mu]);
        y = cb_neighbour(g, x, mu, -1);
        colour_hop<true>(acc, load_link<F64, double>(U, p ^ 1, mu, y), load_spinor<F64, double>(other, j, y),
                         ph && x[mu] == 0, th.re[mu], -th.im[mu]);
    }
    const SpinorField<F64> self = in.h[p], s1 = a1.h[p], s2 = a2.h[p];
    const spinor<double> sv = load_spinor<F64, double>(self, j, cb);
    spinor<double> res;
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int a = 0; a < 3; ++a) res.s[s][a] = cd{fma(cH, acc.s[s][a].re, c0 * sv.s[s][a].re),
                                                     fma(cH, acc.s[s][a].im, c0 * sv.s[s][a].im)};
    if (s1.p) {
        const spinor<double> av = load_spinor<F64, double>(s1, j, cb);
#pragma unroll
        for (int s = 0; s < 4; ++s)
#pragma unroll
            for (int a = 0; a < 3; ++a) res.s[s][a] = cd{fma(c1, av.s[s][a].re, res.s[s][a].re),
                                                         fma(c1, av.s[s][a].im, res.s[s][a].im)};
    }
    if (s2.p) {
        const spinor<double> av = load_spinor<F64, double>(s2, j, cb);
#pragma unroll
        for (int s = 0; s < 4; ++s)
#pragma unroll
            for (int a = 0; a < 3; ++a) res.s[s][a] = cd{fma(c2, av.s[s][a].re, res.s[s][a].re),
                                                         fma(c2, av.s[s][a].im, res.s[s][a].im)};
    }
    double2 *o = out.h[p].p + (long)j * 12 * out.h[p].stride + cb;
#pragma unroll
    for (int k = 0; k < 12; ++k) o[k * out.h[p].stride] = make_double2(res.s[k / 3][k % 3].re, res.s[k / 3][k % 3].im);
}

// backflow combination: u = eta + z1; w = a u - c z2 (one parity, every RHS)
__global__ void __launch_bounds__(128) backflow_combine_kernel(long vh, int nrhs, SpinorField<F64> eta,
                                                               SpinorField<F64> z1, SpinorField<F64> z2,
                                                               SpinorField<F64> u, SpinorField<F64> w, double a,
                                                               double c)
{
    const int j = blockIdx.x % nrhs, tile = blockIdx.x / nrhs;
    const int cb = tile * blockDim.x + threadIdx.x;
    if (cb >= vh) return;
    const spinor<double> e = load_spinor<F64, double>(eta, j, cb), p1 = load_spinor<F64, double>(z1, j, cb),
                         p2 = load_spinor<F64, double>(z2, j, cb);
    spinor<double> uu, ww;
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            uu.s[s][k] = e.s[s][k] + p1.s[s][k];
            ww.s[s][k] = a * uu.s[s][k] - c * p2.s[s][k];
        }
    store_spinor<F64, double>(u, j, cb, uu);
    store_spinor<F64, double>(w, j, cb, ww);
}

namespace {
// a full-lattice FP64 field: even and odd halves of nrhs right-hand sides
struct Full {
    SpinorField<F64> e, o;
    const SpinorField<F64> &half(int p) const { return p ? o : e; }
    Halves halves() const { return Halves{{e, o}}; }
};

Full full_of(DevBuf &b, long stride, int nrhs)
{
    double2 *p = b.as<double2>();
    const long half = (long)12 * stride * nrhs;
    return Full{SpinorField<F64>{p, nullptr, stride}, SpinorField<F64>{p + half, nullptr, stride}};
}
}  // namespace

// out = cH H in + c0 in + c1 a1 + c2 a2 on both parities (in != out; a1, a2 may be null)
static void laplace_stage(lqcd_lattice_s *lat, const LinkField<F64> &U, const Phases &th, const Full &in,
                          const Full *a1, const Full &out, int nrhs, double cH, double c0, double c1, cudaStream_t st,
                          const Full *a2 = nullptr, double c2 = 0.0)
{
    // per output site and RHS: the spinor at 8 neighbours and itself (+ a1, a2), the output; 8 links per site
    const double bytes = double(lat->V) * (nrhs * 192.0 * (2.0 + (a1 ? 1.0 : 0.0) + (a2 ? 1.0 : 0.0)) + 8 * 144.0);
    ProfScope prof("fermion_flow_laplace", bytes, st);
    laplace_kernel<<<dim3(unsigned(ntiles_of(lat->vh) * nrhs), 2), kBlock, 0, st>>>(
        lat->geom, U, th, in.halves(), a1 ? a1->halves() : Halves{}, a2 ? a2->halves() : Halves{}, out.halves(), nrhs,
        cH, c0, c1, c2);
    LQCD_CHECK_LAUNCH();
}

void fermion_flow(lqcd_lattice_s *lat, GaugeSet &g, const lqcd_dirac_params &dp, double *psi_dev, int nrhs,
                  double eps, int nsteps, cudaStream_t st)
{
    const long S = lat->stride;
    const size_t fb = sizeof(double2) * 2 * 12 * (size_t)S * nrhs;
    DevBuf X, bchi, bl1, bl2;
    X.ensure(sizeof(double2) * 2 * 4 * 9 * S);
    bchi.ensure(fb);
    bl1.ensure(fb);
    bl2.ensure(fb);
    const FlowWork fw(S);
    const Full chi = full_of(bchi, S, nrhs), l1 = full_of(bl1, S, nrhs), l2 = full_of(bl2, S, nrhs);
    const Phases th = phases_of(dp);
    const LinkField<F64> U{g.u64.as<const double2>(), nullptr, S};
    spinor_to_soa(lat, psi_dev, nrhs, chi.e, chi.o, st);
    for (int k = 0; k < nsteps; ++k) {
        laplace_stage(lat, U, th, chi, nullptr, l1, nrhs, 0.25 * eps, 1.0 - 2.0 * eps, 0.0, st);  // W0
        flow_stage(lat, g.u64.as<double2>(), X.as<double2>(), fw.s, 0, eps, st);
        laplace_stage(lat, U, th, l1, &chi, l2, nrhs, 8.0 / 9.0 * eps, -8.0 / 9.0 * (1.0 + 8.0 * eps), 17.0 / 9.0,
                      st);  // W1
        flow_stage(lat, g.u64.as<double2>(), X.as<double2>(), fw.s, 1, eps, st);
        laplace_stage(lat, U, th, l2, &l1, chi, nrhs, 0.75 * eps, -6.0 * eps, 1.0, st);  // W2
        flow_stage(lat, g.u64.as<double2>(), X.as<double2>(), fw.s, 2, eps, st);
    }
    spinor_from_soa(lat, psi_dev, nrhs, chi.e, chi.o, st);
    flow_finish(lat, g, st);
}

// S = (beta / 6) sum_t Eplaq[t] from the observables kernel (host value)
static double wilson_action(lqcd_lattice_s *lat, GaugeSet &g, double beta, double *out_dev, cudaStream_t st)
{
    const int T = lat->dims[3];
    gauge_observables(lat, g, out_dev, st);
    std::vector<double> h(T);
    LQCD_CUDA(cudaMemcpyAsync(h.data(), out_dev + T, sizeof(double) * T, cudaMemcpyDeviceToHost, st));
    LQCD_CUDA(cudaStreamSynchronize(st));
    double s = 0.0;
    for (int t = 0; t < T; ++t) s += h[t];
    return beta / 6.0 * s;
}

static double kinetic_energy(lqcd_lattice_s *lat, const double2 *P, double *scratch, cudaStream_t st)
{
    const unsigned nb = unsigned((lat->vh + 127) / 128);
    kinetic_kernel<<<dim3(nb, 8), 128, 0, st>>>(lat->geom, P, scratch);
    LQCD_CHECK_LAUNCH();
    sum_partials_kernel<<<1, 512, 0, st>>>(scratch, long(nb) * 8, scratch + long(nb) * 8);
    LQCD_CHECK_LAUNCH();
    double k = 0.0;
    LQCD_CUDA(cudaMemcpyAsync(&k, scratch + long(nb) * 8, sizeof(double), cudaMemcpyDeviceToHost, st));
    LQCD_CUDA(cudaStreamSynchronize(st));
    return k;
}

int hmc_trajectory(lqcd_lattice_s *lat, GaugeSet &g, double beta, double eps, int nsteps, const double *mom_dev,
                   double u, double *dH, cudaStream_t st)
{
    const long S = lat->stride;
    const int T = lat->dims[3];
    const size_t ubytes = sizeof(double2) * 2 * 4 * 9 * S;
    DevBuf P, backup, scratch;
    P.ensure(ubytes);
    backup.ensure(ubytes);
    const unsigned nb = unsigned((lat->vh + 127) / 128);
    scratch.ensure(sizeof(double) * std::max<size_t>(4 * T, size_t(nb) * 8 + 1));
    double2 *u64 = g.u64.as<double2>();
    LQCD_CUDA(cudaMemcpyAsync(backup.p, u64, ubytes, cudaMemcpyDeviceToDevice, st));
    momenta_kernel<<<unsigned((lat->V + 127) / 128), 128, 0, st>>>(lat->geom, lat->V, mom_dev, P.as<double2>());
    LQCD_CHECK_LAUNCH();
    const double H0 = kinetic_energy(lat, P.as<const double2>(), scratch.as<double>(), st) +
                      wilson_action(lat, g, beta, scratch.as<double>(), st);
    const FlowWork fw(S);
    for (int s = 0; s <= nsteps; ++s) {
        // P += h F(U), F = (beta / 6) Z, then U = exp(eps P) U (not after the last half step)
        const double h = (s == 0 || s == nsteps) ? 0.5 * eps : eps;
        force_step(lat, u64, P.as<double2>(), fw.s, h * beta / 6.0, 1.0, s == nsteps ? 0.0 : eps, "hmc_force",
                   "hmc_links", st);
    }
    const double H1 = kinetic_energy(lat, P.as<const double2>(), scratch.as<double>(), st) +
                      wilson_action(lat, g, beta, scratch.as<double>(), st);
    *dH = H1 - H0;
    const bool acc = u < std::exp(-*dH);
    if (!acc) LQCD_CUDA(cudaMemcpyAsync(u64, backup.p, ubytes, cudaMemcpyDeviceToDevice, st));
    const dim3 gr(unsigned((lat->vh + 127) / 128), 8);
    recon_copies_kernel<<<gr, 128, 0, st>>>(lat->geom, g.u64.as<const double2>(), g.u32.as<float4>(),
                                            g.u16.as<uint4>(), g.u16b.as<uint2>());
    LQCD_CHECK_LAUNCH();
    LQCD_CUDA(cudaStreamSynchronize(st));
    g.clover.clear();
    g.sf_ready = false;  // the SF hopping links belong to the old links
    return acc ? 1 : 0;
}

void gauge_observables(lqcd_lattice_s *lat, GaugeSet &g, double *out_dev, cudaStream_t st)
{
    const int T = lat->dims[3];
    const long v3 = lat->V / T;
    const int nchunk = int((v3 + kBlock - 1) / kBlock);
    lat->red_partial.ensure(sizeof(double) * 4 * (size_t)T * nchunk);
    if (lat->red_counter.bytes < sizeof(unsigned) * (size_t)std::max(4 * T, 4096)) {
        lat->red_counter.ensure(sizeof(unsigned) * (size_t)std::max(4 * T, 4096));
        LQCD_CUDA(cudaMemsetAsync(lat->red_counter.p, 0, lat->red_counter.bytes, st));
    }
    ProfScope prof("gauge_obs", double(lat->V) * 4 * 144.0, st);
    gauge_obs_kernel<<<dim3(nchunk, T), kBlock, 0, st>>>(lat->geom, link_field<F64>(g, lat->stride),
                                                        lat->red_partial.as<double>(),
                                                        lat->red_counter.as<unsigned>(), out_dev);
    LQCD_CHECK_LAUNCH();
}

void gauge_download(lqcd_lattice_s *lat, GaugeSet &g, double *U_dev, cudaStream_t st)
{
    gauge_unpack_kernel<<<unsigned((lat->V + 127) / 128), 128, 0, st>>>(lat->geom, lat->V, g.u64.as<const double2>(),
                                                                        U_dev);
    LQCD_CHECK_LAUNCH();
}

}  // namespace lqcd

namespace lqcd {

// ---------------------------------------------------------------------------
// Fermion backflow: the exact adjoint of the forward steps above, run over the
// steps in reverse order.  One forward step is chi' = M chi with
//   M = (1 + a D0) + d D2 + d b D2 D1 (1 + a D0) - d c D2 D0,
// a = eps/4, b = 8 eps/9, c = 2 eps/9, d = 3 eps/4, Di = Delta(Wi) (Hermitian),
// so one backward step is
//   z2 = d D2 eta,  z1 = b D1 z2,  u = eta + z1,  w = a u - c z2,
//   eta <- u + z2 + D0 w.
// The gauge field at the start of every step is rebuilt from checkpoints:
// a forward pass keeps the field at the start of every m-th step (m =
// ceil(nsteps / nsave)); each segment of m steps is then flowed again from
// its checkpoint, keeping the start field of each of its steps, and walked
// backwards; the stages W1, W2 of a step are recomputed from its start field.
// The resident links are left at flow time 0.
// ---------------------------------------------------------------------------
void fermion_backflow(lqcd_lattice_s *lat, GaugeSet &g, const lqcd_dirac_params &dp, double *eta_dev, int nrhs,
                      double eps, int nsteps, int nsave, cudaStream_t st)
{
    const long S = lat->stride;
    const size_t ub = sizeof(double2) * 2 * 4 * 9 * (size_t)S;  // one gauge field
    const size_t fb = sizeof(double2) * 2 * 12 * (size_t)S * nrhs;
    const int m = nsteps > 0 ? (nsteps + nsave - 1) / nsave : 1;
    const int nck = nsteps > 0 ? (nsteps + m - 1) / m : 0;
    DevBuf X, ck, seg, w1, w2, be, bz1, bz2, bu, bw;
    X.ensure(ub);
    ck.ensure(ub * std::max(nck, 1));
    seg.ensure(ub * m);
    w1.ensure(ub);
    w2.ensure(ub);
    for (DevBuf *b : {&be, &bz1, &bz2, &bu, &bw}) b->ensure(fb);
    const FlowWork fw(S);
    const Full eta = full_of(be, S, nrhs), z1 = full_of(bz1, S, nrhs), z2 = full_of(bz2, S, nrhs),
               u = full_of(bu, S, nrhs), w = full_of(bw, S, nrhs);
    const size_t nlink = ub / sizeof(double2);
    double2 *ckp = ck.as<double2>(), *segp = seg.as<double2>(), *W1 = w1.as<double2>(), *W2 = w2.as<double2>();
    const Phases th = phases_of(dp);
    spinor_to_soa(lat, eta_dev, nrhs, eta.e, eta.o, st);
    // forward pass: checkpoints at the start of steps 0, m, 2m, ... (w1 is the running field)
    LQCD_CUDA(cudaMemcpyAsync(W1, g.u64.p, ub, cudaMemcpyDeviceToDevice, st));
    for (int k = 0; k < nsteps; ++k) {
        if (k % m == 0) LQCD_CUDA(cudaMemcpyAsync(ckp + (k / m) * nlink, W1, ub, cudaMemcpyDeviceToDevice, st));
        if (k + 1 < nsteps)  // the end field of the last step is not needed
            for (int stage = 0; stage < 3; ++stage) flow_stage(lat, W1, X.as<double2>(), fw.s, stage, eps, st);
    }
    const double a = 0.25 * eps, b = 8.0 / 9.0 * eps, c = 2.0 / 9.0 * eps, d = 0.75 * eps;
    const unsigned gvec = unsigned(ntiles_of(lat->vh) * nrhs);
    for (int sgi = nck - 1; sgi >= 0; --sgi) {
        const int k0 = sgi * m, k1 = std::min(nsteps, k0 + m);
        // start fields of the steps k0 .. k1-1 of this segment
        LQCD_CUDA(cudaMemcpyAsync(segp, ckp + sgi * nlink, ub, cudaMemcpyDeviceToDevice, st));
        for (int k = k0 + 1; k < k1; ++k) {
            double2 *dst = segp + (k - k0) * nlink;
            LQCD_CUDA(cudaMemcpyAsync(dst, dst - nlink, ub, cudaMemcpyDeviceToDevice, st));
            for (int stage = 0; stage < 3; ++stage) flow_stage(lat, dst, X.as<double2>(), fw.s, stage, eps, st);
        }
        for (int k = k1 - 1; k >= k0; --k) {
            double2 *W0 = segp + (k - k0) * nlink;
            LQCD_CUDA(cudaMemcpyAsync(W1, W0, ub, cudaMemcpyDeviceToDevice, st));
            flow_stage(lat, W1, X.as<double2>(), fw.s, 0, eps, st);
            LQCD_CUDA(cudaMemcpyAsync(W2, W1, ub, cudaMemcpyDeviceToDevice, st));
            flow_stage(lat, W2, X.as<double2>(), fw.s, 1, eps, st);
            const LinkField<F64> U0{W0, nullptr, S}, U1{W1, nullptr, S}, U2{W2, nullptr, S};
            laplace_stage(lat, U2, th, eta, nullptr, z2, nrhs, d, -8.0 * d, 0.0, st);  // z2 = d D2 eta
            laplace_stage(lat, U1, th, z2, nullptr, z1, nrhs, b, -8.0 * b, 0.0, st);   // z1 = b D1 z2
            for (int p = 0; p < 2; ++p) {
                ProfScope prof("fermion_backflow_combine", double(lat->vh) * nrhs * 5 * 192.0, st);
                backflow_combine_kernel<<<gvec, kBlock, 0, st>>>(lat->vh, nrhs, eta.half(p), z1.half(p), z2.half(p),
                                                                 u.half(p), w.half(p), a, c);
                LQCD_CHECK_LAUNCH();
            }
            laplace_stage(lat, U0, th, w, &u, eta, nrhs, 1.0, -8.0, 1.0, st, &z2, 1.0);  // eta = u + z2 + D0 w
        }
    }
    spinor_from_soa(lat, eta_dev, nrhs, eta.e, eta.o, st);
    LQCD_CUDA(cudaStreamSynchronize(st));  // scratch buffers are freed on return
}

}  // namespace lqcd
