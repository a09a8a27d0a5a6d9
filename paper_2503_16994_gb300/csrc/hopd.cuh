// Hopping kernel for small lattices in FP64: 16 threads per output site.
//
// FP64 runs at two instructions per clock and SM, so one thread per site
// keeps a block of 128 sites busy for 35 us on one SM while the others idle.
// Here a block of four warps takes 8 sites: warp mu does direction mu, and
// its lanes are (site, projected spin s, forward or backward), so each thread
// has one spin projection and one link product (42 FP64 instructions).  The
// eight contributions of a component meet in shared memory, where 96 threads
// (site, component) add them and apply their row of the clover block.  The
// work per site is that of the one-thread form (about 1130 FP64 instructions);
// it only reaches 16 times as many SMs.  Every sum is formed in the order of
// the one-thread kernel, so both store the same bits (the norms are summed in
// another order).
#pragma once
#include "hopfast.cuh"

namespace lqcd {

constexpr int kSplitSites = 8;  // output sites per block
// One thread per site takes 45 us for any number of sites that fit one block
// per SM (152 x 128) and goes up in steps of that; this kernel takes 8.4 us up
// to 512 sites and then 2.8 us per 1000 sites x right-hand sides: 4^4 8.4
// against 45 us, 8192 sites 25 against 45; twelve right-hand sides at 512
// sites 22 against 45, but 83 against 82 at 2048 sites.
constexpr long kSplitMax = 12288;
inline bool split_hop(long vh, int nrhs) { return vh * nrhs <= kSplitMax; }

__host__ __device__ inline int split_blocks(long vh) { return int((vh + kSplitSites - 1) / kSplitSites); }

// x with its sign flipped where neg (no FP64 instruction)
__device__ __forceinline__ double flip(double x, bool neg)
{
    return __hiloint2double(__double2hiint(x) ^ (neg ? int(0x80000000u) : 0), __double2loint(x));
}

// row r of the Hermitian 6x6 block blk: the diagonal entry and the five others in column order
struct CloverRow {
    double d;
    double2 o[5];
};

template <class C>
__device__ __forceinline__ void load_clover_row(const CloverField<C> &f, int parity, int i, int blk, int r,
                                                CloverRow &A)
{
    const double2 *b = f.p + ((long)parity * 36 + blk * 18) * f.stride + i;
    const double2 d = __ldg(b + (r >> 1) * f.stride);
    A.d = (r & 1) ? d.y : d.x;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const int c = k < r ? k : k + 1;
        double2 w = __ldg(b + (3 + tri(min(r, c), max(r, c))) * f.stride);
        w.y = flip(w.y, c < r);  // below the diagonal: the conjugate of the stored entry
        A.o[k] = w;
    }
}

// (A v)_r, v in shared memory with `step` entries from component to component
__device__ __forceinline__ double2 clover_row(const CloverRow &A, const double2 *v, int step, int r)
{
    const double2 x = v[r * step];
    double re = A.d * x.x, im = A.d * x.y;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const double2 y = v[(k < r ? k : k + 1) * step];
        cmad(re, im, A.o[k].x, A.o[k].y, y.x, y.y);
    }
    return make_double2(re, im);
}

// clov2: the C blocks of the twisted inverse (see HopArgs).  S: F64, or A64
// for both parities of host-layout fields in one launch (blockIdx.y).
template <class S, int MODE, bool DAG, bool NORM>
__global__ void __launch_bounds__(128) hopd_kernel(const FastHop<S> a, const CloverField<F64> clov2)
{
    pdl_begin();
    constexpr bool HOST = std::is_same<S, A64>::value;
    const int parity = HOST ? int(blockIdx.y) : a.parity;
    const double tau = a.tau;
    // the word of component 0 at a field's site, and the step to the next component
    auto base = [&](const SpinorField<S> &f, int j, int cb, int odd) {
        return HOST ? f.p + (long)spinor_site<S>(cb, odd) * 12 : f.p + (long)j * 12 * f.stride + cb;
    };
    auto step_of = [&](const SpinorField<S> &f) { return HOST ? 1L : f.stride; };
    __shared__ double2 part[8][12][kSplitSites];
    __shared__ double2 vec[12][kSplitSites];
    __shared__ double red[4];
    const int j = blockIdx.x % a.nrhs, tile = blockIdx.x / a.nrhs;
    if (a.gate_st && a.gate_st[j].status != a.gate) return;
    const int lane = threadIdx.x & 31, mu = threadIdx.x >> 5;
    const bool worker = threadIdx.x < 12 * kSplitSites;  // the second half of the kernel: (site, component)
    const int wsite = threadIdx.x & 7, comp = min(int(threadIdx.x >> 3), 11);
    const int wi = min(tile * kSplitSites + wsite, a.vh - 1);
    const bool wvalid = worker && tile * kSplitSites + wsite < a.vh;
    // the rows of the clover block are on their way while the hops run
    constexpr bool PLAIN = MODE == SELF_PLAIN || MODE == SELF_SUM, CLOV = !PLAIN;
    // the block is an inverse: twisted by B and C
    constexpr bool INV = MODE == HOP_CLOV || MODE == CLOV_SUM || MODE == ADD_CLOV;
    CloverRow A, A2, As;
    if (CLOV && worker) {
        load_clover_row(a.clov, parity, wi, comp / 6, comp % 6, A);
        if (INV && tau != 0.0) load_clover_row(clov2, parity, wi, comp / 6, comp % 6, A2);
        if (MODE == CLOV_SUM && NORM) load_clover_row(a.site, parity, wi, comp / 6, comp % 6, As);
    }
    int wodd = 0;
    if (HOST) {
        const unsigned row = fdiv(unsigned(wi), a.dx), q1 = fdiv(row, a.dy), q2 = fdiv(q1, a.dz);
        wodd = (parity + int(row - q1 * unsigned(a.L[1])) + int(q1 - q2 * unsigned(a.L[2])) + int(q2)) & 1;
    }
    double2 self = make_double2(0.0, 0.0);
    if (MODE != HOP_CLOV && worker) {
        self = *(base(a.self, j, wi, wodd) + comp * step_of(a.self));
        if (MODE == SELF_CLOV || MODE == RESID) vec[comp][wsite] = self;
    }
    {
        const int site = lane & 7, s = (lane >> 3) & 1, back = lane >> 4;
        const int i = min(tile * kSplitSites + site, a.vh - 1);
        const unsigned row = fdiv(unsigned(i), a.dx);
        const int xh = i - int(row) * a.Lxh;
        const unsigned q1 = fdiv(row, a.dy);
        const int y = int(row) - int(q1) * a.L[1];
        const unsigned q2 = fdiv(q1, a.dz);
        const int z = int(q1) - int(q2) * a.L[2];
        const int t = int(q2);
        const int odd = (parity + y + z + t) & 1, x = 2 * xh + odd;
        bool wrap;
        int n;
        if (mu == 0) {
            wrap = x == (back ? 0 : a.L[0] - 1);
            const int xn = back ? (wrap ? a.L[0] - 1 : x - 1) : (wrap ? 0 : x + 1);
            n = int(row) * a.Lxh + (xn >> 1);
        } else {
            const int c = mu == 1 ? y : (mu == 2 ? z : t), L = a.L[mu], o = mu == 1 ? a.oy : (mu == 2 ? a.oz : a.ot);
            wrap = c == (back ? 0 : L - 1);
            const int step = wrap ? -(L - 1) * o : o;
            n = back ? i - step : i + step;
        }
        // the link W = U_mu(x), or U_mu(x - mu)^dag by the transposed planes and the sign of the imaginary parts
        const double2 *up = a.U.p + (long)((back ? parity ^ 1 : parity) * 4 + mu) * 9 * a.U.stride + (back ? n : i);
        const double2 *ip = base(a.in, j, n, mu == 0 ? 1 - odd : odd);
        const long is = step_of(a.in);
        double2 w[3][3];
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int c = 0; c < 3; ++c) w[r][c] = __ldg(up + (back ? 3 * c + r : 3 * r + c) * a.U.stride);
        // (1 + S g_mu) psi = (h, lower): h_s = psi_s - S f psi_(2+o) with o = 1 - s for x, y and s for z, t,
        // f = i, +-1, +-i, 1 (cases of project_f); S = -+ 1 for the forward / backward hop of D, swapped for D^dag
        const int o = mu < 2 ? 1 - s : s;
        const bool minus = (back != 0) == DAG;                    // S = -1
        const bool fneg = ((mu == 1 || mu == 2) && s == 1) == minus;  // -S f without the i is negative
        const bool im = mu == 0 || mu == 2;
        double hr[3], hi[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double2 u = *(ip + (3 * s + c) * is), d = *(ip + (3 * (2 + o) + c) * is);
            hr[c] = u.x + flip(im ? d.y : d.x, fneg != im);
            hi[c] = u.y + flip(im ? d.x : d.y, fneg);
        }
        const bool ph = wrap && ((a.theta_mask >> mu) & 1);
        const double pr = a.th_re[mu], pi = back ? -a.th_im[mu] : a.th_im[mu];
        // lower spin 2 + o takes S f' g_s: f' = i, (1 to o = 0, -1 to o = 1), (i, -i), and -S g_s for t
        const bool lneg = (mu == 3 || (mu != 0 && o == 1)) != minus;
        const int md = mu * 2 + back;
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            double re = 0.0, ii = 0.0;
#pragma unroll
            for (int c = 0; c < 3; ++c) cmad(re, ii, w[r][c].x, flip(w[r][c].y, back != 0), hr[c], hi[c]);
            if (ph) phase_mul(re, ii, pr, pi);
            part[md][3 * s + r][site] = make_double2(re, ii);
            part[md][3 * (2 + o) + r][site] =
                make_double2(flip(im ? ii : re, lneg != im), flip(im ? re : ii, lneg));
        }
    }
    __syncthreads();
    double2 H = make_double2(0.0, 0.0);
    if (worker) {
        H = part[0][comp][wsite];
#pragma unroll
        for (int m = 1; m < 8; ++m) {
            const double2 p = part[m][comp][wsite];
            H = make_double2(H.x + p.x, H.y + p.y);
        }
    }
    const double coef = a.coef;
    if (INV) {  // the block acts on H, or on self + coef H
        if (worker)
            vec[comp][wsite] =
                MODE != CLOV_SUM ? H : make_double2(fma(coef, H.x, self.x), fma(coef, H.y, self.y));
        __syncthreads();
    }
    double n2 = 0.0;
    double2 out = make_double2(0.0, 0.0);
    if (wvalid) {
        const int blk = comp / 6, r = comp % 6;
        const double2 *v = &vec[6 * blk][wsite];
        const double ts = (blk == 0) != DAG ? tau : -tau;  // the twist of this chirality, -tau for the adjoint
        double2 res;
        if (INV) {
            res = clover_row(A, v, kSplitSites, r);
            if (tau != 0.0) {
                const double2 c = clover_row(A2, v, kSplitSites, r);  // B v - i ts C v
                res.x = fma(ts, c.y, res.x);
                res.y = fma(-ts, c.x, res.y);
            }
            if (MODE == HOP_CLOV) res = make_double2(coef * res.x, coef * res.y);
            if (MODE == ADD_CLOV) res = make_double2(fma(coef, res.x, self.x), fma(coef, res.y, self.y));
        } else if (PLAIN) {
            res = make_double2(fma(coef, H.x, self.x), fma(coef, H.y, self.y));
        } else {
            res = clover_row(A, v, kSplitSites, r);
            if (tau != 0.0) {  // + i ts self
                res.x = fma(-ts, self.y, res.x);
                res.y = fma(ts, self.x, res.y);
            }
            res = make_double2(fma(coef, H.x, res.x), fma(coef, H.y, res.y));
        }
        if (MODE == RESID) {
            const double2 b = a.b.p[((long)j * 12 + comp) * a.b.stride + wi];
            res = make_double2(b.x - res.x, b.y - res.y);
        } else {
            base(a.out, j, wi, wodd)[comp * step_of(a.out)] = res;
        }
        n2 = fma(res.x, res.x, res.y * res.y);
        out = res;
    }
    if (MODE == CLOV_SUM && NORM) {  // |self + coef H in - A out|^2
        __syncthreads();  // every row has read its input
        const double2 v = worker ? vec[comp][wsite] : make_double2(0.0, 0.0);
        __syncthreads();
        if (worker) vec[comp][wsite] = out;
        __syncthreads();
        if (wvalid) {
            const int blk = comp / 6;
            const double ts = (blk == 0) != DAG ? tau : -tau;
            double2 ao = clover_row(As, &vec[6 * blk][wsite], kSplitSites, comp % 6);
            ao.x = fma(-ts, out.y, ao.x);
            ao.y = fma(ts, out.x, ao.y);
            n2 = fma(v.x - ao.x, v.x - ao.x, (v.y - ao.y) * (v.y - ao.y));
        }
    }
    if (NORM) {
        n2 = warp_sum(n2);
        if (lane == 0) red[mu] = n2;
        __syncthreads();
        if (threadIdx.x == 0)
            a.red.partial[(long)j * split_blocks(a.vh) + tile] = (red[0] + red[1]) + (red[2] + red[3]);
    }
}

}  // namespace lqcd
