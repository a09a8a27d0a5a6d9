// Launchers of the CG vector kernels (explicit instantiations).
#include "hopfast.cuh"
#include "lqcd_impl.h"

namespace lqcd {

// |x|^2 of an FP64 field -> red.op
__global__ void __launch_bounds__(128) norm2_f64(VecArgs v, SpinorField<F64> x)
{
    const int j = blockIdx.x % v.nrhs, tile = blockIdx.x / v.nrhs;
    if (v.gate_st && v.gate_st[j].status != v.gate) return;
    const int i = tile * blockDim.x + threadIdx.x;
    double n2 = 0.0;
    if (i < v.vh) n2 = norm2_sp(load_spinor<F64, double>(x, j, i));
    reduce_finish(v.red, j, tile, v.ntiles, n2);
}

// the 24 reals of a right-hand side
template <class S, typename R>
__device__ __forceinline__ void load_scaled(const SpinorField<S> &f, int j, int i, R v[24])
{
    const R sc = load_raw<S, R>(f, j, i, v);
    if constexpr (S::W == 8) {
#pragma unroll
        for (int q = 0; q < 24; ++q) v[q] *= sc;
    }
}

// out = A_ee^-1 v (tau != 0: the twisted inverse (B - i s tau C) v of each chirality block, s = +1, -1)
template <class C, typename R>
__device__ __forceinline__ void site_inverse(const CloverField<C> &cl, const CloverField<C> &cl2, R tau, int i,
                                             const R v[24], R out[24])
{
    R A[36];
#pragma unroll
    for (int blk = 0; blk < 2; ++blk) {
        load_clov_block<C, R>(cl, 0, i, blk, A);
        clov6(A, v + 12 * blk, out + 12 * blk);
        if (tau != R(0)) {
            R c[12];
            load_clov_block<C, R>(cl2, 0, i, blk, A);
            clov6(A, v + 12 * blk, c);
            sub_it<6>(out + 12 * blk, blk ? -tau : tau, c);
        }
    }
}

// e += alpha p; p = z + beta p; z = A_ee^-1 p, the input of the next application
// of the operator.  e is updated here, where p is read anyway, and not with r
// (cg_r_update).  Bound by memory (p, z and e in and out and the clover block,
// which the right-hand sides of a site share in cache): for 12 right-hand sides
// on 24^3 x 48 in FP16 240 us, 6.8 TB/s, and 101 for r, where p and z took 152 us
// (5.7 TB/s) and r with e 239; one right-hand side on 32^3 x 64 82 + 39 us,
// before 53 + 92.  (The clover words loaded after the vectors cost 18 us more.)
// SITE false, here and below: CG on Dhat itself (Solver::divided), without the site blocks.
template <class W, class E, bool SITE>
__global__ void __launch_bounds__(128) cg_p_update(VecArgs v, const RhsState *st, SpinorField<W> z, SpinorField<W> p,
                                                   SpinorField<E> e, CloverField<W> cl, CloverField<W> cl2,
                                                   double tau)
{
    const int j = blockIdx.x % v.nrhs, tile = blockIdx.x / v.nrhs;
    if (v.gate_st && v.gate_st[j].status != v.gate) return;
    const int i = tile * blockDim.x + threadIdx.x;
    if (i >= v.vh) return;
    using R = typename real_of<W>::type;
    const R al = alpha_of<R>(st[j]), be = st[j].beta_f;
    R x[24], y[24];
    // FP16: the clover words are on their way with the vectors (36 registers)
    uint4 cw[W::W == 8 ? 9 : 1];
    if constexpr (SITE && W::W == 8) {
#pragma unroll
        for (int k = 0; k < 9; ++k) cw[k] = __ldg(cl.p + k * cl.stride + i);
    }
    load_scaled<W, R>(p, j, i, x);
    load_scaled<E, R>(e, j, i, y);
#pragma unroll
    for (int q = 0; q < 24; ++q) y[q] = fma(al, x[q], y[q]);
    store_raw<E, R>(e, j, i, y);
    load_scaled<W, R>(z, j, i, y);
#pragma unroll
    for (int q = 0; q < 24; ++q) x[q] = fma(be, x[q], y[q]);
    store_raw<W, R>(p, j, i, x);
    if constexpr (!SITE) return;
    if constexpr (SITE && W::W == 8) {
        if (tau == 0.0) {
            float A[36];
#pragma unroll
            for (int blk = 0; blk < 2; ++blk) {
#pragma unroll
                for (int q = 0; q < 18; ++q) {  // reals 36 blk + 2 q, + 1
                    const int h = 18 * blk + q;
                    const float2 f = __half22float2(reinterpret_cast<const __half2 *>(&cw[h / 4])[h % 4]);
                    A[2 * q] = f.x;
                    A[2 * q + 1] = f.y;
                }
                clov6(A, x + 12 * blk, y + 12 * blk);
            }
            store_raw<W, R>(z, j, i, y);
            return;
        }
    }
    site_inverse<W, R>(cl, cl2, R(tau), i, x, y);
    store_raw<W, R>(z, j, i, y);
}

// The same in FP64, a thread per (site, chirality block) in blocks of one warp:
// the site blocks are 264 FP64 instructions, and on a small lattice a block of
// 128 sites with all of them kept one SM busy for 8 us.
template <bool SITE>
__global__ void __launch_bounds__(32) cg_p_update64(VecArgs v, const RhsState *st, SpinorField<F64> z,
                                                    SpinorField<F64> p, SpinorField<F64> e, CloverField<F64> cl,
                                                    CloverField<F64> cl2, double tau)
{
    pdl_begin();
    const int blk = blockIdx.y, j = blockIdx.x % v.nrhs, i = (blockIdx.x / v.nrhs) * 32 + threadIdx.x;
    if (v.gate_st && v.gate_st[j].status != v.gate) return;
    if (i >= v.vh) return;
    const double al = st[j].alpha, be = st[j].beta;
    double2 *eb = e.p + ((long)j * 12 + 6 * blk) * e.stride + i;
    double2 *pb = p.p + ((long)j * 12 + 6 * blk) * p.stride + i, *zb = z.p + ((long)j * 12 + 6 * blk) * z.stride + i;
    double x[12], y[12], A[36];
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const double2 a = pb[k * p.stride], b = zb[k * z.stride], c = eb[k * e.stride];
        eb[k * e.stride] = make_double2(fma(al, a.x, c.x), fma(al, a.y, c.y));
        x[2 * k] = fma(be, a.x, b.x);
        x[2 * k + 1] = fma(be, a.y, b.y);
        pb[k * p.stride] = make_double2(x[2 * k], x[2 * k + 1]);
    }
    if constexpr (!SITE) return;
    load_clov_block<F64, double>(cl, 0, i, blk, A);
    clov6(A, x, y);
    if (tau != 0.0) {
        double c[12];
        load_clov_block<F64, double>(cl2, 0, i, blk, A);
        clov6(A, x, c);
        sub_it<6>(y, blk ? -tau : tau, c);
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) zb[k * z.stride] = make_double2(y[2 * k], y[2 * k + 1]);
}

// e = A_ee^-1 (e + alpha p), the correction in terms of the solution, with the
// step that cg_p_update would have added next (residual updates)
template <class W, class E, bool SITE>
__global__ void __launch_bounds__(128) cg_e_site(VecArgs v, const RhsState *st, SpinorField<W> p, SpinorField<E> e,
                                                 CloverField<E> cl, CloverField<E> cl2, double tau)
{
    const int j = blockIdx.x % v.nrhs, tile = blockIdx.x / v.nrhs;
    if (v.gate_st && v.gate_st[j].status != v.gate) return;
    const int i = tile * blockDim.x + threadIdx.x;
    if (i >= v.vh) return;
    using R = typename real_of<E>::type;
    R x[24], y[24];
    load_scaled<E, R>(e, j, i, x);
    load_scaled<W, R>(p, j, i, y);
    const R al = alpha_of<R>(st[j]);
#pragma unroll
    for (int q = 0; q < 24; ++q) x[q] = fma(al, y[q], x[q]);
    if constexpr (SITE) {
        site_inverse<E, R>(cl, cl2, R(tau), i, x, y);
        store_raw<E, R>(e, j, i, y);
    } else {
        store_raw<E, R>(e, j, i, x);
    }
}

// |x|^2 of the gated-in right-hand sides (CG on Dhat itself, whose hops have no norm of their own)
template <class W>
__global__ void __launch_bounds__(128) norm2_vec(VecArgs v, SpinorField<W> x)
{
    const int j = blockIdx.x % v.nrhs, tile = blockIdx.x / v.nrhs;
    if (v.gate_st && v.gate_st[j].status != v.gate) return;
    const int i = tile * blockDim.x + threadIdx.x;
    using R = typename real_of<W>::type;
    R t = R(0);
    if (i < v.vh) {
        R a[24];
        load_scaled<W, R>(x, j, i, a);
#pragma unroll
        for (int q = 0; q < 24; ++q) t = fma(a[q], a[q], t);
    }
    reduce_finish(v.red, j, tile, v.ntiles, double(t));
}

// *out = max(*out, the bits of the largest |entry| of A_ee^-1 in FP32), which
// order as the values do, infinities and NaN on top; twisted: of its parts B
// and tau C.  One pass over the FP64 blocks of the even sites per clover field.
__global__ void __launch_bounds__(128) site_inverse_max_kernel(int vh, CloverField<F64> cl, CloverField<F64> cl2,
                                                               double tau, unsigned *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned m = 0;
    if (i < vh) {
        auto take = [&](double x) { m = max(m, __float_as_uint(fabsf(float(x)))); };
        for (int k = 0; k < 36; ++k) {
            const double2 w = cl.p[k * cl.stride + i];
            take(w.x);
            take(w.y);
            if (tau != 0.0) {
                const double2 c = cl2.p[k * cl2.stride + i];
                take(tau * c.x);
                take(tau * c.y);
            }
        }
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

// Partial of 128-site tile k of RHS j.  QUAD: the FP32 sums of its four
// 32-site quarters, added in FP32.
template <bool QUAD>
__device__ __forceinline__ double tile_partial(const Reduce &r, int j, int ntiles, int k)
{
    if constexpr (QUAD) {
        const float2 *q = reinterpret_cast<const float2 *>(r.partial_f + ((long)j * ntiles + k) * 4);  // 8-byte aligned
        const float2 a = q[0], b = q[1];
        return double((a.x + b.x) + (a.y + b.y));
    } else {
        return r.partial[(long)j * ntiles + k];
    }
}

// Sum of the per-tile partials of each gated-in RHS (one block per RHS, fixed
// order: deterministic) and its operation.  One warp adds the threads' sums:
// a shuffle tree in each of the 16 warps takes 80 FP64 instructions (16 cycles
// each), twice the time of everything else at 4^4.
constexpr int kFinishThreads = 512;
template <bool QUAD>
__global__ void __launch_bounds__(kFinishThreads) partial_finish_kernel(Reduce r, int ntiles, const RhsState *gate_st,
                                                                       int gate)
{
    __shared__ double sh[kFinishThreads];
    pdl_begin();
    const int j = blockIdx.x;
    if (gate_st && gate_st[j].status != gate) return;
    double t[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) t[q] = 0.0;
    for (int k = threadIdx.x; k < ntiles; k += 8 * kFinishThreads) {
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (k + q * kFinishThreads < ntiles) t[q] += tile_partial<QUAD>(r, j, ntiles, k + q * kFinishThreads);
    }
    sh[threadIdx.x] = ((t[0] + t[1]) + (t[2] + t[3])) + ((t[4] + t[5]) + (t[6] + t[7]));
    __syncthreads();
    if (threadIdx.x >= 32) return;
    double s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < kFinishThreads / 32; ++k) s[k & 3] += sh[threadIdx.x + 32 * k];
    const double sum = warp_sum((s[0] + s[1]) + (s[2] + s[3]));
    if (threadIdx.x == 0) apply_op(r, j, sum);
}

void launch_partial_finish(const Reduce &r, int ntiles, int nrhs, const RhsState *gate_st, int gate, cudaStream_t st,
                           bool quad)
{
    ProfScope prof("norm_finish", double(nrhs) * ntiles * (quad ? 16.0 : 8.0), st);
    if (quad)
        launch_pdl(partial_finish_kernel<true>, dim3(unsigned(nrhs)), kFinishThreads, 0, st, r, ntiles, gate_st, gate);
    else
        launch_pdl(partial_finish_kernel<false>, dim3(unsigned(nrhs)), kFinishThreads, 0, st, r, ntiles, gate_st, gate);
    LQCD_CHECK_LAUNCH();
}

// From here cg_r_update takes four tiles per block: the chip holds about 1200 of
// its blocks, so four times fewer still fill it.  In FP16 8192 tiles (one
// right-hand side on 32^3 x 64) take 39 us instead of 51 and 31104 (12 on
// 24^3 x 48) 101 instead of 108; fewer tiles than 4096 keep a block each.
constexpr unsigned kManyTiles = 4096;
static unsigned grid_of(const VecArgs &v) { return unsigned(v.ntiles * v.nrhs); }
// right-hand sides a launch is expected to work on (accounting only)
static double nact(const VecArgs &v) { return v.nactive >= 0 ? std::min(v.nactive, v.nrhs) : v.nrhs; }

template <class W>
void launch_r_update(const VecArgs &v, SpinorField<W> w, SpinorField<W> r, cudaStream_t st)
{
    ProfScope prof("cg_r_update", double(v.vh) * nact(v) * 3.0 * spinor_bytes<W>(), st);
    const bool many = grid_of(v) >= kManyTiles;
    const unsigned grid = many ? unsigned((v.ntiles + 3) / 4) * unsigned(v.nrhs) : grid_of(v);
    if constexpr (std::is_same<W, F64>::value) {
        if (many) launch_pdl(cg_r_update<W, 4>, dim3(grid), kBlock, 0, st, v, w, r);
        else launch_pdl(cg_r_update<W, 1>, dim3(grid), kBlock, 0, st, v, w, r);
    } else {
        if (many) cg_r_update<W, 4><<<grid, kBlock, 0, st>>>(v, w, r);
        else cg_r_update<W, 1><<<grid, kBlock, 0, st>>>(v, w, r);
    }
    LQCD_CHECK_LAUNCH();
}

template <class W, class E>
void launch_p_update(const VecArgs &v, const RhsState *s, SpinorField<W> z, SpinorField<W> p, SpinorField<E> e,
                     CloverField<W> cl, CloverField<W> cl2, double tau, cudaStream_t st)
{
    const bool site = cl.p != nullptr;
    ProfScope prof("cg_p_update",
                   double(v.vh) * (nact(v) * ((site ? 4.0 : 3.0) * spinor_bytes<W>() + 2.0 * spinor_bytes<E>()) +
                                   (site ? (tau != 0.0 ? 2.0 : 1.0) : 0.0) * clover_bytes<W>()),
                   st);
    if constexpr (std::is_same<W, F64>::value)
        launch_pdl(site ? cg_p_update64<true> : cg_p_update64<false>,
                   dim3(unsigned((v.vh + 31) / 32) * unsigned(v.nrhs), 2), 32, 0, st, v, s, z, p, e, cl, cl2, tau);
    else if (site)
        cg_p_update<W, E, true><<<grid_of(v), kBlock, 0, st>>>(v, s, z, p, e, cl, cl2, tau);
    else
        cg_p_update<W, E, false><<<grid_of(v), kBlock, 0, st>>>(v, s, z, p, e, cl, cl2, tau);
    LQCD_CHECK_LAUNCH();
}

template <class W, class E>
void launch_e_site(const VecArgs &v, const RhsState *s, SpinorField<W> p, SpinorField<E> e, CloverField<E> cl,
                   CloverField<E> cl2, double tau, cudaStream_t st)
{
    const bool site = cl.p != nullptr;
    ProfScope prof("cg_e_site",
                   double(v.vh) * (nact(v) * (2.0 * spinor_bytes<E>() + spinor_bytes<W>()) +
                                   (site ? (tau != 0.0 ? 2.0 : 1.0) : 0.0) * clover_bytes<E>()),
                   st);
    if (site) cg_e_site<W, E, true><<<grid_of(v), kBlock, 0, st>>>(v, s, p, e, cl, cl2, tau);
    else cg_e_site<W, E, false><<<grid_of(v), kBlock, 0, st>>>(v, s, p, e, cl, cl2, tau);
    LQCD_CHECK_LAUNCH();
}

template <class W>
void launch_norm2(const VecArgs &v, SpinorField<W> x, cudaStream_t st)
{
    ProfScope prof("cg_norm2", double(v.vh) * nact(v) * spinor_bytes<W>(), st);
    norm2_vec<W><<<grid_of(v), kBlock, 0, st>>>(v, x);
    LQCD_CHECK_LAUNCH();
}

void launch_site_inverse_max(long vh, CloverField<F64> cl, CloverField<F64> cl2, double tau, unsigned *out,
                             cudaStream_t st)
{
    ProfScope prof("site_inverse_max", double(vh) * (tau != 0.0 ? 2.0 : 1.0) * clover_bytes<F64>(), st);
    site_inverse_max_kernel<<<unsigned(ntiles_of(vh)), kBlock, 0, st>>>(int(vh), cl, cl2, tau, out);
    LQCD_CHECK_LAUNCH();
}

template <class E>
void launch_x_update(const VecArgs &v, const RhsState *s, SpinorField<E> e, SpinorField<F64> x, cudaStream_t st)
{
    ProfScope prof("cg_x_update", double(v.vh) * nact(v) * (2.0 * spinor_bytes<E>() + 2.0 * 192.0), st);
    cg_x_update<E><<<grid_of(v), kBlock, 0, st>>>(v, s, e, x);
    LQCD_CHECK_LAUNCH();
}

template <class W, class WI>
void launch_r_replace(const VecArgs &v, SpinorField<F64> src, SpinorField<WI> w, SpinorField<W> r,
                      SpinorField<F64> save, bool w_scaled, cudaStream_t st)
{
    ProfScope prof("cg_r_replace",
                   double(v.vh) * nact(v) * (192.0 + spinor_bytes<WI>() + spinor_bytes<W>() + (save.p ? 192.0 : 0.0)),
                   st);
    cg_r_replace<W, WI><<<grid_of(v), kBlock, 0, st>>>(v, src, w, r, save, w_scaled);
    LQCD_CHECK_LAUNCH();
}

void launch_norm2_f64(const VecArgs &v, SpinorField<F64> x, cudaStream_t st)
{
    ProfScope prof("norm2_f64", double(v.vh) * v.nrhs * 192.0, st);
    norm2_f64<<<grid_of(v), kBlock, 0, st>>>(v, x);
    LQCD_CHECK_LAUNCH();
}

template <class S, class C>
void launch_clover_apply(long vh, int nrhs, int parity, CloverField<C> cl, SpinorField<S> in, SpinorField<S> out,
                         cudaStream_t st, double tau, CloverField<C> cl2)
{
    ProfScope prof("clover_apply",
                   double(vh) * (nrhs * 2.0 * spinor_bytes<S>() + (tau != 0.0 ? 2.0 : 1.0) * clover_bytes<C>()), st);
    clover_apply_kernel<S, C>
        <<<unsigned(ntiles_of(vh) * nrhs), kBlock, 0, st>>>(int(vh), nrhs, parity, cl, in, out, tau, cl2);
    LQCD_CHECK_LAUNCH();
}

template <class SI, class SO>
void launch_convert(long vh, int nrhs, SpinorField<SI> in, SpinorField<SO> out, cudaStream_t st)
{
    ProfScope prof("convert", double(vh) * nrhs * (spinor_bytes<SI>() + spinor_bytes<SO>()), st);
    convert_kernel<SI, SO><<<unsigned(ntiles_of(vh) * nrhs), kBlock, 0, st>>>(int(vh), nrhs, in, out);
    LQCD_CHECK_LAUNCH();
}

template void launch_convert<F64, F64>(long, int, SpinorField<F64>, SpinorField<F64>, cudaStream_t);
template void launch_convert<F64, F32>(long, int, SpinorField<F64>, SpinorField<F32>, cudaStream_t);
template void launch_convert<F64, F16>(long, int, SpinorField<F64>, SpinorField<F16>, cudaStream_t);
template void launch_convert<F32, F64>(long, int, SpinorField<F32>, SpinorField<F64>, cudaStream_t);
template void launch_convert<F16, F64>(long, int, SpinorField<F16>, SpinorField<F64>, cudaStream_t);
template void launch_norm2<F64>(const VecArgs &, SpinorField<F64>, cudaStream_t);
template void launch_norm2<F32>(const VecArgs &, SpinorField<F32>, cudaStream_t);
template void launch_norm2<F16>(const VecArgs &, SpinorField<F16>, cudaStream_t);
template void launch_r_update<F64>(const VecArgs &, SpinorField<F64>, SpinorField<F64>, cudaStream_t);
template void launch_r_update<F32>(const VecArgs &, SpinorField<F32>, SpinorField<F32>, cudaStream_t);
template void launch_r_update<F16>(const VecArgs &, SpinorField<F16>, SpinorField<F16>, cudaStream_t);
template void launch_p_update<F64, F64>(const VecArgs &, const RhsState *, SpinorField<F64>, SpinorField<F64>,
                                        SpinorField<F64>, CloverField<F64>, CloverField<F64>, double, cudaStream_t);
template void launch_p_update<F32, F32>(const VecArgs &, const RhsState *, SpinorField<F32>, SpinorField<F32>,
                                        SpinorField<F32>, CloverField<F32>, CloverField<F32>, double, cudaStream_t);
template void launch_p_update<F16, F32>(const VecArgs &, const RhsState *, SpinorField<F16>, SpinorField<F16>,
                                        SpinorField<F32>, CloverField<F16>, CloverField<F16>, double, cudaStream_t);
template void launch_e_site<F64, F64>(const VecArgs &, const RhsState *, SpinorField<F64>, SpinorField<F64>,
                                      CloverField<F64>, CloverField<F64>, double, cudaStream_t);
template void launch_e_site<F32, F32>(const VecArgs &, const RhsState *, SpinorField<F32>, SpinorField<F32>,
                                      CloverField<F32>, CloverField<F32>, double, cudaStream_t);
template void launch_e_site<F16, F32>(const VecArgs &, const RhsState *, SpinorField<F16>, SpinorField<F32>,
                                      CloverField<F32>, CloverField<F32>, double, cudaStream_t);
template void launch_x_update<F64>(const VecArgs &, const RhsState *, SpinorField<F64>, SpinorField<F64>, cudaStream_t);
template void launch_x_update<F32>(const VecArgs &, const RhsState *, SpinorField<F32>, SpinorField<F64>, cudaStream_t);
template void launch_r_replace<F64, F64>(const VecArgs &, SpinorField<F64>, SpinorField<F64>, SpinorField<F64>,
                                         SpinorField<F64>, bool, cudaStream_t);
template void launch_r_replace<F32, F64>(const VecArgs &, SpinorField<F64>, SpinorField<F64>, SpinorField<F32>,
                                         SpinorField<F64>, bool, cudaStream_t);
template void launch_r_replace<F16, F64>(const VecArgs &, SpinorField<F64>, SpinorField<F64>, SpinorField<F16>,
                                         SpinorField<F64>, bool, cudaStream_t);
template void launch_r_replace<F32, F32>(const VecArgs &, SpinorField<F64>, SpinorField<F32>, SpinorField<F32>,
                                         SpinorField<F64>, bool, cudaStream_t);
template void launch_r_replace<F16, F32>(const VecArgs &, SpinorField<F64>, SpinorField<F32>, SpinorField<F16>,
                                         SpinorField<F64>, bool, cudaStream_t);
template void launch_clover_apply<F64, F64>(long, int, int, CloverField<F64>, SpinorField<F64>, SpinorField<F64>,
                                            cudaStream_t, double, CloverField<F64>);

}  // namespace lqcd
