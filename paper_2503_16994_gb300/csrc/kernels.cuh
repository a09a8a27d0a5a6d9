// Kernel templates of the Wilson-clover path.  Included by the translation
// units that instantiate them (one per storage precision, plus field_ops.cu).
#pragma once
#include <type_traits>

#include "lqcd_dev.cuh"

namespace lqcd {

// ---------------------------------------------------------------------------
// per right-hand-side solver state (device resident, one struct per RHS)
// ---------------------------------------------------------------------------
// ST_RESUME: just updated in FP64 while the others went on (batched
// solves); runs the second half of its iteration, then becomes ST_ACTIVE.
// ST_FINAL: the recursion's residual has reached the target; the correction is
// added and the FP64 residual of the full lattice that ends every solve
// decides (after a miss the next ones are checked like any update).
enum RhsStatus : int {
    ST_DONE = 0, ST_ACTIVE = 1, ST_UPDATE = 2, ST_MAXITER = 3, ST_IDLE = 4, ST_RESUME = 5, ST_FINAL = 6
};
enum RhsTrust : int { TRUST_NONE = 0, TRUST_OPEN = 1, TRUST_USED = 2, TRUST_MISSED = 3 };

struct RhsState {
    double gamma;    // |z|^2, z = Dhat^dag r (CGLS)
    double alpha, beta;
    double rr;       // |r|^2 of the low-precision residual
    double rr_ref;   // |r|^2 right after the last FP64 residual recomputation
    double scale;    // FP64 residual = scale * r, correction = scale * e
    double bnorm2;   // |b|^2 of the full system
    double target2;  // stop when the FP64 residual norm^2 <= target2
    double delta2;   // reliable-update factor squared
    double acc;      // accumulator for norms (true residual, |b|^2)
    double anchor2;  // |rhat|^2 of the last FP64 residual (the anchor of the incremental updates)
    int status;
    int iter;
    int updates;
    int maxiter;
    int resume;      // status after an FP64 residual that did not finish: ST_ACTIVE or ST_RESUME
    int trust;       // TRUST_OPEN: a converged recursion goes to ST_FINAL instead of ST_UPDATE (then TRUST_USED,
                     // and TRUST_MISSED once FP64 has not confirmed it)
    float alpha_f, beta_f;  // alpha, beta in FP32 (the FP16/FP32 vector kernels; converted once)
};

// What the last block does with a finished per-RHS sum.
enum RedOp : int {
    RED_STORE = 0,   // acc = sum
    RED_ADD = 1,     // acc += sum
    RED_ALPHA = 2,   // alpha = gamma / sum
    RED_BETA = 3,    // beta = sum / gamma (0 on the first pass); gamma = sum
    RED_RUPDATE = 4, // rr = sum; iter++; request an FP64 residual when due
    RED_RHAT = 5,    // sum = |FP64 residual|^2: finish, or resume the inner iteration
    RED_RHAT_COARSE = 6  // sum = |residual|^2 updated with an FP32 operator: resume (never finishes)
};

struct Reduce {
    double *partial;     // [nrhs][ntiles]
    unsigned *counter;   // [nrhs], zero between uses
    RhsState *st;        // [nrhs]
    int op;
    float *partial_f;    // [nrhs][4 ntiles]: FP32 sums per 32 sites (FP16/FP32 hopping kernels), or null
};

__device__ __forceinline__ void apply_op(const Reduce &r, int j, double sum)
{
    RhsState &s = r.st[j];
    switch (r.op) {
    case RED_STORE: s.acc = sum; break;
    case RED_ADD: s.acc += sum; break;
    case RED_ALPHA:
        s.alpha = sum > 0.0 ? s.gamma / sum : 0.0;
        s.alpha_f = float(s.alpha);
        break;
    case RED_BETA:
        s.beta = s.gamma > 0.0 ? sum / s.gamma : 0.0;
        s.beta_f = float(s.beta);
        s.gamma = sum;
        break;
    case RED_RUPDATE:
        s.rr = sum;
        s.iter += 1;
        if (s.trust == TRUST_OPEN && s.scale * s.scale * sum <= s.target2) {
            s.status = ST_FINAL;
            s.trust = TRUST_USED;
        } else if (sum <= s.delta2 * s.rr_ref || s.scale * s.scale * sum <= s.target2 || s.iter >= s.maxiter ||
                   !(sum == sum)) {
            s.status = ST_UPDATE;
        }
        break;
    case RED_RHAT:
        s.updates += 1;
        // far above the recursion's residual: what it gathered is of no use, begin again (beta = 0)
        if (sum > 4.0 * s.scale * s.scale * s.rr) s.gamma = 0.0;
        s.alpha = s.alpha_f = 0.f;  // alpha p is in e (cg_e_site), and e in x
        s.rr = sum / (s.scale * s.scale);
        s.rr_ref = s.rr;
        s.anchor2 = sum;
        if (sum <= s.target2)
            s.status = ST_DONE;
        else if (s.iter >= s.maxiter || !(sum == sum))
            s.status = ST_MAXITER;
        else
            s.status = s.resume;
        break;
    case RED_RHAT_COARSE:
        s.alpha = s.alpha_f = 0.f;
        s.rr = sum / (s.scale * s.scale);
        s.rr_ref = s.rr;
        s.status = (sum == sum) ? s.resume : ST_UPDATE;  // a NaN goes to the FP64 update
        break;
    }
}

// Sum of v over a block of at most 128 threads (result valid in warp 0).  The
// values meet in shared memory and one warp adds them, four to a lane: 8 FP64
// instructions of a warp instead of the 25 of a shuffle tree in every warp
// (block_sum).  An FP64 instruction takes this GPU's SM 16 cycles, so the
// tree of every block is 0.2 us of its SM.
__device__ __forceinline__ double block_sum4(double v, double *sh)
{
    __syncthreads();
    sh[threadIdx.x] = v;
    __syncthreads();
    if (threadIdx.x >= 32) return 0.0;
    double t[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) t[k] = threadIdx.x + 32 * k < blockDim.x ? sh[threadIdx.x + 32 * k] : 0.0;
    return warp_sum((t[0] + t[1]) + (t[2] + t[3]));
}

// Block-wide sums of v[0..n), written as the partials of tiles tile .. tile +
// n - 1; the last block of RHS j to arrive sums all partials in a fixed order
// (deterministic, and the same for every n) and applies the operation.  Must be
// called by every thread of the block (128).
template <int K>
__device__ __forceinline__ void reduce_finish(const Reduce &r, int j, int tile, int ntiles, const double (&v)[K])
{
    __shared__ double sh[128];
    __shared__ int last;
    const int n = min(K, ntiles - tile);
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const double s = block_sum4(v[k], sh);
        if (threadIdx.x == 0 && k < n) r.partial[(long)j * ntiles + tile + k] = s;
    }
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned prev = atomicAdd(&r.counter[j], unsigned(n));
        last = prev + n == unsigned(ntiles);
    }
    __syncthreads();
    if (last) {
        __threadfence();
        double t = 0.0;
        const double *p = r.partial + (long)j * ntiles;
        for (int k = threadIdx.x; k < ntiles; k += 8 * blockDim.x) {
            double q[8];  // eight loads in flight
#pragma unroll
            for (int u = 0; u < 8; ++u) q[u] = k + u * blockDim.x < ntiles ? __ldcg(p + k + u * blockDim.x) : 0.0;
#pragma unroll
            for (int u = 0; u < 8; ++u) t += q[u];
        }
        t = block_sum4(t, sh);
        if (threadIdx.x == 0) {
            r.counter[j] = 0;
            apply_op(r, j, t);
        }
    }
}

__device__ __forceinline__ void reduce_finish(const Reduce &r, int j, int tile, int ntiles, double v)
{
    const double a[1] = {v};
    reduce_finish<1>(r, j, tile, ntiles, a);
}

template <typename T>
__device__ __forceinline__ T warp_sum_t(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sums of the hopping kernels, added up by partial_finish_kernel (launched
// after them): no fence and no atomic, so no block waits for its own stores.
// Must be called by every thread of the block (128).
//
// FP64 kernels: the block's sum of v is RHS j's partial of this tile.
__device__ __forceinline__ void reduce_partial(const Reduce &r, int j, int tile, int ntiles, double v)
{
    __shared__ double sh[32];
    v = warp_sum_t(v);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    if (wid == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        v = warp_sum_t(lane < nw ? sh[lane] : 0.0);
        if (lane == 0) r.partial[(long)j * ntiles + tile] = v;
    }
}

// FP16/FP32 kernels, whose per-thread values are FP32 sums already (FP64 adds
// are scarce on this GPU): the sum of each warp, in FP32.  No barrier: a block
// that works through several groups of right-hand sides would line its warps up
// after each (12 on 24^3 x 48 in FP16, SELF_SUM: 254 us, 265 with the barriers).
__device__ __forceinline__ void warp_partial(const Reduce &r, int j, int tile, int ntiles, float v)
{
    v = warp_sum_t(v);
    if ((threadIdx.x & 31) == 0) r.partial_f[((long)j * ntiles + tile) * 4 + (threadIdx.x >> 5)] = v;
}

// Twisted mass in FP16/FP32: the threads' values are added in FP64 from the
// first addition on (a sum over 128 sites also leaves the range of FP32 where no
// site does), one partial per tile.  Must be called by every thread of the block.
__device__ __forceinline__ void block_partial(const Reduce &r, int j, int tile, int ntiles, double v)
{
    __shared__ double sh[128];
    const double s = block_sum4(v, sh);
    if (threadIdx.x == 0) r.partial[(long)j * ntiles + tile] = s;
}

// ---------------------------------------------------------------------------
// hopping term with fused epilogues
//
// H psi (x) = sum_mu [ (1 - s g_mu) U~_mu(x) psi(x+mu) + (1 + s g_mu) U~_mu(x-mu)^dag psi(x-mu) ]
// with s = +1 (D) or s = -1 (D^dag = g5 D g5, which swaps the projectors).
// Output sites have parity `parity`; psi lives on the other parity.
// ---------------------------------------------------------------------------
enum HopMode : int {
    HOP_CLOV = 0,   // out = coef * C (H in)
    SELF_CLOV = 1,  // out = C self + coef * H in
    SELF_PLAIN = 2, // out = self + coef * H in
    CLOV_SUM = 3,   // out = C (self + coef * H in), C an inverse; its norm is |self + coef * H in - A out|^2
    RESID = 4,      // |b - (C self + coef * H in)|^2 only, nothing stored
    ADD_CLOV = 5,   // out = self + coef * C (H in)
    SELF_SUM = 6,   // out = self + coef * H in (the solver's; SELF_PLAIN is its set-up's)
    TWIST = 8       // added to a mode inside the launcher: the site term with its twisted mass
};

template <class S, class L, class C>
struct HopArgs {
    Geom g;
    int parity;
    int nrhs;
    int ntiles;
    SpinorField<S> in, self, out, b;
    LinkField<L> U;
    CloverField<C> clov;   // clover blocks used by the epilogue (output parity taken from `parity`)
    CloverField<C> clov2;  // twisted mass: the C blocks of the inverse (clov then holds B), else unused
    CloverField<C> site;   // CLOV_SUM with the norm: the site blocks A
    double tau;            // twisted mass 2 kappa mu of the site term (0: none); the dagger uses -tau
    double coef;
    double th_re[4], th_im[4];
    const RhsState *gate_st;  // nullptr: every RHS runs
    int gate;                 // RHS j runs only if gate_st[j].status == gate
    Reduce red;
    int nactive = -1;         // launch accounting only: right-hand sides expected to pass the gate (-1: all)
    bool fixed_shape = false; // true: the scalar one-RHS-per-thread shape, neither tuned nor forced by
                              // the environment (its bits do not depend on the tuner's choice)
};

template <typename R> __device__ __forceinline__ spinor<R> axpy_sp(R c, const spinor<R> &x, const spinor<R> &y)
{
    spinor<R> r;
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int k = 0; k < 3; ++k) r.s[s][k] = c * x.s[s][k] + y.s[s][k];
    return r;
}

// out += i t g5 v: in the chiral basis g5 = +1 on spins 0, 1 and -1 on spins
// 2, 3, so the twisted-mass site term i tau g5 is a diagonal phase
template <typename R> __device__ __forceinline__ void add_twist(spinor<R> &out, R t, const spinor<R> &v)
{
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        const R ts = s < 2 ? t : -t;
#pragma unroll
        for (int k = 0; k < 3; ++k) out.s[s][k] = out.s[s][k] + ts * mul_i(v.s[s][k]);
    }
}

// (A + i t g5)^-1 v = (B - i t g5 C) v for the Hermitian blocks B = A C and
// C = (A^2 + t^2)^-1 of each chirality (A Hermitian)
template <typename R>
__device__ __forceinline__ spinor<R> twisted_inverse(const clover_block<R> B[2], const clover_block<R> C[2], R t,
                                                     const spinor<R> &v)
{
    spinor<R> r = clover_apply(B, v);
    add_twist(r, -t, clover_apply(C, v));
    return r;
}

template <typename R> __device__ __forceinline__ double norm2_sp(const spinor<R> &x)
{
    R acc = R(0);
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int k = 0; k < 3; ++k) acc += norm2(x.s[s][k]);
    return double(acc);
}

// ---------------------------------------------------------------------------
// CG vector kernels (one parity, nrhs right-hand sides)
// ---------------------------------------------------------------------------
struct VecArgs {
    int vh, nrhs, ntiles;
    const RhsState *gate_st;
    int gate;
    Reduce red;
    int nactive = -1;  // launch accounting only: right-hand sides expected to pass the gate (-1: all)
};

// an FP64 spinor by plain loads (a field that the same launch, or one in flight, also writes)
__device__ __forceinline__ spinor<double> load_spinor_f64_rw(const SpinorField<F64> &f, int j, int i)
{
    spinor<double> a;
    double *v = reinterpret_cast<double *>(&a);
    const double2 *b = f.p + (long)j * 12 * f.stride + i;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        const double2 w = b[k * f.stride];
        v[2 * k] = w.x;
        v[2 * k + 1] = w.y;
    }
    return a;
}

// a vector of the CG update kernels: FP64 ones are launched while the kernel
// before them still runs (launch_pdl), so they are read by plain loads
template <class S, typename R>
__device__ __forceinline__ spinor<R> load_vec(const SpinorField<S> &f, int j, int i)
{
    if constexpr (std::is_same<S, F64>::value && std::is_same<R, double>::value) return load_spinor_f64_rw(f, j, i);
    else return load_spinor<S, R>(f, j, i);
}

template <typename R> __device__ __forceinline__ R alpha_of(const RhsState &s)
{
    if constexpr (std::is_same<R, float>::value) return s.alpha_f;
    else return s.alpha;
}

// r -= alpha w ; |r|^2 -> RED_RUPDATE  (e += alpha p follows where p is read
// next: cg_p_update, cg_e_site).  K tiles per block: each block waits for its
// stores (the fence before its partials count) and for an atomic, 1.7 of the 4 us
// that a block of one tile lives.
template <class W, int K>
__global__ void __launch_bounds__(128) cg_r_update(VecArgs v, SpinorField<W> w, SpinorField<W> r)
{
    pdl_begin();
    const int j = blockIdx.x % v.nrhs, tile = blockIdx.x / v.nrhs * K;
    if (v.gate_st && v.gate_st[j].status != v.gate) return;
    using R = typename std::conditional<std::is_same<W, F64>::value, double, float>::type;
    const R al = alpha_of<R>(v.red.st[j]);
    double n2[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        n2[k] = 0.0;
        const int i = (tile + k) * blockDim.x + threadIdx.x;
        if (i < v.vh) {
            const spinor<R> wv = load_vec<W, R>(w, j, i), rv = load_vec<W, R>(r, j, i);
            n2[k] = store_spinor<W, R>(r, j, i, axpy_sp(-al, wv, rv));
        }
    }
    reduce_finish<K>(v.red, j, tile, v.ntiles, n2);
}

// x += scale e ; e = 0   (FP64 x)
template <class E>
__global__ void __launch_bounds__(128) cg_x_update(VecArgs v, const RhsState *st, SpinorField<E> e, SpinorField<F64> x)
{
    const int j = blockIdx.x % v.nrhs, tile = blockIdx.x / v.nrhs;
    if (v.gate_st && v.gate_st[j].status != v.gate) return;
    const int i = tile * blockDim.x + threadIdx.x;
    if (i >= v.vh) return;
    spinor<double> ev = load_spinor<E, double>(e, j, i);
    spinor<double> xv = load_spinor<F64, double>(x, j, i);
    store_spinor<F64, double>(x, j, i, axpy_sp(st[j].scale, ev, xv));
    spinor<double> z;
    zero(z);
    store_spinor<E, double>(e, j, i, z);
}

// rhat = src - c w (FP64 arithmetic): the FP64 update has src = bhat, w =
// Dhat x in FP64 and c = 1; the incremental update has src = the previous
// rhat, w = Dhat e in FP32 and c = scale (w_scaled).  r = rhat / scale (low
// precision); |rhat|^2 -> RED_RHAT(_COARSE); save (if set, may be src): rhat
// kept in FP64 for the next incremental update
template <class W, class WI>
__global__ void __launch_bounds__(128) cg_r_replace(VecArgs v, SpinorField<F64> src, SpinorField<WI> w,
                                                    SpinorField<W> r, SpinorField<F64> save, bool w_scaled)
{
    const int j = blockIdx.x % v.nrhs, tile = blockIdx.x / v.nrhs;
    if (v.gate_st && v.gate_st[j].status != v.gate) return;
    const int i = tile * blockDim.x + threadIdx.x;
    double n2 = 0.0;
    if (i < v.vh) {
        const double c = w_scaled ? v.red.st[j].scale : 1.0;
        spinor<double> rh = axpy_sp(-c, load_spinor<WI, double>(w, j, i), load_spinor_f64_rw(src, j, i));
        if (save.p) store_spinor<F64, double>(save, j, i, rh);
        n2 = norm2_sp(rh);
        const double inv = 1.0 / v.red.st[j].scale;
        using R = typename std::conditional<std::is_same<W, F64>::value, double, float>::type;
        spinor<R> rl;
#pragma unroll
        for (int s = 0; s < 4; ++s)
#pragma unroll
            for (int k = 0; k < 3; ++k) rl.s[s][k] = cx<R>{R(rh.s[s][k].re * inv), R(rh.s[s][k].im * inv)};
        store_spinor<W, R>(r, j, i, rl);
    }
    reduce_finish(v.red, j, tile, v.ntiles, n2);
}

// out = in, converted between storage formats
template <class SI, class SO>
__global__ void __launch_bounds__(128) convert_kernel(int vh, int nrhs, SpinorField<SI> in, SpinorField<SO> out)
{
    const int j = blockIdx.x % nrhs, tile = blockIdx.x / nrhs;
    const int i = tile * blockDim.x + threadIdx.x;
    if (i >= vh) return;
    store_spinor<SO, double>(out, j, i, load_spinor<SI, double>(in, j, i));
}

// out = C in (clover blocks of parity `parity`); with tau != 0 the twisted
// inverse (B - i tau g5 C2) in, cl holding B and cl2 C
template <class S, class C>
__global__ void __launch_bounds__(128) clover_apply_kernel(int vh, int nrhs, int parity, CloverField<C> cl,
                                                           SpinorField<S> in, SpinorField<S> out, double tau,
                                                           CloverField<C> cl2)
{
    const int j = blockIdx.x % nrhs, tile = blockIdx.x / nrhs;
    const int i = tile * blockDim.x + threadIdx.x;
    if (i >= vh) return;
    using R = typename std::conditional<std::is_same<S, F64>::value, double, float>::type;
    clover_block<R> blk[2];
    load_clover<C, R>(cl, parity, i, blk);
    const spinor<R> v = load_spinor<S, R>(in, j, i);
    if (tau != 0.0) {
        clover_block<R> blk2[2];
        load_clover<C, R>(cl2, parity, i, blk2);
        store_spinor<S, R>(out, j, i, twisted_inverse(blk, blk2, R(tau), v));
    } else {
        store_spinor<S, R>(out, j, i, clover_apply(blk, v));
    }
}

}  // namespace lqcd
