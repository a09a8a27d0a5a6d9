// FP64-storage instantiations of the hopping kernel, and D on the host layout.
#include "dslash_inst.cuh"

namespace lqcd {
template void launch_hop<F64, F64, F64>(const HopArgs<F64, F64, F64> &, int, bool, bool, cudaStream_t);

void launch_dirac(const HopArgs<F64, F64, F64> &a, const double *in, double *out, bool dag, cudaStream_t st)
{
    FastHop<A64> f = make_shape<A64>(a);
    f.in = {reinterpret_cast<double2 *>(const_cast<double *>(in)), nullptr, a.g.stride};  // read only
    f.self = f.in;
    f.out = {reinterpret_cast<double2 *>(out), nullptr, a.g.stride};
    f.U = {a.U.p, nullptr, a.U.stride};
    f.clov = {a.clov.p, a.clov.stride};
    // D psi (x) on every site: the spinor at 8 neighbours and itself, 8 links, the clover blocks
    ProfScope prof("dirac_f64", 2.0 * double(a.g.vh) * (2 * 192.0 + 8 * 144.0 + 576.0), st);
    if (split_hop(a.g.vh, 1)) {
        const dim3 grid{unsigned(split_blocks(a.g.vh)), 2};
        if (dag) hopd_kernel<A64, SELF_CLOV, true, false><<<grid, 128, 0, st>>>(f, CloverField<F64>{});
        else hopd_kernel<A64, SELF_CLOV, false, false><<<grid, 128, 0, st>>>(f, CloverField<F64>{});
    } else {
        const dim3 grid{unsigned(f.ntiles), 2};
        if (dag) dirac_kernel<true><<<grid, kBlock, 0, st>>>(f);
        else dirac_kernel<false><<<grid, kBlock, 0, st>>>(f);
    }
    LQCD_CHECK_LAUNCH();
}
}  // namespace lqcd
