// Launcher of the paired (two right-hand sides per thread, packed FP32x2)
// hopping kernel; included by one translation unit per storage precision.
#pragma once
#include "hopfast.cuh"
#include "lqcd_impl.h"

namespace lqcd {

template <class S, int MODE, bool DAG, bool NORM>
static void hopp_go(const FastHop<S> &f, cudaStream_t st)
{
    const int ngr = (f.nrhs + 1) / 2;
    const unsigned grid = unsigned(padded_tiles(f) * ((ngr + f.gpb - 1) / f.gpb));
    if (f.minb >= 4)
        hopp_kernel<S, MODE, DAG, NORM, 4><<<grid, kBlock, 0, st>>>(f);
    else if (f.minb == 3)
        hopp_kernel<S, MODE, DAG, NORM, 3><<<grid, kBlock, 0, st>>>(f);
    else
        hopp_kernel<S, MODE, DAG, NORM, 1><<<grid, kBlock, 0, st>>>(f);
}

template <class S, int MODE>
static void hopp_mode(const FastHop<S> &f, bool dag, bool norm, cudaStream_t st)
{
    if (dag) norm ? hopp_go<S, MODE, true, true>(f, st) : hopp_go<S, MODE, true, false>(f, st);
    else norm ? hopp_go<S, MODE, false, true>(f, st) : hopp_go<S, MODE, false, false>(f, st);
}

template <class S>
void hopp_dispatch(const FastHop<S> &f, int mode, bool dag, bool norm, cudaStream_t st)
{
    switch (mode) {
    case HOP_CLOV: hopp_mode<S, HOP_CLOV>(f, dag, norm, st); break;
    case SELF_CLOV: hopp_mode<S, SELF_CLOV>(f, dag, norm, st); break;
    case HOP_CLOV + TWIST: hopp_mode<S, HOP_CLOV + TWIST>(f, dag, norm, st); break;
    default: hopp_mode<S, SELF_CLOV + TWIST>(f, dag, norm, st); break;
    }
}

}  // namespace lqcd
