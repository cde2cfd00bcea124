// ea_server_general.cuh -- launches of the staged server where a message has several scales per tile
// (PASS_SHORT) or one for several tiles, in translation units of their own.
#pragma once

#include "ea_server.cuh"

namespace ea {

// (instantiated in ea_server_general_<mode>_q<QS>.cu).
template <int MODE, int QS>
cudaError_t launch_server_general(const ServerArgs &a, cudaStream_t s)
{
    switch (a.qw.kind) {
    case QK_SIGN: return launch_server_staged_kernel<MODE, QK_SIGN, QS, true>(a, s);
    case QK_UNIF: return launch_server_staged_kernel<MODE, QK_UNIF, QS, true>(a, s);
    case QK_POW2:  // without scales: the short blocks are Q_s's
        if constexpr (has_scale<QS>()) return launch_server_staged_kernel<MODE, QK_POW2, QS, true>(a, s);
        return cudaErrorNotSupported;
    default:
        if constexpr (has_scale<QS>()) return launch_server_staged_kernel<MODE, QK_IDENT, QS, true>(a, s);
        return cudaErrorNotSupported;
    }
}

}  // namespace ea
