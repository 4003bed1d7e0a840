// dslash_f64_apply.cu -- the operator applications' hop kernels: both parities
// in one grid, on the caller's canonical fields.
#include "blas.h"
#include "dslash_launch.cuh"

namespace eofa {
cudaError_t launch_apply_f64(int kind, const HopPair& p, const SCoef<double>& c, cudaStream_t st) {
    switch (p.a[0].g.Ls) {
        case 4: return launch_pair_ls<4>(kind, p, c, st);
        case 8: return launch_pair_ls<8>(kind, p, c, st);
        case 12: return launch_pair_ls<12>(kind, p, c, st);
        case 16: return launch_pair_ls<16>(kind, p, c, st);
        default: return cudaErrorNotSupported;
    }
}
// once per device, so that an application can be captured whatever ran before
cudaError_t setup_apply_f64(int Ls, cudaStream_t st) {
    switch (Ls) {
        case 4: return setup_apply_ls<4>(st);
        case 8: return setup_apply_ls<8>(st);
        case 12: return setup_apply_ls<12>(st);
        case 16: return setup_apply_ls<16>(st);
        default: return cudaErrorNotSupported;
    }
}
}  // namespace eofa
