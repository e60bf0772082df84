// lbfd_step_small.cu -- a 2-D step in one launch for grids too small to
// fill the GPU: FP64 and mixed forms, and the rule that picks it.
#include "lbfd_step_small.cuh"

namespace lbfd {

// The rule, in warps of 32 cells against the 608 SM partitions of the GPU
// (us per step of an isothermal channel in a graph; big = the best of the
// variants' tiles with their list kernel):
//   FP32 cells     8192  32768  65536  98304 131072 196608 262144
//     two lanes     5.9    6.8    7.4    9.1   11.0   15.3   19.6
//     one lane      7.2    7.6    8.5    9.2   10.1   12.0   14.9
//     big           7.6    7.7    9.2   12.4   12.6   12.7   15.6
//   FP64 cells     4096   8192  12288  16384  32768  98304 262144
//     two lanes    26.1   27.8   35.1   42.6   79.2    210    532
//     one lane     37.2   37.4   37.4   40.6   65.3    176    401
//     big          38.7   38.6   38.6   57.7   73.1    188    421
// Two lanes per cell as long as the partitions hold few warps each: FP64 (one
// instruction per 64 cycles and partition) at most one, FP32 (latency) five.
// One lane per cell up to 16 (FP32; beyond, the packed pairs' fewer
// instructions win) or 32 (FP64; beyond, the larger tiles' smaller halo).
bool small2d_applies(int precision, int nx, int ny, const BoundaryLists& b)
{
    return b.all2.nrest == 0 && small_warps(nx, ny) <= PARTITIONS * (precision == 0 ? 32 : 16);
}

cudaError_t launch_step_small2d(int precision, const StepParams<double>& Pd, const StepParams<float>& Pf, StateView in,
                                StateView out, const BoundaryLists& b, cudaStream_t stream)
{
    const long long w = small_warps(Pd.nx, Pd.ny);
    auto run = [&](const auto& P, auto zero, bool split) {
        using R = decltype(zero);
        if (P.omega_hi == R(1))
            return split ? launch_small<R, R, true, true>(P, in, out, b, stream)
                         : launch_small<R, R, true, false>(P, in, out, b, stream);
        return split ? launch_small<R, R, false, true>(P, in, out, b, stream)
                     : launch_small<R, R, false, false>(P, in, out, b, stream);
    };
    return precision == 0 ? run(Pd, 0.0, 3 * w <= 2 * PARTITIONS) : run(Pf, 0.f, w <= 5 * PARTITIONS);
}

}  // namespace lbfd
