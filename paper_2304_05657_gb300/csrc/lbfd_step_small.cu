// lbfd_step_small.cu -- a 2-D step in one launch for grids too small to
// fill the GPU: FP64 and mixed forms, and the rule that picks it.
#include "lbfd_step_small.cuh"

namespace lbfd {

// The rule, in warps of 32 cells against the 608 SM partitions of the GPU
// (us per step of an isothermal channel in a graph; big = the best of the
// variants' tiles):
//   FP32 cells     8192  12288  32768  65536  98304 131072 196608 262144
//     two lanes     4.8    5.0    6.1    9.2   11.2   13.8   18.7   23.6
//     one lane      5.0    5.0    5.4    6.9    9.8   10.8   14.6   17.4
//     big           6.7    7.1    7.2    9.6    9.4   11.5   12.4   15.9
//   FP64 cells     4096   8192  12288  16384  32768  98304 262144
//     two lanes    25.6   27.8   35.8   40.4   85.7    221    536
//     one lane     35.8   35.5   35.7   38.0   58.6    183    415
//     big          36.5   36.5   36.5   36.5   65.4    178    408
// Two lanes per cell as long as that leaves the partitions at most one warp
// each.  One lane per cell up to 8 warps (FP32; beyond, the larger tiles'
// smaller halo and the packed pairs win) or 32 (FP64; beyond, the halo).
bool small2d_applies(int precision, int nx, int ny, const BoundaryLists& b)
{
    return b.all2.nrest == 0 && small_warps(nx, ny) <= PARTITIONS * (precision == 0 ? 32 : 8);
}

cudaError_t launch_step_small2d(int precision, const StepParams<double>& Pd, const StepParams<float>& Pf, StateView in,
                                StateView out, const BoundaryLists& b, cudaStream_t stream)
{
    const long long w = small_warps(Pd.nx, Pd.ny);
    const bool split = 2 * w <= PARTITIONS;
    auto run = [&](const auto& P, auto zero) {
        using R = decltype(zero);
        if (P.omega_hi == R(1))
            return split ? launch_small<R, R, true, true>(P, in, out, b, stream)
                         : launch_small<R, R, true, false>(P, in, out, b, stream);
        return split ? launch_small<R, R, false, true>(P, in, out, b, stream)
                     : launch_small<R, R, false, false>(P, in, out, b, stream);
    };
    return precision == 0 ? run(Pd, 0.0) : run(Pf, 0.f);
}

}  // namespace lbfd
