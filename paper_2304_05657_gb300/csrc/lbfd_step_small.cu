// lbfd_step_small.cu -- a 2-D step in one launch for grids too small to
// fill the GPU: FP64 and mixed forms, and the rule that picks it.
#include "lbfd_step_small.cuh"

namespace lbfd {

// The rules, in warps of 32 cells against the 608 SM partitions of the GPU
// (us per step of an isothermal channel in a graph).  Lanes per cell: two as
// long as that leaves the partitions at most one warp each.
//   FP32 cells     8192  12288  32768    FP64 cells     4096   8192  12288  16384
//     two lanes     4.8    5.0    6.1      two lanes    25.6   27.8   35.8   40.4
//     one lane      5.0    5.0    5.4      one lane     35.8   35.5   35.7   38.0
// Against the tiles of variants 1 (32x8) and 2 (32x4):
//   FP32 cells   8192 16384 32768 49152 57344 65536 73728 81920 98304 155648
//     small       4.6   5.0   5.4   6.2   6.4   7.0   6.9   7.6   9.8   12.1
//     variant 1   4.9   5.2   5.2   6.2   6.4   6.6   6.2   7.7   7.8    9.6
//     variant 2   4.7   4.9   5.5   5.8   5.9   6.5   6.4   7.1   7.8    9.9
//   FP64 cells  24576 32768 40960 49152 65536 73728 81920 98304 131072 163840 204800 245760 262144 409600
//     small        52    59    76    87   126   151   154   184    213    272    330    389    417    649
//     variant 1    65    65   122   122   127   122   180   179    236    297    350    407    410    635
//     variant 2    64    67    92    95   127   124   151   180    210    268    326    384    413    638
// and with many cells next to walls (us per pass): 86 271 cells of channels
// between solid rows, FP32, 24 steps: small 268, variant 1 300; 522 880 cells of
// a burner, FP64, 4 steps: 3 359, 3 646.  No one line is right for both kinds, so
// variants 2-4 run their own tiles beyond one warp a partition where these are
// one launch too (no cell for a list): with variant 1, the default, as the small
// form the autotuner has both to choose from.  Variant 1 and 5-12 (a list beside
// the tiles) are the small form up to 8 warps a partition in FP32 and 32 in FP64.
// There 5-12 are slower in FP32 (98304 cells 11.6-13.8 us, 155648 13.5-14.5) and
// mostly in FP64 (131072 cells 230-260, 196608 319-350, 262144 423), where they
// take 60 or 115 us on 32768 cells by the order in which the two kernels' blocks
// are placed: a few timed launches do not tell.
bool small2d_applies(int precision, int variant, int nx, int ny, const BoundaryLists& b)
{
    const bool own = variant >= 2 && variant <= 4 && b.all2.nout == 0;
    return b.all2.nrest == 0 && small_warps(nx, ny) <= PARTITIONS * (own ? 1 : (precision == 0 ? 32 : 8));
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
