// lbfd_step3d.cu -- launchers of the 3-D (D3Q27) tile kernels.
#include <algorithm>
#include <cmath>

#include "lbfd_internal.h"
#include "lbfd_step_tiled3d.cuh"

namespace lbfd {

// block shape: 32x4 cells in FP32 (a warp reads whole 128-byte row
// segments), 16x8 in FP64 (240 staged points per 128 cells instead of 288,
// and less padding on ragged grids; its loads are not the bound)
template <typename R>
struct Tile3Shape {
    static constexpr int TX = sizeof(R) == 8 ? 16 : 32, TY = 128 / TX;
};

// z-planes a block marches through, at most zmax.  Few planes per block
// balance the SMs and keep their blocks resident together; each block pays
// for 4 staged planes more (~0.2 of a plane's work each).  A step is
// modelled from the measured us per plane of 1 .. R blocks sharing an SM (R
// resident): blocks in rounds of R on the fullest SM, or, with many rounds,
// the steady rate and half a round of tail.  Measured us per step over z:
//   128x64x64 FP32:   4: 91   7: 85   8: 94   9: 100  16: 139   (picks 7)
//   256x128x128 FP32: 4: 511  5: 496  7: 494  8: 500  11: 490  16: 527   (5)
//   101x53x47 FP64:   4: 941  5: 1087 7: 1143 8: 941  9: 1057  16: 1049   (8)
//   128x64x64 FP64:   4: 1714 5: 1680 7: 1646 8: 1859 9: 1978  16: 1985   (9)
// The last pick is the model's error: three FP64 blocks on an SM that holds two
// take about 194 us a plane, not 109 + 63.
static int planes_per_block(bool fp64, long long columns, int nz, int zmax)
{
    static const double us32[] = {0.0, 6.4, 7.9, 9.4, 10.9}, us64[] = {0.0, 63.0, 109.0};
    const double* us = fp64 ? us64 : us32;
    const int R = fp64 ? 2 : 4;
    const double steady = fp64 ? 109.0 : 8.4, sms = 152.0, fill = 4 * 0.2;
    // (fewer than 4 measured slower; and a grid has at most 65535 pieces)
    const int top = nz < zmax ? nz : zmax, enough = (nz + 65534) / 65535;
    const int low = std::min(top, std::max(4, enough));
    double cost[64], least = 1e300;
    for (int z = low; z <= top; ++z) {
        const double n = (double)columns * nz / z / sms;  // blocks per SM
        double t;
        if (n > 2 * R) {
            t = (n / R * steady + 0.5 * us[R]) * (z + fill);
        } else {  // whole pieces, then the last, shorter ones
            const int full = (int)ceil((double)columns * (nz / z) / sms);
            const int all = (int)ceil((double)columns * ((nz + z - 1) / z) / sms);
            auto rounds = [&](int k) { return k / R * us[R] + us[k % R]; };
            t = rounds(full) * (z + fill) + (rounds(all) - rounds(full)) * (nz % z + fill);
        }
        cost[z] = t;
        least = t < least ? t : least;
    }
    int best = low;  // the fewest planes within the model's accuracy
    while (cost[best] > 1.02 * least) ++best;
    return best;
}

// The interior cells go to the tile kernel; on the side stream (same input
// state, disjoint writes) the cells near inlet and outlet faces go through
// their coded neighbourhoods (b.face_coded) and the general form takes the
// other cells near domain faces (b.face), and the cells next to in-domain
// solids (b.wall) go through their coded neighbourhoods (or, with curved
// walls, the general form with the face rules compiled out).
// SPLIT: the tile kernel does a1-a7 and a per-cell kernel a8-a10 (two
// smaller kernels instead of one; Lambda and grad rho pass through aux)
// Otherwise the tile kernel updates the coded cells too, next to in-domain
// solids and (faces) near inlet and outlet faces; with curved walls both
// go through the general form.
// zmax: the most planes per block; variants that differ only in it (16 or 32)
// are one kernel with the same or, on large grids, a few more planes
// (512x256x256 FP32: 10 and 11).
// MINB: resident blocks per SM.  FP32: four (128 registers) when the
// collision needs only the low moments, else three; FP64: two.
template <bool HI1, typename S, typename R, int MINB, bool SPLIT = false>
static cudaError_t launch_t3(int zmax, bool faces, const StepParams<R>& P, StateView in, StateView out, const uint8_t* solid,
                             const BoundaryLists& bin, const SideStream& side, cudaStream_t stream)
{
    constexpr int TX = Tile3Shape<R>::TX, TY = Tile3Shape<R>::TY;
    constexpr size_t smem = tile3_smem_bytes<R, TX, TY>();
    auto kern = step_kernel_tiled3d<S, R, TX, TY, MINB, HI1>;
    auto fkern = step_kernel_fd3d<S, R, TX, TY>;
    auto fcode = step_kernel_wallcode<3, S, R, true, HI1>;
    auto wcode = step_kernel_wallcode<3, S, R, false, HI1>;
    cudaError_t e = SPLIT ? cudaFuncSetAttribute(fkern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)
                          : cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (bin.words == nullptr || (SPLIT && bin.aux == nullptr)) return cudaErrorInvalidValue;
    BoundaryLists b = bin;
    if (!SPLIT && !P.curved) {
        b.nwall = 0;
        if (faces) b.nface_coded = b.nface_tile;
    }
    const bool fork = (b.nface > 0 || b.nface_coded > 0 || b.nwall > 0) && side.stream != nullptr;
    if (fork) {
        if ((e = cudaEventRecord(side.fork, stream)) != cudaSuccess) return e;
        if ((e = cudaStreamWaitEvent(side.stream, side.fork, 0)) != cudaSuccess) return e;
    }
    cudaStream_t bs = fork ? side.stream : stream;
    const int prio = fork ? side.priority : 0;
    if (b.nface > 0) {
        const unsigned nb = (unsigned)((b.nface + 127) / 128);
        e = launch_prio(step_kernel_boundary<3, S, R, true, HI1>, dim3(nb), dim3(128), 0, bs, prio, P, (const S*)in.g,
                        (S*)out.g, (const S*)in.T, (S*)out.T, (const S*)in.Y, (S*)out.Y, solid, b.face, b.nface);
        if (e != cudaSuccess) return e;
    }
    if (b.nface_coded > 0) {  // cells near inlet/outlet faces with their codes
        const unsigned nb = (unsigned)((b.nface_coded + 127) / 128);
        e = launch_prio(fcode, dim3(nb), dim3(128), 0, bs, prio, P, (const S*)in.g,
                        (S*)out.g, (const S*)in.T, (S*)out.T, (const S*)in.Y, (S*)out.Y, b.face_coded, b.face_code,
                        b.nface_coded);
        if (e != cudaSuccess) return e;
    }
    if (b.nwall > 0) {
        const unsigned nb = (unsigned)((b.nwall + 127) / 128);
        if (!P.curved && b.wall_code != nullptr)  // staircase walls: the coded neighbourhoods
            e = launch_prio(wcode, dim3(nb), dim3(128), 0, bs, prio, P, (const S*)in.g,
                            (S*)out.g, (const S*)in.T, (S*)out.T, (const S*)in.Y, (S*)out.Y, b.wall, b.wall_code,
                            b.nwall);
        else
            e = launch_prio(step_kernel_boundary<3, S, R, false, HI1>, dim3(nb), dim3(128), 0, bs, prio, P,
                            (const S*)in.g, (S*)out.g, (const S*)in.T, (S*)out.T, (const S*)in.Y, (S*)out.Y, solid,
                            b.wall, b.nwall);
        if (e != cudaSuccess) return e;
    }
    dim3 grid((P.nx + TX - 1) / TX, (P.ny + TY - 1) / TY);
    const int zc = planes_per_block(sizeof(R) == 8, (long long)grid.x * grid.y, P.nz, zmax);
    grid.z = (P.nz + zc - 1) / zc;
    if constexpr (SPLIT) {
        fkern<<<grid, dim3(TX, TY), smem, stream>>>(P, zc, (const S*)in.g, (const S*)in.T, (S*)out.T, (const S*)in.Y,
                                                    (S*)out.Y, b.words, (R*)b.aux);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        step_kernel_collide3d<S, R, HI1><<<dim3((P.nx + 127) / 128, P.ny, P.nz), 128, 0, stream>>>(
            P, (const S*)in.g, (S*)out.g, (const S*)in.T, (const S*)in.Y, b.words, (const R*)b.aux);
    } else {
        kern<<<grid, dim3(TX, TY), smem, stream>>>(P, zc, (const S*)in.g, (S*)out.g, (const S*)in.T, (S*)out.T,
                                                   (const S*)in.Y, (S*)out.Y, b.words, P.curved ? 0 : (faces ? 2 : 1));
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (fork) {
        if ((e = cudaEventRecord(side.join, side.stream)) != cudaSuccess) return e;
        if ((e = cudaStreamWaitEvent(stream, side.join, 0)) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// HI1: omega_hi = 1 (the collision from the moments of orders 0-2)
template <bool HI1, typename S, typename R>
static cudaError_t launch_3d_tiles(int variant, const StepParams<R>& P, StateView in, StateView out,
                                   const uint8_t* solid, const BoundaryLists& b, const SideStream& side,
                                   cudaStream_t stream)
{
    constexpr int MINB = sizeof(R) == 8 ? 2 : (HI1 ? 4 : 3);
    switch (variant) {
    case 1: return launch_t3<HI1, S, R, MINB>(16, true, P, in, out, solid, b, side, stream);
    case 2: return launch_t3<HI1, S, R, MINB>(32, true, P, in, out, solid, b, side, stream);
    // variant 3: FP32 with omega_hi != 1 at four blocks per SM (128 registers)
    // instead of three; elsewhere the same as 1
    case 3: return launch_t3<HI1, S, R, sizeof(R) == 4 ? 4 : 2>(16, true, P, in, out, solid, b, side, stream);
    // variants 4, 5: as 1, 2 split into an FD tile kernel and a collision kernel
    case 4: return launch_t3<HI1, S, R, MINB, true>(16, false, P, in, out, solid, b, side, stream);
    case 5: return launch_t3<HI1, S, R, MINB, true>(32, false, P, in, out, solid, b, side, stream);
    // variants 6, 7: as 1, 2 with the cells near open faces in a list kernel
    // of their own
    case 6: return launch_t3<HI1, S, R, MINB>(16, false, P, in, out, solid, b, side, stream);
    case 7: return launch_t3<HI1, S, R, MINB>(32, false, P, in, out, solid, b, side, stream);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_step3d_tiled(int precision, int variant, const StepParams<double>& Pd, const StepParams<float>& Pf,
                                StateView in, StateView out, const uint8_t* solid, const BoundaryLists& b,
                                const SideStream& side, cudaStream_t stream)
{
    if (precision == 0) {
        if (Pd.omega_hi == 1.0) return launch_3d_tiles<true, double, double>(variant, Pd, in, out, solid, b, side, stream);
        return launch_3d_tiles<false, double, double>(variant, Pd, in, out, solid, b, side, stream);
    }
    if (Pf.omega_hi == 1.f) return launch_3d_tiles<true, float, float>(variant, Pf, in, out, solid, b, side, stream);
    return launch_3d_tiles<false, float, float>(variant, Pf, in, out, solid, b, side, stream);
}

}  // namespace lbfd
