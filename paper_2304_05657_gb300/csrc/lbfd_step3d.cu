// lbfd_step3d.cu -- launchers of the 3-D (D3Q27) tile kernels.
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

// z-planes a block marches through, at most zmax: the cost of a launch is
// (planes + the ring's fill of 4 staged planes, ~0.15 of a plane's work
// each) times the larger of the blocks of the fullest SM (its issue slots or
// FP64 pipe are shared) and the waves of resident blocks times the factor by
// which a block alone on an SM is slower than its share of a full one.
// Without it a 101x53x47 FP64 grid ran as 168 blocks of 16 planes (two on
// 16 of the 152 SMs), a 128x64x64 FP32 grid as 128 of 32 planes or 256 of
// 16; now as 147 of 16 and 512 of 8.
static int planes_per_block(bool fp64, long long columns, int nz, int zmax)
{
    const double fill = 4 * 0.15, alone = fp64 ? 1.3 : 2.3;
    const long long sms = 152, resident = sms * (fp64 ? 2 : 4);
    int best = 1;
    double cost = 1e300;
    for (int z = nz < zmax ? nz : zmax; z >= 1; --z) {
        const long long blocks = columns * ((nz + z - 1) / z);
        const double c = (z + fill) * fmax((double)((blocks + sms - 1) / sms),
                                           alone * (double)((blocks + resident - 1) / resident));
        if (c < cost * 0.999) {
            cost = c;
            best = z;
        }
    }
    return best;
}

// The interior cells go to the tile kernel; on the side stream (same input
// state, disjoint writes) the cells near inlet and outlet faces go through
// their coded neighbourhoods (b.face_coded) and the general form takes the
// other cells near domain faces (b.face), and the cells next to in-domain
// solids (b.wall) go through their coded neighbourhoods (or, with curved
// walls, the general form with the face rules compiled out).
// the tile kernel instance: MINB > 0 caps its registers for MINB blocks per SM
template <typename S, typename R, int TX, int TY, int MINB, bool HI1>
static auto tile3_kernel()
{
    if constexpr (MINB > 0) return step_kernel_tiled3d_capped<S, R, TX, TY, MINB, HI1>;
    else return step_kernel_tiled3d<S, R, TX, TY, HI1>;
}

// SPLIT: the tile kernel does a1-a7 and a per-cell kernel a8-a10 (two
// smaller kernels instead of one; Lambda and grad rho pass through aux)
// WALLS: the wall-aware tile kernel also updates the cells next to
// in-domain solids, so the wall list runs only with curved walls
template <bool HI1, typename S, typename R, int MINB = 0, bool SPLIT = false, bool WALLS = false>
static cudaError_t launch_t3(int zmax, const StepParams<R>& P, StateView in, StateView out, const uint8_t* solid,
                             const BoundaryLists& bin, const SideStream& side, cudaStream_t stream)
{
    constexpr int TX = Tile3Shape<R>::TX, TY = Tile3Shape<R>::TY;
    constexpr size_t smem = tile3_smem_bytes<R, TX, TY>();
    auto kern = tile3_kernel<S, R, TX, TY, MINB, HI1>();
    auto fkern = step_kernel_fd3d<S, R, TX, TY>;
    auto wkern = step_kernel_tiled3d_walls<S, R, TX, TY, HI1>;
    auto fcode = step_kernel_wallcode<3, S, R, true, HI1>;
    auto wcode = step_kernel_wallcode<3, S, R, false, HI1>;
    cudaError_t e = SPLIT   ? cudaFuncSetAttribute(fkern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)
                    : WALLS ? cudaFuncSetAttribute(wkern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)
                            : cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (bin.interior == nullptr || (SPLIT && bin.aux == nullptr)) return cudaErrorInvalidValue;
    BoundaryLists b = bin;
    if (WALLS && !P.curved) b.nwall = 0;
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
                                                    (S*)out.Y, b.interior, (R*)b.aux);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        step_kernel_collide3d<S, R, HI1><<<dim3((P.nx + 127) / 128, P.ny, P.nz), 128, 0, stream>>>(
            P, (const S*)in.g, (S*)out.g, (const S*)in.T, (const S*)in.Y, b.interior, (const R*)b.aux);
    } else if constexpr (WALLS) {
        wkern<<<grid, dim3(TX, TY), smem, stream>>>(P, zc, (const S*)in.g, (S*)out.g, (const S*)in.T, (S*)out.T,
                                                    (const S*)in.Y, (S*)out.Y, b.interior, solid);
    } else {
        kern<<<grid, dim3(TX, TY), smem, stream>>>(P, zc, (const S*)in.g, (S*)out.g, (const S*)in.T, (S*)out.T,
                                                   (const S*)in.Y, (S*)out.Y, b.interior);
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
    switch (variant) {
    case 1: return launch_t3<HI1, S, R>(16, P, in, out, solid, b, side, stream);
    case 2: return launch_t3<HI1, S, R>(32, P, in, out, solid, b, side, stream);
    // variant 3: as 1 with the registers capped for four blocks per SM (FP32)
    case 3: return launch_t3<HI1, S, R, sizeof(R) == 4 ? 4 : 0>(16, P, in, out, solid, b, side, stream);
    // variants 4, 5: as 1, 2 split into an FD tile kernel and a collision kernel
    case 4: return launch_t3<HI1, S, R, 0, true>(16, P, in, out, solid, b, side, stream);
    case 5: return launch_t3<HI1, S, R, 0, true>(32, P, in, out, solid, b, side, stream);
    // variants 6, 7: as 1, 2 with the cells next to in-domain solids in the
    // tile kernel (wall-aware), no wall list
    case 6: return launch_t3<HI1, S, R, 0, false, true>(16, P, in, out, solid, b, side, stream);
    case 7: return launch_t3<HI1, S, R, 0, false, true>(32, P, in, out, solid, b, side, stream);
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
