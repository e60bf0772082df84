// The 3-D tile kernel's cell of an in-plane byte offset (cell_at), for FP32 and
// FP64 planes of up to the largest grids that fit the device: prints the number
// of cells for which it is not the cell itself.  Built and run on the CPU by
// tests/test_plane_offsets_host.py; no GPU call is made.
#include <cstdio>

#include "lbfd_step_tiled3d.cuh"

template <typename S>
static int wrong(long long cells)
{
    int n = 0;
    const long long last = cells - 1, probe[] = {0, 1, 31, last / 4, last / 2 - 1, last / 2, last / 2 + 1, last - 1, last};
    for (const long long base : {0ll, 7 * cells})
        for (const long long c : probe) n += lbfd::cell_at<S>(base, (unsigned)(c * (long long)sizeof(S))) != base + c;
    return n;
}

int main()
{
    // planes of 2^18 cells (512x512), and the largest: 2^30 FP32, 2^29 FP64
    printf("%d %d\n", wrong<float>(1ll << 18) + wrong<double>(1ll << 18), wrong<float>(1ll << 30) + wrong<double>(1ll << 29));
    return 0;
}
