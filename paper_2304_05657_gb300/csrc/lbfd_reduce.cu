// lbfd_reduce.cu -- FP64 reductions over the fluid cells (flame position,
// mass, heat release, fuel consumption, max T, non-finite count) and the
// per-cell field read-out kernel.
//
// Observables: flame front by maximum heat release (Sec. IV.A dead-zone
// analysis; Sec. IV.B burner), consumption speed integrals (Sec. IV.C,
// Eq. 40), and an integral flame position (unburnt length).
#include <cmath>

#include "lbfd_device.cuh"
#include "lbfd_internal.h"

namespace lbfd {

__device__ __forceinline__ unsigned long long order_key(double v)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

template <typename S>
__device__ __forceinline__ double hrr_of(const StepParams<double>& P, double T, const double* Y, double* rho_out,
                                         double* q_out)
{
    double invW = 0.0;
#pragma unroll
    for (int k = 0; k < NSP; ++k) invW += Y[k] * P.inv_Wk[k];
    const double rho = P.T_in * P.invW_in / (T * invW);
    const double yf = Y[P.fuel] > 0.0 ? Y[P.fuel] : 0.0;
    const double yo = Y[P.oxid] > 0.0 ? Y[P.oxid] : 0.0;
    const double q = P.A_lat * yf * yo * ::exp(-P.Ta / T);
    *rho_out = rho;
    *q_out = q;
    return rho * P.Q_cp * q;
}

// Heat-release maximum on the line y = (y0 + y1)/2, z = nz/2 by one block of
// 256 threads: red[8] = value, red[9] = its x (the smaller on ties).
template <int DIM, typename S>
__device__ void centreline(const StepParams<double>& P, const S* __restrict__ T, const S* __restrict__ Y,
                           const uint8_t* __restrict__ solid, int y0, int y1, double* red)
{
    double best = -INFINITY;
    int bx = -1;
    const int yc = (y0 + y1) / 2, zc = DIM == 3 ? P.nz / 2 : 0;
    for (int x = threadIdx.x; x < P.nx; x += blockDim.x) {
        const long long c = x + (long long)P.nx * (yc + (long long)P.ny * zc);
        if (solid[c]) continue;
        const double Tc = val(T[c]);
        double Yc[NSP];
        bool bad = !isfinite(Tc);
#pragma unroll
        for (int k = 0; k < NSP; ++k) {
            Yc[k] = val(Y[(long long)k * P.N + c]);
            bad |= !isfinite(Yc[k]);
        }
        if (bad) continue;
        double rho, q;
        const double h = hrr_of<S>(P, Tc, Yc, &rho, &q);
        if (h > best) {  // x increases along the loop: ties keep the smaller x
            best = h;
            bx = x;
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const double ob = __shfl_down_sync(0xffffffffu, best, off);
        const int ox = __shfl_down_sync(0xffffffffu, bx, off);
        if (ox >= 0 && (bx < 0 || ob > best || (ob == best && ox < bx))) {
            best = ob;
            bx = ox;
        }
    }
    __shared__ double sb[32];
    __shared__ int sx[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) {
        sb[wid] = best;
        sx[wid] = bx;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const int nw = blockDim.x >> 5;
        for (int w = 1; w < nw; ++w) {
            if (sx[w] >= 0 && (bx < 0 || sb[w] > best || (sb[w] == best && sx[w] < bx))) {
                best = sb[w];
                bx = sx[w];
            }
        }
        red[8] = best;
        red[9] = (double)bx;
    }
}

// red layout: [0] sum Y_F, [1] mass, [2] hrr, [3] fuel, [4] max-T key (u64),
// [5] non-finite count (u64), [6] fluid count (u64), [7] x=0 section count (u64),
// [8] centre-line max hrr, [9] its x, [10] count of finished blocks (u32,
// back to 0 at the end).  With `part` (8 words per block) the block sums are
// stored there and the last block adds them in block order, so that the
// result does not depend on the order in which blocks finish; without it
// (the fixed scratch of the allocation-free form) they are added to `red`
// atomically.  Block 0 scans the centre line meanwhile (a serial chain of FP64
// work on one SM: after the sums it would add 10 to 20 us where nx is 1024 and
// more); the others take the sums: one launch.
template <int DIM, typename S>
__global__ void __launch_bounds__(256) diag_kernel(StepParams<double> P, const S* __restrict__ g,
                                                   const S* __restrict__ T, const S* __restrict__ Y,
                                                   const uint8_t* __restrict__ solid, int y0, int y1, double* red,
                                                   double* part)
{
    constexpr int Q = DIM == 2 ? 9 : 27;
    if (blockIdx.x == 0) {
        centreline<DIM, S>(P, T, Y, solid, y0, y1, red);
        return;
    }
    const unsigned nsum = gridDim.x - 1, self = blockIdx.x - 1;
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    unsigned long long tkey = 0ull, nonf = 0ull, nfl = 0ull, sec = 0ull;
    const long long stride = (long long)nsum * blockDim.x;
    const int rows = y1 - y0;
    const long long ncount = (long long)P.nx * rows * P.nz;  // cells with y0 <= y < y1
    for (long long t = (long long)self * blockDim.x + threadIdx.x; t < ncount; t += stride) {
        const long long r = t / P.nx;
        const long long c = t % P.nx + (long long)P.nx * (y0 + r % rows + (long long)P.ny * (r / rows));
        if (solid[c]) continue;
        ++nfl;
        if (c % P.nx == 0) ++sec;
        const double Tc = val(T[c]);
        double Yc[NSP];
        bool bad = !isfinite(Tc);
#pragma unroll
        for (int k = 0; k < NSP; ++k) {
            Yc[k] = val(Y[(long long)k * P.N + c]);
            bad |= !isfinite(Yc[k]);
        }
#pragma unroll
        for (int i = 0; i < Q; ++i) bad |= !isfinite(val(g[(long long)i * P.N + c]));
        if (bad) {
            ++nonf;
            continue;
        }
        double rho, q;
        const double h = hrr_of<S>(P, Tc, Yc, &rho, &q);
        s[0] += Yc[P.fuel];
        s[1] += rho;
        s[2] += h;
        s[3] += rho * q;
        const unsigned long long k = order_key(Tc);
        tkey = k > tkey ? k : tkey;
    }
    // warp then block reduction
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
        for (int j = 0; j < 4; ++j) s[j] += __shfl_down_sync(0xffffffffu, s[j], off);
        const unsigned long long o = __shfl_down_sync(0xffffffffu, tkey, off);
        tkey = o > tkey ? o : tkey;
        nonf += __shfl_down_sync(0xffffffffu, nonf, off);
        nfl += __shfl_down_sync(0xffffffffu, nfl, off);
        sec += __shfl_down_sync(0xffffffffu, sec, off);
    }
    __shared__ double sh[8][4];
    __shared__ unsigned long long shk[8][4];
    __shared__ bool last;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) {
#pragma unroll
        for (int j = 0; j < 4; ++j) sh[wid][j] = s[j];
        shk[wid][0] = tkey;
        shk[wid][1] = nonf;
        shk[wid][2] = nfl;
        shk[wid][3] = sec;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const int nw = blockDim.x >> 5;
        for (int w = 1; w < nw; ++w) {
            for (int j = 0; j < 4; ++j) s[j] += sh[w][j];
            tkey = shk[w][0] > tkey ? shk[w][0] : tkey;
            nonf += shk[w][1];
            nfl += shk[w][2];
            sec += shk[w][3];
        }
        unsigned long long* ru = reinterpret_cast<unsigned long long*>(red);
        if (part) {
            double* pb = part + 8 * (size_t)self;
            unsigned long long* pu = reinterpret_cast<unsigned long long*>(pb);
            for (int j = 0; j < 4; ++j) pb[j] = s[j];
            pu[4] = tkey;
            pu[5] = nonf;
            pu[6] = nfl;
            pu[7] = sec;
        } else {
            for (int j = 0; j < 4; ++j) atomicAdd(&red[j], s[j]);
            atomicMax(&ru[4], tkey);
            atomicAdd(&ru[5], nonf);
            atomicAdd(&ru[6], nfl);
            atomicAdd(&ru[7], sec);
        }
        __threadfence();  // this block's sums before its count
        last = atomicInc(reinterpret_cast<unsigned*>(&red[10]), nsum - 1) == nsum - 1;
    }
    __syncthreads();
    if (!last || !part) return;
    __threadfence();
    {
        // word j = thread % 8 of a run of consecutive blocks per thread, the 32
        // runs then joined in order
        __shared__ unsigned long long run[32][8];
        const int j = threadIdx.x & 7, r = threadIdx.x >> 3;
        const unsigned len = (nsum + 31) / 32;
        const unsigned long long* pu = reinterpret_cast<const unsigned long long*>(part) + j;
        auto join = [&](double& d, unsigned long long& u, unsigned long long w) {
            if (j < 4) d += __longlong_as_double((long long)w);
            else if (j == 4) u = w > u ? w : u;
            else u += w;
        };
        double d = 0.0;
        unsigned long long u = 0ull;
#pragma unroll 10
        for (unsigned k = 0; k < len; ++k) {
            const unsigned b = r * len + k;
            if (b < nsum) join(d, u, __ldcg(pu + 8 * (size_t)b));
        }
        run[r][j] = j < 4 ? (unsigned long long)__double_as_longlong(d) : u;
        __syncthreads();
        if (threadIdx.x < 8) {
            d = 0.0;
            u = 0ull;
            for (int k = 0; k < 32; ++k) join(d, u, run[k][j]);
            reinterpret_cast<unsigned long long*>(red)[j] = j < 4 ? (unsigned long long)__double_as_longlong(d) : u;
        }
    }
}

template <int DIM, typename S>
static cudaError_t diag_launch(const StepParams<double>& P, StateView st, const uint8_t* solid, int y0, int y1,
                               double* red, double* part, cudaStream_t stream)
{
    if (!part) {
        const cudaError_t e = cudaMemsetAsync(red, 0, RED_WORDS * sizeof(double), stream);
        if (e != cudaSuccess) return e;
    }
    const long long want = ((long long)P.nx * (y1 - y0) * P.nz + 255) / 256;
    const unsigned blocks = (unsigned)(want < DIAG_BLOCKS ? want : DIAG_BLOCKS) + 1;  // and the centre line's
    diag_kernel<DIM, S><<<blocks, 256, 0, stream>>>(P, (const S*)st.g, (const S*)st.T, (const S*)st.Y, solid, y0, y1,
                                                    red, part);
    return cudaGetLastError();
}

cudaError_t launch_diagnostics(int dim, int precision, const StepParams<double>& P, StateView st,
                               const uint8_t* solid, int y0, int y1, double* red, double* part, cudaStream_t stream)
{
    if (precision == 0)
        return dim == 2 ? diag_launch<2, double>(P, st, solid, y0, y1, red, part, stream)
                        : diag_launch<3, double>(P, st, solid, y0, y1, red, part, stream);
    if (precision == 2)
        return dim == 2 ? diag_launch<2, Tan>(P, st, solid, y0, y1, red, part, stream) : cudaErrorInvalidValue;
    if (precision == 3)
        return dim == 2 ? diag_launch<2, Tanf>(P, st, solid, y0, y1, red, part, stream) : cudaErrorInvalidValue;
    return dim == 2 ? diag_launch<2, float>(P, st, solid, y0, y1, red, part, stream)
                    : diag_launch<3, float>(P, st, solid, y0, y1, red, part, stream);
}

// Per column x of a 2-D grid: the peak heat release over the fluid cells of
// rows y0 <= y < y1 (the reaction front where it crosses the column, Sec.
// IV.A) and the distance of that cell's centre to the nearer edge of the
// row band (walls half-way between cells): out[x] = peak (0 when the column
// has no fluid cell there), out[nx + x] = distance (smallest y on ties).
// One warp per 32 columns and PEAK_ROWS rows (a cell's rate is about 70 FP64
// instructions of 64 cycles: a thread per column took 70 to 230 us for 17 to
// 65 rows), the chunks' maxima at part[chunk][2][nx]; then the maximum over
// the chunks in row order.
constexpr int PEAK_ROWS = 4;
template <typename S>
__global__ void __launch_bounds__(32) column_peaks_kernel(StepParams<double> P, const S* __restrict__ T,
                                                          const S* __restrict__ Y,
                                                          const uint8_t* __restrict__ solid, int y0, int y1,
                                                          double* __restrict__ part)
{
    const unsigned gx = (P.nx + 31) / 32;
    const int x = (int)(blockIdx.x % gx) * 32 + threadIdx.x, chunk = (int)(blockIdx.x / gx);
    if (x >= P.nx) return;
    const int ya = y0 + chunk * PEAK_ROWS, yb = ya + PEAK_ROWS < y1 ? ya + PEAK_ROWS : y1;
    double best = -1.0;
    int by = y0;
    for (int y = ya; y < yb; ++y) {
        const long long c = (long long)x + (long long)P.nx * y;
        if (solid[c]) continue;
        double Yc[NSP];
#pragma unroll
        for (int k = 0; k < NSP; ++k) Yc[k] = val(Y[(long long)k * P.N + c]);
        double rho, q;
        const double h = hrr_of<S>(P, val(T[c]), Yc, &rho, &q);
        if (h > best) {
            best = h;
            by = y;
        }
    }
    part[(size_t)(2 * chunk) * P.nx + x] = best;
    part[(size_t)(2 * chunk + 1) * P.nx + x] = (double)by;
}
__global__ void __launch_bounds__(128) column_peaks_join_kernel(int nx, int chunks, int y0, int y1,
                                                                const double* __restrict__ part,
                                                                double* __restrict__ out)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= nx) return;
    double best = -1.0, by = y0;
    for (int j = 0; j < chunks; ++j) {
        const double h = part[(size_t)(2 * j) * nx + x];
        if (h > best) {
            best = h;
            by = part[(size_t)(2 * j + 1) * nx + x];
        }
    }
    const double d0 = by - y0 + 0.5, d1 = y1 - 0.5 - by;
    out[x] = best < 0.0 ? 0.0 : best;
    out[nx + x] = d0 < d1 ? d0 : d1;
}

static int peak_chunks(int y0, int y1) { return (y1 - y0 + PEAK_ROWS - 1) / PEAK_ROWS; }
size_t column_peaks_words(int nx, int y0, int y1) { return (size_t)nx * (2 + 2 * (size_t)peak_chunks(y0, y1)); }

cudaError_t launch_column_peaks(int precision, const StepParams<double>& P, StateView st, const uint8_t* solid,
                                int y0, int y1, double* out, cudaStream_t stream)
{
    const int chunks = peak_chunks(y0, y1);
    const unsigned grid = (unsigned)((P.nx + 31) / 32) * (unsigned)chunks;
    double* part = out + 2 * (size_t)P.nx;
    if (precision == 0)
        column_peaks_kernel<double><<<grid, 32, 0, stream>>>(P, (const double*)st.T, (const double*)st.Y, solid, y0,
                                                             y1, part);
    else if (precision == 1)
        column_peaks_kernel<float><<<grid, 32, 0, stream>>>(P, (const float*)st.T, (const float*)st.Y, solid, y0, y1,
                                                            part);
    else
        return cudaErrorInvalidValue;
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    column_peaks_join_kernel<<<(unsigned)((P.nx + 127) / 128), 128, 0, stream>>>(P.nx, chunks, y0, y1, part, out);
    return cudaGetLastError();
}

// field ids follow include/lbfd.h
template <int DIM, typename S>
__global__ void __launch_bounds__(256) field_kernel(StepParams<double> P, const S* __restrict__ g,
                                                    const S* __restrict__ T, const S* __restrict__ Y,
                                                    const uint8_t* __restrict__ solid, int field,
                                                    double* __restrict__ out)
{
    constexpr int Q = DIM == 2 ? 9 : 27;
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= P.ncell) return;
    if (field >= 16) {
        out[c] = val(g[(long long)(field - 16) * P.N + c]);
        return;
    }
    if (field == 0) {
        out[c] = val(T[c]);
        return;
    }
    if (field >= 1 && field <= NSP) {
        out[c] = val(Y[(long long)(field - 1) * P.N + c]);
        return;
    }
    const double Tc = val(T[c]);
    double Yc[NSP];
#pragma unroll
    for (int k = 0; k < NSP; ++k) Yc[k] = val(Y[(long long)k * P.N + c]);
    double rho, q;
    const double h = hrr_of<S>(P, Tc, Yc, &rho, &q);
    double v = 0.0;
    if (field >= 6 && field <= 8) {
        const int a = field - 6;
        if (a < DIM) {
            double m = 0.0;
#pragma unroll
            for (int i = 0; i < Q; ++i) m += (double)ccomp<DIM>(i, a) * val(g[(long long)i * P.N + c]);
            v = 3.0 * m / rho;
        }
    } else if (field == 9) {
#pragma unroll
        for (int i = 0; i < Q; ++i) v += val(g[(long long)i * P.N + c]);
    } else if (field == 10) {
        v = rho;
    } else if (field == 11) {
        v = h;
    }
    out[c] = v;
}

// the whole state (g_0..g_{Q-1}, T, Y_0..Y_{NSP-1}) of listed cells
template <typename S>
__global__ void __launch_bounds__(256) cells_kernel(long long N, int Q, const S* __restrict__ g,
                                                    const S* __restrict__ T, const S* __restrict__ Y,
                                                    const long long* __restrict__ cells, long long n,
                                                    double* __restrict__ out)
{
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const long long c = cells[t];
    double* o = out + t * (Q + 1 + NSP);
    for (int i = 0; i < Q; ++i) o[i] = val(g[(long long)i * N + c]);
    o[Q] = val(T[c]);
    for (int k = 0; k < NSP; ++k) o[Q + 1 + k] = val(Y[(long long)k * N + c]);
}

cudaError_t launch_cells(int dim, int precision, const StepParams<double>& P, StateView st, const long long* cells,
                         long long n, double* out, cudaStream_t stream)
{
    if (n <= 0) return cudaSuccess;
    const int Q = dim == 2 ? 9 : 27;
    const unsigned blocks = (unsigned)((n + 255) / 256);
    if (precision == 2)
        cells_kernel<Tan><<<blocks, 256, 0, stream>>>(P.N, Q, (const Tan*)st.g, (const Tan*)st.T, (const Tan*)st.Y,
                                                      cells, n, out);
    else if (precision == 3)
        cells_kernel<Tanf><<<blocks, 256, 0, stream>>>(P.N, Q, (const Tanf*)st.g, (const Tanf*)st.T,
                                                       (const Tanf*)st.Y, cells, n, out);
    else if (precision == 0)
        cells_kernel<double><<<blocks, 256, 0, stream>>>(P.N, Q, (const double*)st.g, (const double*)st.T,
                                                         (const double*)st.Y, cells, n, out);
    else
        cells_kernel<float><<<blocks, 256, 0, stream>>>(P.N, Q, (const float*)st.g, (const float*)st.T,
                                                        (const float*)st.Y, cells, n, out);
    return cudaGetLastError();
}

cudaError_t launch_field(int dim, int precision, const StepParams<double>& P, StateView st, const uint8_t* solid,
                         int field, double* out, cudaStream_t stream)
{
    const unsigned blocks = (unsigned)((P.ncell + 255) / 256);
    if (precision == 2) {
        if (dim != 2) return cudaErrorInvalidValue;
        field_kernel<2, Tan><<<blocks, 256, 0, stream>>>(P, (const Tan*)st.g, (const Tan*)st.T, (const Tan*)st.Y,
                                                          solid, field, out);
        return cudaGetLastError();
    }
    if (precision == 3) {
        if (dim != 2) return cudaErrorInvalidValue;
        field_kernel<2, Tanf><<<blocks, 256, 0, stream>>>(P, (const Tanf*)st.g, (const Tanf*)st.T, (const Tanf*)st.Y,
                                                          solid, field, out);
        return cudaGetLastError();
    }
    if (precision == 0) {
        if (dim == 2)
            field_kernel<2, double><<<blocks, 256, 0, stream>>>(P, (const double*)st.g, (const double*)st.T,
                                                                 (const double*)st.Y, solid, field, out);
        else
            field_kernel<3, double><<<blocks, 256, 0, stream>>>(P, (const double*)st.g, (const double*)st.T,
                                                                 (const double*)st.Y, solid, field, out);
    } else {
        if (dim == 2)
            field_kernel<2, float><<<blocks, 256, 0, stream>>>(P, (const float*)st.g, (const float*)st.T,
                                                                (const float*)st.Y, solid, field, out);
        else
            field_kernel<3, float><<<blocks, 256, 0, stream>>>(P, (const float*)st.g, (const float*)st.T,
                                                                (const float*)st.Y, solid, field, out);
    }
    return cudaGetLastError();
}

}  // namespace lbfd
