// State copies into/out of the padded layout and the FP64 diagnostics
// reductions (mass, kinetic energy, max |u| for the time-step rule, per-field
// rms and max, non-finite flag).
#include <algorithm>
#include <cmath>
#include <cstdint>

#include "kernels.cuh"

namespace gbfd {

namespace {

// Four consecutive values moved with 16-byte accesses (one float4, or two
// double2), converted on the way.
template <class T>
struct Quad {
    T v[4];
};
template <class T>
__device__ __forceinline__ Quad<T> load_quad(const T *p);
template <>
__device__ __forceinline__ Quad<float> load_quad(const float *p)
{
    const float4 a = *reinterpret_cast<const float4 *>(p);
    return {{a.x, a.y, a.z, a.w}};
}
template <>
__device__ __forceinline__ Quad<double> load_quad(const double *p)
{
    const double2 a = reinterpret_cast<const double2 *>(p)[0];
    const double2 b = reinterpret_cast<const double2 *>(p)[1];
    return {{a.x, a.y, b.x, b.y}};
}
template <class T>
__device__ __forceinline__ void store_quad(T *p, const T (&v)[4]);
template <>
__device__ __forceinline__ void store_quad(float *p, const float (&v)[4])
{
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
template <>
__device__ __forceinline__ void store_quad(double *p, const double (&v)[4])
{
    reinterpret_cast<double2 *>(p)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2 *>(p)[1] = make_double2(v[2], v[3]);
}

constexpr int COPY_THREADS = 256;

// Group of LPR lanes that take ROWS rows at once, every load issued before the
// first store.  Chosen by row_group below.
template <int LPR, int ROWS>
constexpr int kRowsPerBlock = COPY_THREADS / LPR * ROWS;

// Every padded row (interior and ghost rows, interior and ghost columns) of
// every field from the compact source; ghosts take the periodic image.  VEC:
// source rows 16-byte aligned (nx % 4 == 0 and an aligned base), so values move
// in 16-byte accesses, four columns at a time; the four ghost columns on each
// side are the first and the last four of the row, written by the thread that
// holds them.  The source may be device memory or pinned host memory mapped into
// the device address space.  IDX: unsigned when the rows can be counted in it
// (with 64-bit row arithmetic 256^3 took 127 us, 5.0 TB/s; here 107).
template <class TD, class TSrc, bool VEC, int LPR, int ROWS, class IDX>
__global__ void __launch_bounds__(COPY_THREADS) k_scatter(const TSrc *__restrict__ src,
                                                         TD *__restrict__ dst, Layout L, IDX nrows)
{
    const int lane = threadIdx.x % LPR;
    const IDX row0 = (IDX)blockIdx.x * kRowsPerBlock<LPR, ROWS> + threadIdx.x / LPR * ROWS;
    const TSrc *s[ROWS];
    TD *d[ROWS];
    int n = 0;
#pragma unroll
    for (int k = 0; k < ROWS; ++k) {
        const IDX row = row0 + k;
        if (row >= nrows)
            break;
        const int Y = (int)(row % (IDX)L.rows);
        const IDX fz = row / (IDX)L.rows;
        const int z = (int)(fz % (IDX)L.nz), f = (int)(fz / (IDX)L.nz);
        int y = Y - GY;  // ny >= 8 > GY: one wrap is enough
        y = y < 0 ? y + L.ny : (y >= L.ny ? y - L.ny : y);
        s[k] = src + (((long long)f * L.nz + z) * L.ny + y) * L.nx;
        d[k] = dst + (long long)f * L.fpitch + (long long)z * L.plane + (long long)Y * L.P;
        n = k + 1;
    }
    if (VEC) {
        for (int x = 4 * lane; x < L.nx; x += 4 * LPR) {
            Quad<TSrc> q[ROWS];
#pragma unroll
            for (int k = 0; k < ROWS; ++k)
                if (k < n)
                    q[k] = load_quad(s[k] + x);
#pragma unroll
            for (int k = 0; k < ROWS; ++k)
                if (k < n) {
                    const TD v[4] = {(TD)q[k].v[0], (TD)q[k].v[1], (TD)q[k].v[2], (TD)q[k].v[3]};
                    store_quad(d[k] + GX + x, v);
                    if (x == 0)
                        store_quad(d[k] + GX + L.nx, v);
                    if (x == L.nx - 4)
                        store_quad(d[k], v);
                }
        }
    } else {
#pragma unroll
        for (int k = 0; k < ROWS; ++k)
            if (k < n) {
                for (int x = lane; x < L.nx; x += LPR)
                    d[k][GX + x] = (TD)s[k][x];
                if (lane < 2 * GX)
                    d[k][lane < GX ? lane : L.nx + lane] =
                        (TD)s[k][lane < GX ? L.nx - GX + lane : lane - GX];
            }
    }
}

// Interior rows back to the compact layout, in the same way.
template <class TS, class TD, bool VEC, int LPR, int ROWS, class IDX>
__global__ void __launch_bounds__(COPY_THREADS) k_gather(const TS *__restrict__ src,
                                                        TD *__restrict__ dst, Layout L, IDX nrows)
{
    const int lane = threadIdx.x % LPR;
    const IDX row0 = (IDX)blockIdx.x * kRowsPerBlock<LPR, ROWS> + threadIdx.x / LPR * ROWS;
    const TS *s[ROWS];
    int n = 0;
#pragma unroll
    for (int k = 0; k < ROWS; ++k) {
        const IDX row = row0 + k;
        if (row >= nrows)
            break;
        const int y = (int)(row % (IDX)L.ny);
        const IDX fz = row / (IDX)L.ny;
        s[k] = src + lidx(L, (int)(fz / (IDX)L.nz), (int)(fz % (IDX)L.nz), y, 0);
        n = k + 1;
    }
    TD *d = dst + (long long)row0 * L.nx;
    if (VEC) {
        for (int x = 4 * lane; x < L.nx; x += 4 * LPR) {
            Quad<TS> q[ROWS];
#pragma unroll
            for (int k = 0; k < ROWS; ++k)
                if (k < n)
                    q[k] = load_quad(s[k] + x);
#pragma unroll
            for (int k = 0; k < ROWS; ++k)
                if (k < n) {
                    const TD v[4] = {(TD)q[k].v[0], (TD)q[k].v[1], (TD)q[k].v[2], (TD)q[k].v[3]};
                    store_quad(d + (long long)k * L.nx + x, v);
                }
        }
    } else {
#pragma unroll
        for (int k = 0; k < ROWS; ++k)
            if (k < n)
                for (int x = lane; x < L.nx; x += LPR)
                    d[(long long)k * L.nx + x] = (TD)s[k][x];
    }
}

// 16-byte accesses need every row start aligned: the compact side's base
// and row length (nx % 4 == 0 keeps rows of 4- and 8-byte values on 16-byte
// boundaries once the base is), the padded side's interior rows are 128-byte
// aligned by construction.
inline bool quad_ok(const void *compact, int nx)
{
    return ((uintptr_t)compact % 16) == 0 && nx % 4 == 0;
}

// Lanes per row and rows at once, measured against a warp per row on 19 shapes from
// 8^3 to 256^3 in all four pairs of types (us, set or get): 8 lanes up to nx = 32, 16 up to
// 64 (64^3 FP32 8.2 -> 5.1, FP64 8.2 -> 6.2; 2000 x 8 x 8 28.7 -> 8.3), else a warp.  Two
// rows at once pay in FP32 on both sides when the rows fill the SMs (get 256^3 102.5 ->
// 98.4, 140^3 24.6 -> 20.5); with FP64 on one side they are up to 1.5 times slower
// (get 200 x 136 x 105 34.9 -> 49.7), as with few long rows (set 2048 x 16 x 16 6.2 ->
// 8.3), except from FP64 to FP32 in whole passes of the warp (set 256^3 161.6 -> 152.6).
// Host memory is written a warp per row (FP64 64^3 139 -> 89 us).
template <class TFrom, class TTo, class F>
cudaError_t row_group(long long nrows, int nx, bool vec, bool to_host, F &&f)
{
    using std::integral_constant;
    constexpr bool F32 = sizeof(TFrom) == 4 && sizeof(TTo) == 4;
    constexpr int kFilled = 4 * 152;  // blocks of two rows per warp
    auto g = [&](auto v, auto lpr, auto rows) {
        constexpr int PER = kRowsPerBlock<decltype(lpr)::value, decltype(rows)::value>;
        const unsigned grid = (unsigned)((nrows + PER - 1) / PER);
        if (nrows < (1LL << 31))
            f(v, lpr, rows, grid, (unsigned)nrows);
        else
            f(v, lpr, rows, grid, (unsigned long long)nrows);
        return cudaGetLastError();
    };
    const integral_constant<int, 1> one{};
    const integral_constant<int, 32> warp{};
    if (!vec)
        return g(std::false_type{}, warp, one);
    if (nx <= 32 && !to_host)
        return g(std::true_type{}, integral_constant<int, 8>{}, one);
    if (nx <= 64 && !to_host)
        return g(std::true_type{}, integral_constant<int, 16>{}, one);
    if constexpr (sizeof(TTo) == 4)
        if (F32 ? nrows >= (long long)kFilled * kRowsPerBlock<32, 2>
                : nx % 128 == 0 || nx >= 512)
            return g(std::true_type{}, warp, integral_constant<int, 2>{});
    return g(std::true_type{}, warp, one);
}

template <class TD, class TSrc>
cudaError_t scatter_t(const TSrc *src, TD *dst, const Layout &L, int nf, cudaStream_t stream)
{
    return row_group<TSrc, TD>(
        (long long)nf * L.nz * L.rows, L.nx, quad_ok(src, L.nx), false,
        [&](auto v, auto lpr, auto rows, unsigned grid, auto nrows) {
            k_scatter<TD, TSrc, decltype(v)::value, decltype(lpr)::value, decltype(rows)::value,
                      decltype(nrows)><<<grid, COPY_THREADS, 0, stream>>>(src, dst, L, nrows);
        });
}

template <class TS, class TD>
cudaError_t gather_t(const TS *src, TD *dst, const Layout &L, int nf, bool to_host,
                     cudaStream_t stream)
{
    return row_group<TS, TD>(
        (long long)nf * L.nz * L.ny, L.nx, quad_ok(dst, L.nx), to_host,
        [&](auto v, auto lpr, auto rows, unsigned grid, auto nrows) {
            k_gather<TS, TD, decltype(v)::value, decltype(lpr)::value, decltype(rows)::value,
                     decltype(nrows)><<<grid, COPY_THREADS, 0, stream>>>(src, dst, L, nrows);
        });
}

// ------------------------------------------------------ ghost planes in z

// With walls in z (Layout::gz = GZW): the ghost planes of nf fields as the
// mirror images of the interior about the wall points z = 0 and z = nz - 1,
// f(-k) = p_f f(k) and f(nz - 1 + k) = p_f f(nz - 1 - k), k = 1..3, where
// p_f = -1 for the fields flagged in odd_mask (bit f) and +1 otherwise.  Whole
// padded planes are copied (ghost rows and columns included: the producing
// kernel has already made them periodic copies).  One thread per 16 bytes of
// the 2 GZW ghost planes of every field (a padded plane is a whole number of
// 128-byte rows).
template <class T>
__global__ void __launch_bounds__(256) k_fill_ghosts_z(T *__restrict__ origin, Layout L, int nf,
                                                      int odd_mask)
{
    chain_wait();
    chain_next();
    constexpr int V = 16 / sizeof(T);
    const long long pv = L.plane / V;  // 16-byte vectors per plane
    const long long total = (long long)nf * 2 * GZW * pv;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const long long e = i % pv;
        long long r = i / pv;
        const int k = 1 + (int)(r % GZW);
        r /= GZW;
        const int side = (int)(r % 2);
        const int f = (int)(r / 2);
        const int zsrc = side ? L.nz - 1 - k : k;
        const int zdst = side ? L.nz - 1 + k : -k;
        const T *src = origin + (long long)f * L.fpitch + (long long)zsrc * L.plane;
        T *dst = origin + (long long)f * L.fpitch + (long long)zdst * L.plane;
        // a plane is the P * rows values from its (Y, X) = (0, 0) element,
        // which is 16-byte aligned (128 - GX w bytes past a 128-byte boundary)
        uint4 v = reinterpret_cast<const uint4 *>(src)[e];
        if ((odd_mask >> f) & 1) {
            T *t = reinterpret_cast<T *>(&v);
#pragma unroll
            for (int j = 0; j < V; ++j)
                t[j] = -t[j];
        }
        reinterpret_cast<uint4 *>(dst)[e] = v;
    }
}

}  // namespace

cudaError_t launch_fill_ghosts_z(void *origin, const Layout &L, int nf, int odd_mask,
                                 cudaStream_t stream, int *launches)
{
    if (!L.gz)
        return cudaSuccess;
    const long long total = (long long)nf * 2 * GZW * (L.plane * L.w / 16);
    const int blocks = (int)((total + 255) / 256 < 4096 ? (total + 255) / 256 : 4096);
    *launches += 1;
    if (L.w == 8)
        return launch_chained<k_fill_ghosts_z<double>>(dim3(blocks), dim3(256), 0, false, stream,
                                                       (double *)origin, L, nf, odd_mask);
    return launch_chained<k_fill_ghosts_z<float>>(dim3(blocks), dim3(256), 0, false, stream,
                                                  (float *)origin, L, nf, odd_mask);
}

namespace {

// ---------------------------------------------------------------- reductions

constexpr int DIAG_THREADS = 256;
constexpr int NQ = 16;  // reduced quantities per block

// q[0] sum rho, q[1] sum rho|u|^2/2, q[2] max|u|^2, q[3] sum |u|^2,
// q[4..8] sum f^2, q[9..13] max |f|, q[14] non-finite count.
template <class TS>
__global__ void __launch_bounds__(DIAG_THREADS) k_diag_partial(const TS *__restrict__ st,
                                                                Layout L, int nf,
                                                                double *__restrict__ part)
{
    double q[NQ];
#pragma unroll
    for (int i = 0; i < NQ; ++i)
        q[i] = 0.0;
    const long long nrows = (long long)L.nz * L.ny;
    for (long long r = blockIdx.x; r < nrows; r += gridDim.x) {
        const int z = (int)(r / L.ny), y = (int)(r % L.ny);
        for (int x = threadIdx.x; x < L.nx; x += blockDim.x) {
            double v[5];
#pragma unroll
            for (int f = 0; f < 5; ++f)
                v[f] = f < nf ? (double)st[lidx(L, f, z, y, x)] : 0.0;
            const double rho = exp(v[0]);
            const double uu = v[1] * v[1] + v[2] * v[2] + v[3] * v[3];
            q[0] += rho;
            q[1] += 0.5 * rho * uu;
            q[2] = fmax(q[2], uu);
            q[3] += uu;
#pragma unroll
            for (int f = 0; f < 5; ++f) {
                q[4 + f] += v[f] * v[f];
                q[9 + f] = fmax(q[9 + f], fabs(v[f]));
                if (!isfinite(v[f]))
                    q[14] += 1.0;
            }
        }
    }
    // fixed-order block tree reduction
    __shared__ double sh[DIAG_THREADS];
    for (int i = 0; i < 15; ++i) {
        const bool ismax = (i == 2) || (i >= 9 && i <= 13);
        sh[threadIdx.x] = q[i];
        __syncthreads();
        for (int s = DIAG_THREADS / 2; s > 0; s >>= 1) {
            if (threadIdx.x < s) {
                const double a = sh[threadIdx.x], b = sh[threadIdx.x + s];
                sh[threadIdx.x] = ismax ? fmax(a, b) : a + b;
            }
            __syncthreads();
        }
        if (threadIdx.x == 0)
            part[(long long)blockIdx.x * NQ + i] = sh[0];
        __syncthreads();
    }
}

__global__ void __launch_bounds__(DIAG_THREADS) k_diag_final(const double *__restrict__ part,
                                                              int nblocks, long long npts,
                                                              double dv, double *__restrict__ out)
{
    __shared__ double sh[DIAG_THREADS];
    __shared__ double res[NQ];
    for (int i = 0; i < 15; ++i) {
        const bool ismax = (i == 2) || (i >= 9 && i <= 13);
        double a = 0.0;
        for (int b = threadIdx.x; b < nblocks; b += DIAG_THREADS) {
            const double v = part[(long long)b * NQ + i];
            a = ismax ? fmax(a, v) : a + v;
        }
        sh[threadIdx.x] = a;
        __syncthreads();
        for (int s = DIAG_THREADS / 2; s > 0; s >>= 1) {
            if (threadIdx.x < s) {
                const double x = sh[threadIdx.x], y = sh[threadIdx.x + s];
                sh[threadIdx.x] = ismax ? fmax(x, y) : x + y;
            }
            __syncthreads();
        }
        if (threadIdx.x == 0)
            res[i] = sh[0];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double n = (double)npts;
        out[0] = dv * res[0];
        out[1] = dv * res[1];
        out[2] = sqrt(res[2]);
        out[3] = sqrt(res[3] / n);
        for (int f = 0; f < 5; ++f) {
            out[4 + f] = sqrt(res[4 + f] / n);
            out[9 + f] = res[9 + f];
        }
        out[14] = res[14] > 0.0 ? 1.0 : 0.0;
        out[15] = 0.0;
    }
}

// max |u|^2 alone, for the time-step rule: the same FP64 value as the full
// reduction's, NaNs skipped as by fmax.  The FP64 pipe (2 lanes per SM and
// clock) is what the full reduction waits for (its sums and exp(lnrho): 365 us
// at 200 x 136 x 105), so FP32 storage forms |u|^2 in FP32 first, whose relative
// error is below 2^-22, and only values within 2^-20 of the block's largest, or
// not comparable (overflow, NaN, tiny), are squared in FP64: about one per block
// of 4096 points.
// A thread reads UMAX_VEC times 16 bytes of each velocity component, all issued
// before the first is used; the padded planes are scanned as they lie (ghost
// columns and rows hold copies, padding zeros).
constexpr int UMAX_VEC = 4;
template <class TS>
__global__ void __launch_bounds__(DIAG_THREADS) k_umax(const TS *__restrict__ st,
                                                       long long fpitch, long long nvec,
                                                       unsigned long long *__restrict__ out)
{
    constexpr int V = 16 / sizeof(TS);
    const long long base = (long long)blockIdx.x * (DIAG_THREADS * UMAX_VEC) + threadIdx.x;
    uint4 q[UMAX_VEC][3];
#pragma unroll
    for (int k = 0; k < UMAX_VEC; ++k) {
        const long long i = base + k * DIAG_THREADS;
#pragma unroll
        for (int f = 0; f < 3; ++f)
            q[k][f] = i < nvec ? __ldg(reinterpret_cast<const uint4 *>(st + (1 + f) * fpitch) + i)
                               : make_uint4(0, 0, 0, 0);
    }
    double best = 0.0;
    auto val = [&](int k, int f, int j) { return reinterpret_cast<const TS *>(&q[k][f])[j]; };
    if constexpr (sizeof(TS) == 8) {
#pragma unroll
        for (int k = 0; k < UMAX_VEC; ++k)
#pragma unroll
            for (int j = 0; j < V; ++j) {
                const double x = val(k, 0, j), y = val(k, 1, j), z = val(k, 2, j);
                best = fmax(best, x * x + y * y + z * z);
            }
    } else {
        float s[UMAX_VEC][V], m = 0.f;
#pragma unroll
        for (int k = 0; k < UMAX_VEC; ++k)
#pragma unroll
            for (int j = 0; j < V; ++j) {
                const float x = val(k, 0, j), y = val(k, 1, j), z = val(k, 2, j);
                s[k][j] = x * x + y * y + z * z;
                m = s[k][j] < INFINITY ? fmaxf(m, s[k][j]) : m;
            }
        // (non-negative FP32 values order as their bits)
        __shared__ unsigned sh[DIAG_THREADS / 32];
        const unsigned wm = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
        if (threadIdx.x % 32 == 0)
            sh[threadIdx.x / 32] = wm;
        __syncthreads();
        unsigned bm = 0;
#pragma unroll
        for (int k = 0; k < DIAG_THREADS / 32; ++k)
            bm = max(bm, sh[k]);
        const float top = __uint_as_float(bm);
        const float lim = top > 1e-30f ? top * (1.f - 0x1p-20f) : 0.f;
        // a loop over the few, read again: unrolled and predicated, their FP64
        // instructions take their slots in every warp (50 us instead of 5 at
        // 200 x 136 x 105)
        unsigned pick = 0;
#pragma unroll
        for (int k = 0; k < UMAX_VEC; ++k)
#pragma unroll
            for (int j = 0; j < V; ++j)
                pick |= !(s[k][j] < lim) ? 1u << (k * V + j) : 0u;
#pragma unroll 1
        for (; pick; pick &= pick - 1) {
            const int e = __ffs(pick) - 1;
            const long long i = (base + e / V * DIAG_THREADS) * V + e % V;
            const bool in = i < nvec * V;
            const double x = in ? (double)st[fpitch + i] : 0.0, y = in ? (double)st[2 * fpitch + i] : 0.0,
                         z = in ? (double)st[3 * fpitch + i] : 0.0;
            best = fmax(best, x * x + y * y + z * z);
        }
    }
    // (and non-negative FP64 values as theirs)
    unsigned long long v = (unsigned long long)__double_as_longlong(best);
    for (int k = 16; k > 0; k >>= 1)
        v = max(v, __shfl_xor_sync(0xffffffffu, v, k));
    if (threadIdx.x % 32 == 0 && v)
        atomicMax(out, v);
}

}  // namespace

cudaError_t launch_umax(const void *state, const Layout &L, double *out, cudaStream_t stream,
                        int *launches)
{
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(double), stream);
    if (e != cudaSuccess)
        return e;
    // whole planes: a multiple of 128 bytes, from a 16-byte aligned start
    const long long nvec = (long long)L.nz * L.plane * L.w / 16;
    const unsigned blocks = (unsigned)((nvec + DIAG_THREADS * UMAX_VEC - 1) / (DIAG_THREADS * UMAX_VEC));
    if (L.w == 8)
        k_umax<double><<<blocks, DIAG_THREADS, 0, stream>>>((const double *)state, L.fpitch, nvec,
                                                           (unsigned long long *)out);
    else
        k_umax<float><<<blocks, DIAG_THREADS, 0, stream>>>((const float *)state, L.fpitch, nvec,
                                                          (unsigned long long *)out);
    *launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_scatter(const void *src, int src_fp64, void *dst, const Layout &L, int nf,
                           cudaStream_t stream, int *launches)
{
    *launches += 1;
    if (L.w == 8)
        return src_fp64 ? scatter_t((const double *)src, (double *)dst, L, nf, stream)
                        : scatter_t((const float *)src, (double *)dst, L, nf, stream);
    return src_fp64 ? scatter_t((const double *)src, (float *)dst, L, nf, stream)
                    : scatter_t((const float *)src, (float *)dst, L, nf, stream);
}

cudaError_t launch_gather(const void *src, const Layout &L, void *dst, int dst_fp64, int nf,
                          bool to_host, cudaStream_t stream, int *launches)
{
    *launches += 1;
    if (L.w == 8)
        return dst_fp64 ? gather_t((const double *)src, (double *)dst, L, nf, to_host, stream)
                        : gather_t((const double *)src, (float *)dst, L, nf, to_host, stream);
    return dst_fp64 ? gather_t((const float *)src, (double *)dst, L, nf, to_host, stream)
                    : gather_t((const float *)src, (float *)dst, L, nf, to_host, stream);
}

namespace {

__global__ void k_forcing_tables(int kx, int ky, int kz, double cphi, double sphi, int nx, int ny,
                                 int nz, double2 *__restrict__ tab, float2 *__restrict__ tab32)
{
    // the kernels of the step before still read the tables: only the phases
    // are formed ahead of them
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    int n, k, idx;
    if (i < nx) {
        n = nx, k = kx, idx = i;
    } else if (i < nx + ny) {
        n = ny, k = ky, idx = i - nx;
    } else {
        n = nz, k = kz, idx = i - nx - ny;
    }
    // exact integer reduction of the phase k idx / n (in turns)
    long long m = ((long long)k * idx) % n;
    m += m < 0 ? n : 0;
    double sn, cs;
    sincospi(2.0 * (double)m / (double)n, &sn, &cs);
    if (i < nx) {
        const double c2 = cs * cphi - sn * sphi, s2 = sn * cphi + cs * sphi;
        cs = c2;
        sn = s2;
    }
    chain_wait();
    chain_next();
    if (i >= nx + ny + nz)
        return;
    tab[i] = make_double2(cs, sn);
    tab32[i] = make_float2((float)cs, (float)sn);
}

}  // namespace

cudaError_t launch_forcing_tables(int kx, int ky, int kz, double phi, int nx, int ny, int nz,
                                  double2 *tab, float2 *tab32, cudaStream_t stream,
                                  int *launches)
{
    const int n = nx + ny + nz;
    *launches += 1;
    return launch_chained<k_forcing_tables>(dim3((n + 63) / 64), dim3(64), 0, false, stream, kx, ky,
                                            kz, cos(phi), sin(phi), nx, ny, nz, tab, tab32);
}

int diag_blocks(const Layout &L)
{
    const long long rows = (long long)L.nz * L.ny;
    return (int)(rows < 1216 ? rows : 1216);  // 8 blocks per SM on 152 SMs
}

cudaError_t launch_diagnostics(const void *state, const Layout &L, int nf, double dv,
                               double *partials, int nblocks, double *out, cudaStream_t stream,
                               int *launches)
{
    if (L.w == 8)
        k_diag_partial<double><<<nblocks, DIAG_THREADS, 0, stream>>>((const double *)state, L, nf,
                                                                     partials);
    else
        k_diag_partial<float><<<nblocks, DIAG_THREADS, 0, stream>>>((const float *)state, L, nf,
                                                                    partials);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return e;
    k_diag_final<<<1, DIAG_THREADS, 0, stream>>>(partials, nblocks,
                                                 (long long)L.nx * L.ny * L.nz, dv, out);
    *launches += 2;
    return cudaGetLastError();
}

}  // namespace gbfd
