// Weight (and bias) gradients of the correction network's convolutions on the
// tcgen05 tensor cores:
//   dW[co][tap][ci] = sum_p dY[p][co] X[p + tap][ci],   db[co] = sum_p dY[p][co],
// p over every grid point of every sample.  Included by cnn.cu only.
//
// The contraction runs over the points, so both operands are read as
// MN-major core matrices: 8 x-consecutive points (K) of one 16-byte chunk of
// 8 channels (M or N) are 128 contiguous bytes of the padded chunk-major
// activations, and a TMA box places them in shared memory as they are.  Two
// of the three tap directions become matrix rows and columns:
//
//   * A (M = 128) is the 32-channel operand, staged as [y][z][chunk][8 x]: 16
//     chunks at a uniform 128-byte stride are four consecutive z planes, so
//     one MMA against B plane zb takes A planes zb - 1 .. zb + 2.  Row block
//     j = 0, 1, 2 is the z shift; block 3 is never read (a tcgen05 MMA of
//     M = 96 does not exist).
//   * B is staged as [z][y][chunk][x]: consecutive chunks run on into the next
//     row, so N covers the three y shifts of a chunk set.
//       WIDE (layer 2, 32 channels): rows of 8 + 2 points, N = 3 x 32 = 96, one
//         MMA per x shift (the descriptor starts 16 bytes later).
//       else (layers 1 and 3, 8 channels hold all real ones): the TMA map has
//         an x-shift dimension of stride 16 bytes, so a row is three shifted
//         copies of 8 points and N = (3 y x 3 x + 1 unread) x 8 = 80: one MMA
//         for all nine in-plane shifts.
//
// A tcgen05 MMA of M = 128, K = 16 costs 45 cycles at N <= 32, 52 at 80, 56 at
// 96 (gbfd_tc_mma_cycles), so stacking shifts along N is what makes the 27
// taps cheap: 168 (WIDE) and 52 cycles per 16 points where one MMA per tap
// would take 405.  Every pair (A point, B point) enters exactly once: A's
// map covers interior x and y (the zero fill outside drops the rest of ragged
// tiles) and B's map interior z; the other coordinates use the periodic copies.
//
// Accuracy: products of BF16 values are exact in FP32; the running sums leave
// tensor memory every FLUSH tiles (a chain of at most FLUSH * 32 FP32
// additions) and are carried on in FP32 registers, CTA sums are added in a
// fixed order (deterministic).
//
// Bound: for layer 2 the MMAs with their operand reads (96 per 512-point tile,
// 7 KB of shared memory each), for layers 1 and 3 the L2-to-SM copies (77 KB
// per tile against 32 MMAs).  Measured at 8 samples of 64^3: layer 2 0.106 ms,
// layers 1 and 3 0.072 ms each, where FP32 sums on CUDA cores took 9.63, 4.89
// and 5.40 ms (an Adam step 21.1 -> 1.37 ms by this alone).
#pragma once

namespace gbfd {
namespace cnn {
namespace wg {

constexpr int TX = 8, TY = 16, ZB = 4;  // points of a tile: x, y, z
constexpr int AZ = ZB + 2;              // A planes
constexpr int BY = TY + 2;              // B rows
constexpr int KSTEPS = TY / 2;          // K = 16 points: two rows of 8
constexpr int THREADS = 320;
constexpr int FLUSH = 4;                // tiles per accumulation in tensor memory
constexpr int MROWS = 96;               // rows read back: 3 z shifts x 32 channels

// Warp roles: 0 the TMA copies, 1 the MMAs (and the TMEM allocation), 3 and 7
// the bias sums, the others the accumulators: TMEM lane quarter warp % 4
// (0, 1, 2 = the z shift), columns split between two warps.
constexpr int BIAS_WARPS = 2, ACC_WARPS = 6;

template <bool WIDE>
struct Smem {
    static constexpr int A_ROW = AZ * 4 * 128;  // bytes from row y to y + 1
    static constexpr int A_BYTES = TY * A_ROW;
    static constexpr int B_CHUNK = WIDE ? (TX + 2) * 16 : TX * 16;
    static constexpr int B_ROW = (WIDE ? 4 : 3) * B_CHUNK;
    static constexpr int B_PLANE = BY * B_ROW;
    static constexpr int B_BYTES = ZB * B_PLANE;
    static constexpr int N = WIDE ? 96 : 80;
    static constexpr int NMMA = WIDE ? 3 : 1;  // MMAs per K step
    static constexpr int COLS = NMMA * N;      // accumulator columns
    static constexpr int USED = WIDE ? 288 : 72;  // of these, read back
    static constexpr int HALF = USED / 2;         // per accumulator warp
    static constexpr int NACC = WIDE ? 1 : 2;
    static constexpr int TCOLS = WIDE ? 512 : 256;
    static constexpr int NSTAGE = 2;
    // the last window of A reads one plane (512 bytes) past the box, the last
    // one of B one chunk: the unread row block and columns
    static constexpr int A_PITCH = (A_BYTES + 512 + 127) / 128 * 128;
    static constexpr int B_PITCH = (B_BYTES + B_CHUNK + 127) / 128 * 128;
    static constexpr int STAGE = A_PITCH + B_PITCH;
    static constexpr int RED_OFF = NSTAGE * STAGE;  // bias reduction, 64 x 8 floats
    static constexpr int BAR_OFF = RED_OFF + 64 * 8 * 4;
    // full[NSTAGE], empty[NSTAGE], accf[NACC], acce[NACC], stopped, TMEM
    // address, abort flag, five counts
    static constexpr int BYTES = BAR_OFF + (2 * NSTAGE + 2 * NACC + 1) * 8 + 8 + 24;
    static_assert(NACC * COLS <= TCOLS, "TMEM columns");
    static_assert(STAGE % 128 == 0 && A_PITCH % 128 == 0, "TMA destinations");
    static_assert(BYTES <= 227 * 1024, "shared memory");
    static_assert((ZB - 1) * 512 + (TY - 1) * A_ROW + 2048 <= A_PITCH, "A windows");
    static_assert((ZB - 1) * B_PLANE + (TY - 1) * B_ROW + (NMMA - 1) * 16 + (N / 8 - 1) * B_CHUNK +
                          128 <= B_PITCH, "B windows");
};

struct Args {
    int n, nb;     // grid side, samples in use
    int bias_b;    // the bias gradient sums operand B (dY) instead of A
    float *part;   // [CTA][USED columns][MROWS], then [32] bias sums
    int *dev_error;
};

template <bool WIDE>
__host__ __device__ constexpr int part_floats()
{
    return Smem<WIDE>::USED * MROWS + 32;
}

__device__ __forceinline__ void tma_load_5d(void *dst, const CUtensorMap *map, uint64_t *bar, int c0,
                                            int c1, int c2, int c3, int c4)
{
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5, %6, %7}], [%2];" ::"r"(tiled::smem_u32(dst)),
        "l"((uint64_t)map), "r"(tiled::smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4)
        : "memory");
}

template <bool WIDE>
__global__ void __launch_bounds__(THREADS, 1)
    k_wgrad_tc(const __grid_constant__ CUtensorMap amap, const __grid_constant__ CUtensorMap bmap,
               const Args a)
{
    using S = Smem<WIDE>;
    constexpr int NSTAGE = S::NSTAGE, NACC = S::NACC;
    extern __shared__ __align__(1024) unsigned char smem[];
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + S::BAR_OFF);
    uint64_t *empty = full + NSTAGE;
    uint64_t *accf = empty + NSTAGE;
    uint64_t *acce = accf + NACC;
    uint64_t *stopped = acce + NACC;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(stopped + 1);
    volatile int *abort = reinterpret_cast<volatile int *>(tslot + 1);
    // copies issued / waited for, windows committed / drained, MMAs cut short
    int *cnt = reinterpret_cast<int *>(tslot + 2);
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;

    if (threadIdx.x == 0) {
        for (int s = 0; s < NSTAGE; ++s) {
            tiled::mbar_init(&full[s], 1);
            tiled::mbar_init(&empty[s], 1 + BIAS_WARPS);
        }
        for (int s = 0; s < NACC; ++s) {
            tiled::mbar_init(&accf[s], 1);
            tiled::mbar_init(&acce[s], ACC_WARPS);
        }
        tiled::mbar_init(stopped, 1);
        *abort = 0;
        cnt[0] = cnt[1] = cnt[2] = cnt[3] = cnt[4] = 0;
        tiled::fence_mbar_init();
    }
    if (warp == 1)
        tc::tmem_alloc(tslot, S::TCOLS);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem =
        __shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t *>(tslot), 0);
    chain_wait();
    chain_next();

    const int n = a.n;
    const int tx_n = (n + TX - 1) / TX, ty_n = (n + TY - 1) / TY, tz_n = (n + ZB - 1) / ZB;
    const int ntiles = a.nb * tz_n * ty_n * tx_n;
    const int mine = ((int)blockIdx.x < ntiles)
                         ? (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    auto origin = [&](int i, int &x0, int &y0, int &z0, int &b) {
        int r = (int)blockIdx.x + i * (int)gridDim.x;
        x0 = (r % tx_n) * TX;
        r /= tx_n;
        y0 = (r % ty_n) * TY;
        r /= ty_n;
        z0 = (r % tz_n) * ZB;
        b = r / tz_n;
    };
    float *part = a.part + (long long)blockIdx.x * part_floats<WIDE>();

    if (warp == 0) {
        if (lane == 0) {
            for (int i = 0; i < mine; ++i) {
                const int s = i % NSTAGE;
                if (!wait_or_abort(&empty[s], ((i / NSTAGE) & 1) ^ 1, abort))
                    break;
                int x0, y0, z0, b;
                origin(i, x0, y0, z0, b);
                unsigned char *st = smem + s * S::STAGE;
                tiled::mbar_expect_tx(&full[s], S::A_BYTES + S::B_BYTES);
                // A: interior (x, y), planes z0 - 1 .. z0 + ZB (padded z0 ..);
                // B: interior z, rows and x from the padded frame on
                tma_load_5d(st, &amap, &full[s], 8 * x0, 0, z0, y0, b);
                tma_load_5d(st + S::A_PITCH, &bmap, &full[s], 8 * x0, 0, y0, z0, b);
                cnt[0] = i + 1;
            }
        }
    } else if (warp == 1) {
        // the whole warp runs the loop, one lane issues (tc::mma_bf16_elect)
        const uint32_t elected = tc::elect_one();
        constexpr uint32_t idesc = tc::idesc_bf16_f32(MT, S::N) | tc::kIdescTransA | tc::kIdescTransB;
        // MN-major, no swizzle: LBO = from 8 points to the next 8 (one row
        // on), SBO = from one 8-channel chunk to the next
        const uint64_t ad0 = tc::smem_desc(tc::smem_u32(smem), S::A_ROW, 128);
        const uint64_t bd0 = tc::smem_desc(tc::smem_u32(smem + S::A_PITCH), S::B_ROW, S::B_CHUNK);
        auto wait = [&](uint64_t *bar, int phase) {
            return __all_sync(0xffffffffu, wait_or_abort(bar, phase, abort));
        };
        int i = 0;
#pragma unroll 1
        for (; i < mine; ++i) {
            const int s = i % NSTAGE, win = i / FLUSH, acc = win % NACC;
            if (i % FLUSH == 0 && !wait(&acce[acc], ((win / NACC) & 1) ^ 1))
                break;
            if (!wait(&full[s], (i / NSTAGE) & 1))
                break;
            cnt[1] = i + 1;
            tc::fence_after_sync();
            const uint64_t so = (uint64_t)((s * S::STAGE) >> 4);
            const uint32_t d = tmem + acc * S::COLS;
            const uint32_t keep = i % FLUSH != 0;
#pragma unroll
            for (int z = 0; z < ZB; ++z)
#pragma unroll
                for (int k = 0; k < KSTEPS; ++k)
#pragma unroll
                    for (int m = 0; m < S::NMMA; ++m)
                        tc::mma_bf16_elect(
                            elected, d + m * S::N,
                            ad0 + so + (uint64_t)((2 * k * S::A_ROW + z * 512) >> 4),
                            bd0 + so + (uint64_t)((z * S::B_PLANE + 2 * k * S::B_ROW + m * 16) >> 4),
                            idesc, (z == 0 && k == 0) ? keep : 1u);
            tc::commit_elect(elected, &empty[s]);
            if (i % FLUSH == FLUSH - 1 || i == mine - 1) {
                tc::commit_elect(elected, &accf[acc]);
                cnt[2] = win + 1;
            }
        }
        if (i < mine) {  // a wait gave up: the MMAs issued so far are waited for below
            tc::commit_elect(elected, stopped);
            cnt[4] = 1;
        }
    } else if (warp == 3 || warp == 7) {
        // bias gradient: 8 channels of one point per 16-byte load; 8 lanes
        // read 8 x-consecutive points
        const int t = (warp == 7 ? 32 : 0) + lane;
        float sum[8];
#pragma unroll
        for (int c = 0; c < 8; ++c)
            sum[c] = 0.f;
        auto add = [&](const unsigned char *p) {
            const uint4 v = *reinterpret_cast<const uint4 *>(p);
            const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u[c]));
                sum[2 * c] += f.x;
                sum[2 * c + 1] += f.y;
            }
        };
        for (int i = 0; i < mine; ++i) {
            const int s = i % NSTAGE;
            int ok = 0;
            if (lane == 0)
                ok = wait_or_abort(&full[s], (i / NSTAGE) & 1, abort);
            if (!__shfl_sync(0xffffffffu, ok, 0))
                break;
            if (lane != 0)
                (void)tiled::mbar_try_wait(&full[s], (i / NSTAGE) & 1);
            int x0, y0, z0, b;
            origin(i, x0, y0, z0, b);
            const unsigned char *st = smem + s * S::STAGE;
            if (!a.bias_b) {
                // A: chunk (t / 8) % 4 of the points x = t % 8, rows of this
                // warp's parity, planes z0 .. z0 + ZB - 1 inside the grid
                const unsigned char *p = st + ((t / 8) % 4) * 128 + (t % 8) * 16 + 512;
                const int nz = min(ZB, n - z0);
                for (int z = 0; z < nz; ++z)
#pragma unroll 4
                    for (int y = t / 32; y < TY; y += 2)
                        add(p + z * 512 + y * S::A_ROW);
            } else {
                // B (narrow): the unshifted copy, interior rows
                const unsigned char *p = st + S::A_PITCH + S::B_CHUNK + (t % 8) * 16;
                const int ny = min(TY, n - y0);
                for (int r = t / 8; r < ZB * ny; r += 8) {
                    const int z = r / ny, y = r % ny;
                    add(p + z * S::B_PLANE + (y + 1) * S::B_ROW);
                }
            }
            __syncwarp();
            if (lane == 0)
                mbar_arrive(&empty[s]);
        }
        float *red = reinterpret_cast<float *>(smem + S::RED_OFF);
#pragma unroll
        for (int c = 0; c < 8; ++c)
            red[t * 8 + c] = sum[c];
    } else {
        // accumulators: tensor memory -> FP32 registers once per window
        const int q = warp % 4, half = (warp == 2 || warp >= 8) ? 1 : 0;
        const uint32_t tl = tmem + ((uint32_t)(q * 32) << 16) + half * S::HALF;
        float v[S::HALF];
#pragma unroll
        for (int c = 0; c < S::HALF; ++c)
            v[c] = 0.f;
        const int nwin = (mine + FLUSH - 1) / FLUSH;
        for (int w = 0; w < nwin; ++w) {
            const int acc = w % NACC;
            int ok = 0;
            if (lane == 0)
                ok = wait_or_abort(&accf[acc], (w / NACC) & 1, abort);
            if (!__shfl_sync(0xffffffffu, ok, 0))
                break;
            if (lane != 0)
                (void)tiled::mbar_try_wait(&accf[acc], (w / NACC) & 1);
            tc::fence_after_sync();
            static_assert(S::HALF % 16 == 0 || S::HALF % 16 == 4, "column pieces");
            float x[16];
#pragma unroll
            for (int c = 0; c + 16 <= S::HALF; c += 16) {
                tc::tmem_ld16(tl + acc * S::COLS + c, x);
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    v[c + j] += x[j];
            }
            if constexpr (S::HALF % 16 == 4) {
                // 36 = 2 x 16 + 4: the 8-column load's upper half is unused
                tc::tmem_ld8(tl + acc * S::COLS + S::HALF - 4, x);
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    v[S::HALF - 4 + j] += x[j];
            }
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0)
                mbar_arrive(&acce[acc]);
            if (warp == 4 && lane == 0)
                cnt[3] = w + 1;
        }
#pragma unroll
        for (int c = 0; c < S::HALF; ++c)
            part[(half * S::HALF + c) * MROWS + q * 32 + lane] = v[c];
    }
    __syncthreads();
    if (*abort) {
        // a wait gave up: let the copies and MMAs still in flight land before
        // the shared memory and TMEM go away (bounded, abort ignored)
        if (threadIdx.x == 0) {
            atomicExch(a.dev_error, 2);
            volatile int never = 0;
            for (int j = cnt[1]; j < cnt[0]; ++j)
                (void)wait_or_abort(&full[j % NSTAGE], (j / NSTAGE) & 1, &never);
            for (int j = cnt[3]; j < cnt[2]; ++j)
                (void)wait_or_abort(&accf[j % NACC], (j / NACC) & 1, &never);
            if (cnt[4])
                (void)wait_or_abort(stopped, 0, &never);
        }
        __syncthreads();
    } else if (threadIdx.x < 32) {
        // the 64 partial bias sums of 8 channels, in a fixed order
        const float *red = reinterpret_cast<const float *>(smem + S::RED_OFF);
        const int co = threadIdx.x;
        float sum = 0.f;
        if (!a.bias_b) {
            for (int w = 0; w < 2; ++w)
                for (int x = 0; x < 8; ++x)
                    sum += red[(w * 32 + (co / 8) * 8 + x) * 8 + co % 8];
        } else if (co < 8) {
            for (int t = 0; t < 64; ++t)
                sum += red[t * 8 + co];
        }
        part[S::USED * MROWS + co] = sum;
    }
    tc::fence_after_sync();
    if (warp == 1)
        tc::tmem_dealloc(tmem, S::TCOLS);
}

// g of one layer from the CTAs' partial sums, added in a fixed order: 32
// values x 8 groups of CTAs per block.  Partial sum (col, row), row = 32 j +
// channel of A: see the operand stacking above; SWAP (layer 3): A is X and B
// is dY, else A is dY.  Padding channels of g are set to zero.
template <int CO, int CI, bool WIDE, bool SWAP>
__global__ void __launch_bounds__(256) k_wgrad_reduce(const float *part, int nparts,
                                                      float *__restrict__ g)
{
    chain_wait();
    chain_next();
    constexpr int PF = part_floats<WIDE>();
    __shared__ float sh[8][32];
    const int lane = threadIdx.x % 32, grp = threadIdx.x / 32;
    const int i = blockIdx.x * 32 + lane;
    const int per = (nparts + 7) / 8;
    float s = 0.f;
    if (i < PF)
#pragma unroll 4
        for (int p = grp * per; p < min(nparts, (grp + 1) * per); ++p)
            s += part[(long long)p * PF + i];
    sh[grp][lane] = s;
    __syncthreads();
    if (grp != 0 || i >= PF)
        return;
    s = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w)
        s += sh[w][lane];
    constexpr int NW = CO * TAPS * CI;
    const int bias = i - Smem<WIDE>::USED * MROWS;
    if (bias >= 0) {
        if (bias < CO)
            g[NW + bias] = s;
        return;
    }
    const int col = i / MROWS, row = i % MROWS, j = row / 32, ca = row % 32;
    int yi, xi, cb;
    if (WIDE) {
        xi = col / 96, yi = (col % 96) / 32, cb = col % 32;
    } else {
        yi = col / 24, xi = (col / 8) % 3, cb = col % 8;
    }
    if (!SWAP) {
        g[(ca * TAPS + (2 - j) * 9 + yi * 3 + xi) * CI + cb] = s;
        if (CI > 8 && !WIDE)  // input channels beyond the 8 staged ones are padding
            g[(ca * TAPS + (2 - j) * 9 + yi * 3 + xi) * CI + cb + 8] = 0.f;
    } else {
        const int tap = j * 9 + (2 - yi) * 3 + (2 - xi);
        g[(cb * TAPS + tap) * CI + ca] = s;
        g[((cb + 8) * TAPS + tap) * CI + ca] = 0.f;
    }
}

}  // namespace wg
}  // namespace cnn
}  // namespace gbfd
