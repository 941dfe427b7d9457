// Coarse-grid correction network: three periodic 3x3x3 convolutions
// (5 -> 32 -> 32 -> 5 channels, exact GELU after the first two) applied to a
// coarse solver state after each RK3 step, trained on the GPU.
//
// * Convolutions (forward, and the input gradient of the backward pass) are
//   implicit GEMMs on the tcgen05 tensor cores: M = 128 grid points per MMA,
//   N = the output channels of the three z taps of one (dy, dx) tap (they
//   share the A window), K = 9 (dy, dx) taps x input channels; BF16 operands
//   in shared memory as K-major core matrices, FP32 accumulators in TMEM.
// * A persistent, warp-specialised CTA per SM streams columns of the grid along
//   z: one warp loads each plane plus its periodic one-point halo with ONE TMA
//   box into a ring of stages, one warp issues the plane's MMAs from shifted
//   descriptors into a ring of TMEM accumulators (one per output plane), and
//   sixteen epilogue warps drain finished planes (bias, GELU or GELU', BF16
//   stores), so loads, MMAs and epilogues of neighbouring planes overlap.  The weights
//   (B operand) stay in shared memory.  Activations are kept in a padded,
//   chunk-major layout whose one-point frame holds the periodic copies, so a
//   halo never wraps.  The input gradient is the same kernel with the
//   weights transposed in channels and flipped in taps.
// * The weight gradient sums over all grid points (K = points) on the tensor
//   cores too (wgrad.cuh), split over CTAs and reduced in a fixed order
//   (deterministic).
// * MSE loss, Adam (FP32 master weights, BF16 copies in both GEMM layouts),
//   input normalisation, the residual update of the solver state, and the
//   centred box filter that makes training targets from fine-grid runs.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/gbfd.h"
#include "gelu.cuh"
#include "kernels.cuh"
#include "tcgen05.cuh"
#include "tiled_impl.cuh"

namespace gbfd {
bool ctx_view(gbfd_ctx *c, float **origin, Layout *L, int *nf, cudaStream_t *s);
}

namespace gbfd {
namespace cnn {

using bf16 = __nv_bfloat16;

constexpr int TAPS = 27;
constexpr int MT = 128;    // points per tile (MMA M)
constexpr int NC = 5;      // physical channels (lnrho, u_x, u_y, u_z, s)
constexpr int C0 = 16;     // padded input channels of layer 1
constexpr int CH = 32;     // hidden channels
constexpr int C3 = 16;     // padded output channels of layer 3

enum { EPI_GELU = 0, EPI_LINEAR = 1, EPI_DGELU = 2 };

// Packed FP32 parameters: W[co_pad][tap][ci_pad] then b[co_pad], per layer;
// padded channel counts per layer: (32, 16), (32, 32), (16, 32).
__host__ __device__ constexpr int dim_co(int l) { return l == 2 ? C3 : CH; }
__host__ __device__ constexpr int dim_ci(int l) { return l == 0 ? C0 : CH; }

__host__ __device__ constexpr int wcount(int l) { return dim_co(l) * TAPS * dim_ci(l); }
__host__ __device__ constexpr int pcount(int l) { return wcount(l) + dim_co(l); }
__host__ __device__ constexpr int poff(int l)
{
    return l == 0 ? 0 : (l == 1 ? pcount(0) : pcount(0) + pcount(1));
}
constexpr int kParams = pcount(0) + pcount(1) + pcount(2);
// real (unpadded) sizes, in the W[o][c][3][3][3] + b[o] order, layers 1..3
constexpr int kRealOut[3] = {CH, CH, NC};
constexpr int kRealIn[3] = {NC, CH, CH};
constexpr int kRealParams = (CH * NC * 27 + CH) + (CH * CH * 27 + CH) + (NC * CH * 27 + NC);

// element index of (row n, col k) of an N x K operand in core-matrix order
__host__ __device__ inline int core_idx(int n, int k, int K)
{
    return (n / 8) * (K * 8) + (k / 8) * 64 + (n % 8) * 8 + (k % 8);
}

// Activations live in a padded, chunk-major layout: act[c8][b][zp][yp][xp][8]
// (BF16; c8 = channel / 8, padded coordinates xp = x + 1 in 0..n+1, the
// outermost ones holding the periodic copies of the opposite faces), so that
// a tile's one-point halo is one rectangular, in-bounds box and the 8
// channels of one chunk of one point are 16 contiguous bytes.  Whoever writes
// a point also writes its periodic copies.  Index below in units of 16-byte
// chunks.
__host__ __device__ __forceinline__ long long aidx(int c8, int b, int zp, int yp, int xp, int n,
                                                   int B)
{
    const long long m = n + 2;
    return ((((long long)c8 * B + b) * m + zp) * m + yp) * m + xp;
}

// Calls f(xp, yp, zp) for the padded position of interior point (x, y, z)
// and for each of its periodic copies in the one-point frame (up to 8 at a
// corner; n >= 2).
template <class F>
__device__ __forceinline__ void each_copy(int x, int y, int z, int n, F &&f)
{
    const int xs[2] = {x + 1, x == 0 ? n + 1 : 0}, nxs = (x == 0 || x == n - 1) ? 2 : 1;
    const int ys[2] = {y + 1, y == 0 ? n + 1 : 0}, nys = (y == 0 || y == n - 1) ? 2 : 1;
    const int zs[2] = {z + 1, z == 0 ? n + 1 : 0}, nzs = (z == 0 || z == n - 1) ? 2 : 1;
    for (int iz = 0; iz < nzs; ++iz)
        for (int iy = 0; iy < nys; ++iy)
            for (int ix = 0; ix < nxs; ++ix)
                f(xs[ix], ys[iy], zs[iz]);
}

struct ConvArgs {
    const bf16 *wB;      // [N][27*CIN] in core-matrix order
    const float *bias;   // [N]                      (EPI_GELU, EPI_LINEAR)
    float4 *hsave;       // pre-activation (EPI_GELU; NULL: not kept), [N/4][B n^3] quads
    bf16 *yb;            // padded chunk-major output (EPI_GELU: GELU(h), EPI_DGELU: dh)
    float *yf;           // [npts][8]                (EPI_LINEAR)
    const float4 *hprev; // the same quads           (EPI_DGELU)
    int n;               // grid side
    int npts;            // batch * n^3
    int B;               // samples allocated in the padded arrays
    int run;             // output planes of a run (conv_run)
    int *dev_error;
};

// A conv column is TXT x TYT points of every z plane of a sample: one M = 128
// MMA row block per plane, row r = point (x0 + r % TXT, y0 + r / TXT).  A plane
// of its input plus the one-point halo, HX x HY points of CIN channels, is ONE
// TMA box of the padded chunk-major input, (8 channels, HX, HY, 1, CIN / 8
// chunks): in shared memory chunk c of halo point (hx, hy) sits at
// c * CS + (hy * HX + hx) * 16.  The A operand of in-plane tap (dy, dx) is that
// buffer at a shifted start: core matrices of 8 x-consecutive rows (16-byte row
// stride), row groups one halo row apart (SBO = HX * 16), K chunks CS apart
// (LBO).
//
// The three z taps of one (dy, dx) read the same A window (input plane j, j = 0
// one below the first output plane, feeds output planes j - dz for dz = 0, 1,
// 2), so they are ONE MMA with their weights stacked along N (N = 3 NO for NO
// output channels): a tcgen05 MMA of M = 128, K = 16 costs about the same for
// N = 16 or 32 as for 96 (measured on GB300: 45 cycles for N <= 32, 56 for
// N = 96, 64 for 128).  The accumulators of the output planes form a ring of
// RING slots in TMEM, slot s at column NO (RING - 1 - s), so that planes j, j - 1
// and j - 2 are consecutive columns; an MMA is cut in two where the ring wraps
// and loses the groups outside the column at its ends.  Every MMA accumulates,
// so the ring starts at zero and the epilogue zeroes the columns it has read.
//
// Streaming reads and multiplies every input plane once per run of output
// planes (plus two at its ends); four-plane tiles with their own halo took six
// planes for four.
constexpr int TXT = 8, TYT = 16;
constexpr int HX = TXT + 2, HY = TYT + 2, HPTS = HX * HY;
static_assert(TXT * TYT == MT, "one MMA row block per plane");
constexpr int TAPS_XY = 9;  // (dy, dx) taps; dz is stacked along N

// Warp roles of the convolution CTA (one per SM, persistent): warp 0 issues the
// TMA loads, warp 1 the MMAs (and owns the TMEM allocation), warps 2-17 are the
// epilogue: two groups of eight take the planes in turn, so that one plane's
// waits and stores overlap the next one's arithmetic (with one group every plane
// paid its whole latency).  Warp w reads TMEM lanes 32 (w % 4) .. 32 (w % 4) + 31;
// the first four warps of a group take the first half of the output channels.
constexpr int EPI_WARPS = 8, EPI_GROUPS = 2;
constexpr int CONV_THREADS = 32 * (2 + EPI_WARPS * EPI_GROUPS);
constexpr int RING = 16;     // accumulator slots (output planes)
constexpr int ACC_STEP = 4;  // slots that the MMAs claim at a time
static_assert(RING % ACC_STEP == 0 && RING >= ACC_STEP + 3, "claimed slots were drained");

template <int CIN, int NO, int EPI>
struct ConvSmem {
    static constexpr int N = 3 * NO;          // MMA N: the three z taps' output channels
    static constexpr int K = TAPS_XY * CIN;   // B operand K: (dy, dx) taps x input channels
    static constexpr int CH8 = CIN / 8;
    static constexpr int B_BYTES = N * K * 2;
    static constexpr int CS = HPTS * 16;  // chunk stride of the TMA box
    static constexpr int A_BYTES = CH8 * CS;
    static constexpr int NSTAGE = CIN >= 32 ? 10 : 16;  // input planes in flight
    static constexpr int A_OFF = (B_BYTES + 1023) / 1024 * 1024;
    static constexpr int A_PITCH = (A_BYTES + 127) / 128 * 128;
    static constexpr int BAR_OFF = A_OFF + NSTAGE * A_PITCH;
    // full[NSTAGE], empty[NSTAGE], acc_full[RING], acc_empty[RING], stopped,
    // then the TMEM address, the abort flag, six counts, the biases
    static constexpr int BIAS_OFF = BAR_OFF + (2 * NSTAGE + 2 * RING + 1) * 8 + 8 + 24;
    static constexpr int BYTES = BIAS_OFF + NO * 4;
    static constexpr int TCOLS = RING * NO;
    static_assert(TCOLS == 256 || TCOLS == 512, "TMEM columns");
    static_assert(CS % 16 == 0 && (CS >> 4) < (1 << 14) && ((K * 16) >> 4) < (1 << 14),
                  "descriptor offsets");
    static_assert(BAR_OFF % 8 == 0 && BYTES <= 227 * 1024, "shared memory");
};

// Zeroes 16 (or 8) consecutive FP32 columns of this warp's 32 TMEM lanes; the
// stores are complete after wait_st().
__device__ __forceinline__ void tmem_zero16(uint32_t taddr)
{
    const uint32_t z = 0;
    __syncwarp();
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1};" ::"r"(taddr),
        "r"(z)
        : "memory");
}

__device__ __forceinline__ void tmem_zero8(uint32_t taddr)
{
    const uint32_t z = 0;
    __syncwarp();
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1};" ::"r"(taddr),
        "r"(z)
        : "memory");
}

__device__ __forceinline__ void wait_st()
{
    __syncwarp();
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tiled::smem_u32(bar))
                 : "memory");
}

// Bounded wait that also gives up when another role has raised the CTA's
// abort flag; a wait that runs out (about 2 s) raises it.
__device__ __forceinline__ bool wait_or_abort(uint64_t *bar, uint32_t parity, volatile int *abort)
{
    if (tiled::mbar_try_wait(bar, parity))
        return true;
    const uint64_t t0 = tiled::global_ns();
    while (true) {
        if (tiled::mbar_try_wait(bar, parity))
            return true;
        if (*abort)
            return false;
        if (tiled::global_ns() - t0 > 2000000000ull) {
            *abort = 1;
            return false;
        }
    }
}

// The CTA's runs of up to `run` output planes along z inside one column:
// f(x0, y0, sample, z0, planes) for each.  Every role walks them the same way.
// CTAs that work at the same time take neighbouring columns at the same height,
// so that the halo rows and the 128-byte rows they share meet in L2.
template <class F>
__device__ __forceinline__ void each_run(int n, int nb, int run, F &&f)
{
    const int tx_n = (n + TXT - 1) / TXT, ty_n = (n + TYT - 1) / TYT, tz_n = (n + run - 1) / run;
    const int units = nb * tz_n * ty_n * tx_n;
    for (int u = blockIdx.x; u < units; u += gridDim.x) {
        int r = u;
        const int x0 = (r % tx_n) * TXT;
        r /= tx_n;
        const int y0 = (r % ty_n) * TYT;
        r /= ty_n;
        const int z0 = (r % tz_n) * run;
        if (!f(x0, y0, r / tz_n, z0, min(run, n - z0)))
            return;
    }
}

template <int CIN, int NO, int EPI>
__global__ void __launch_bounds__(CONV_THREADS, 1)
    k_conv_tc(const __grid_constant__ CUtensorMap xmap, const ConvArgs a)
{
    using SM = ConvSmem<CIN, NO, EPI>;
    constexpr int NSTAGE = SM::NSTAGE;
    constexpr int KSTEPS = CIN / 16;  // MMAs per (dy, dx) tap and input plane
    constexpr int SBO_B = SM::K * 16;
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char *sB = smem;
    unsigned char *sA = smem + SM::A_OFF;
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + SM::BAR_OFF);
    uint64_t *empty = full + NSTAGE;
    uint64_t *accf = empty + NSTAGE;
    uint64_t *acce = accf + RING;
    uint64_t *stopped = acce + RING;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(stopped + 1);
    volatile int *abort = reinterpret_cast<volatile int *>(tslot + 1);
    // copies issued / waited for, planes committed, MMAs cut short, planes
    // drained by each group
    int *cnt = reinterpret_cast<int *>(tslot + 2);
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;

    // epilogue geometry: two warps per TMEM lane quarter, each taking half
    // of the output channels
    constexpr int NH = NO / 2;  // channels per epilogue warp
    static_assert(NH == 16 || NH == 8, "epilogue column chunks");
    const int e = warp - 2;
    const int group = e / EPI_WARPS;
    const int q = warp % 4, c0 = (e % EPI_WARPS / 4) * NH;
    float *sbias = reinterpret_cast<float *>(smem + SM::BIAS_OFF);
    // zeroes NH columns of the warp's lanes; complete after wait_st()
    auto zero_cols = [&](uint32_t taddr) {
        if constexpr (NH == 16)
            tmem_zero16(taddr);
        else
            tmem_zero8(taddr);
    };

    // the weights (B operand) stay in shared memory for the whole launch
    for (int i = threadIdx.x; i < SM::B_BYTES / 16; i += CONV_THREADS)
        reinterpret_cast<uint4 *>(sB)[i] = reinterpret_cast<const uint4 *>(a.wB)[i];
    if (threadIdx.x == 0) {
        for (int s = 0; s < NSTAGE; ++s) {
            tiled::mbar_init(&full[s], 1);
            tiled::mbar_init(&empty[s], 1);
        }
        for (int s = 0; s < RING; ++s) {
            tiled::mbar_init(&accf[s], 1);
            tiled::mbar_init(&acce[s], EPI_WARPS);  // one arrival per epilogue warp
        }
        tiled::mbar_init(stopped, 1);
        *abort = 0;
        for (int i = 0; i < 6; ++i)
            cnt[i] = 0;
        tiled::fence_mbar_init();
    }
    if (EPI != EPI_DGELU && threadIdx.x < NO)
        sbias[threadIdx.x] = a.bias[threadIdx.x];
    if (warp == 1)
        tc::tmem_alloc(tslot, SM::TCOLS);
    tc::fence_smem_to_async();  // the weights, written by the generic proxy, feed the MMAs
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    // (the shuffle tells the compiler that the address is the warp's)
    const uint32_t tmem =
        __shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t *>(tslot), 0);
    // every MMA accumulates: the accumulators start at zero
    if (warp >= 2) {
        const uint32_t tl = tmem + ((uint32_t)(q * 32) << 16) + c0;
#pragma unroll 1
        for (int j = group; j < RING; j += EPI_GROUPS)
            zero_cols(tl + j * NO);
        wait_st();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    // everything above (weights, barriers, TMEM) may overlap the tail of the
    // kernel before this one in the stream, which never writes the weights
    // (the input staging kernel, another convolution or the gradient
    // reduction); the activations it writes are read only below
    chain_wait();
    chain_next();
    const int n = a.n;
    const long long n3 = (long long)n * n * n;
    const int nb = (int)(a.npts / n3);

    if (warp == 0) {
        // producer: one haloed plane per stage the MMAs freed
        if (lane == 0) {
            int i = 0;
            each_run(n, nb, a.run, [&](int x0, int y0, int b, int z0, int m) {
                for (int j = 0; j < m + 2; ++j, ++i) {
                    const int s = i % NSTAGE;
                    if (!wait_or_abort(&empty[s], ((i / NSTAGE) & 1) ^ 1, abort))
                        return false;
                    tiled::mbar_expect_tx(&full[s], SM::A_BYTES);
                    // padded coordinates of the halo's first point: (x0 - 1) +
                    // 1; x and the 8 channels of a chunk form one 160-byte row
                    tiled::tma_load_4d(sA + s * SM::A_PITCH, &xmap, &full[s], 8 * x0, y0,
                                       b * (n + 2) + z0 + j, 0);
                    cnt[0] = i + 1;
                }
                return true;
            });
        }
    } else if (warp == 1) {
        // MMA issuer: per input plane, 9 (dy, dx) taps x KSTEPS MMAs of up to
        // 3 NO columns; the commits free the stage and hand finished output
        // planes to the epilogue.  The whole warp runs the loop, one lane issues
        // (tc::mma_bf16_elect)
        const uint32_t elected = tc::elect_one();
        // descriptors of the stage and weight bases; every tap's operand
        // is a compile-time byte offset from them (the start address is
        // the descriptor's low field, in 16-byte units, and shared
        // memory addresses stay below 2^18 bytes, so adding the offset
        // cannot carry into the next field)
        const uint64_t bd0 = tc::smem_desc(tc::smem_u32(sB), 128, SBO_B);
        const uint64_t ad0 = tc::smem_desc(tc::smem_u32(sA), SM::CS, HX * 16);
        // CNT z taps from dz0 on, into consecutive slots down from `slot`
        auto issue = [&](uint64_t ad, int slot, int dz0, auto cntc) {
            constexpr uint32_t idesc = tc::idesc_bf16_f32(MT, decltype(cntc)::value * NO);
            const uint64_t bd = bd0 + (uint64_t)(dz0 * (NO / 8) * (SBO_B >> 4));
            const uint32_t d = tmem + (uint32_t)(NO * (RING - 1 - slot));
#pragma unroll
            for (int t = 0; t < TAPS_XY; ++t)
#pragma unroll
                for (int k = 0; k < KSTEPS; ++k)
                    tc::mma_bf16_elect(
                        elected, d,
                        ad + (uint64_t)((((t / 3) * HX + t % 3) * 16 + 2 * k * SM::CS) >> 4),
                        bd + (uint64_t)((t * KSTEPS + k) * 16), idesc, 1u);
        };
        auto issue_n = [&](uint64_t ad, int slot, int dz0, int cnt_z) {
            if (cnt_z == 3)
                issue(ad, slot, 0, std::integral_constant<int, 3>{});
            else if (cnt_z == 2)
                issue(ad, slot, dz0, std::integral_constant<int, 2>{});
            else
                issue(ad, slot, dz0, std::integral_constant<int, 1>{});
        };
        // Between two planes' MMAs lies what the tensor pipe waits for, so it is
        // kept short: counters instead of divisions, and the accumulator slots
        // waited for and fenced ACC_STEP at a time.
        int i = 0, s = 0, ph = 0;  // input planes so far; their stage and phase
        int done = 0, o_next = 0;  // output planes of earlier runs; slots waited for
        bool ok = true;
        auto wait = [&](uint64_t *bar, int phase) {
            if (!tiled::mbar_try_wait(bar, phase))
                ok = wait_or_abort(bar, phase, abort);
            ok = __all_sync(0xffffffffu, ok);
            return ok;
        };
        each_run(n, nb, a.run, [&](int, int, int, int, int m) {
#pragma unroll 1
            for (int j = 0; j < m + 2; ++j) {
                // z taps whose output plane j - dz lies in the run, cut
                // where the slots wrap
                const int lo = max(0, j - m + 1), hi = min(2, j);
                const int slot = (done + j - lo) % RING;
                const int first = min(hi - lo + 1, slot + 1);
                const uint64_t ad = ad0 + (uint64_t)((s * SM::A_PITCH) >> 4);
                if (j < m && done + j == o_next) {
                    // the next output planes: their slots must be drained and zero
                    for (int k = 0; k < ACC_STEP; ++k, ++o_next)
                        if (!wait(&acce[o_next % RING], ((o_next / RING) & 1) ^ 1))
                            return false;
                    tc::fence_after_sync();
                }
                if (!wait(&full[s], ph))
                    return false;
                cnt[1] = ++i;
                issue_n(ad, slot, lo, first);
                if (first < hi - lo + 1)
                    issue_n(ad, RING - 1, lo + first, hi - lo + 1 - first);
                tc::commit_elect(elected, &empty[s]);
                if (j >= 2) {
                    tc::commit_elect(elected, &accf[(done + j - 2) % RING]);
                    cnt[2] = done + j - 1;
                }
                if (++s == NSTAGE) {
                    s = 0;
                    ph ^= 1;
                }
            }
            done += m;
            return true;
        });
        if (!ok) {  // a wait gave up: the MMAs issued so far are waited for below
            tc::commit_elect(elected, stopped);
            cnt[3] = 1;
        }
    } else {
        // epilogue, per output plane: TMEM -> registers, zero those columns,
        // then bias / GELU / GELU' and the stores (with the periodic copies)
        const int r = q * 32 + lane;  // row of the M block = TMEM lane
        const int lx = r % TXT, ly = r / TXT;
        const uint32_t tl = tmem + ((uint32_t)(q * 32) << 16) + c0;
        const long long hq = (long long)a.B * n3;  // quads per channel group of h
        const long long m2 = (long long)(n + 2) * (n + 2), yc = m2 * (n + 2) * a.B;
        uint4 *yb = reinterpret_cast<uint4 *>(a.yb);
        int o0 = 0;  // output planes of earlier runs
        each_run(n, nb, a.run, [&](int x0, int y0, int b, int z0, int m) {
            const int x = x0 + lx, y = y0 + ly;
            const bool inside = x < n && y < n;
            // the point's chunk in the padded output, plane 0 of the frame, and
            // the offsets of its periodic copies in x and y (0: none)
            const long long col = aidx(c0 / 8, b, 0, y + 1, x + 1, n, a.B);
            const long long dx = x == 0 ? n : (x == n - 1 ? -n : 0);
            const long long dy = (long long)(n + 2) * (y == 0 ? n : (y == n - 1 ? -n : 0));
#pragma unroll 1
            for (int k = (group + o0) & 1; k < m; k += EPI_GROUPS) {
                const int o = o0 + k, z = z0 + k, slot = o % RING;
                const long long p = (long long)b * n3 + ((long long)z * n + y) * n + x;
                // the saved pre-activations, on their way during the wait (the
                // forward pass wrote them several kernels ahead in the chain: read-only
                // loads are safe)
                float4 hv[EPI == EPI_DGELU ? NH / 4 : 1];
                if constexpr (EPI == EPI_DGELU) {
                    if (inside)
#pragma unroll
                        for (int c = 0; c < NH / 4; ++c)
                            hv[c] = __ldg(a.hprev + (c0 / 4 + c) * hq + p);
                }
                // one lane waits, the warp follows it (the TMEM accesses below
                // are warp-collective)
                int ok = 0;
                if (lane == 0)
                    ok = wait_or_abort(&accf[slot], (o / RING) & 1, abort);
                if (!__shfl_sync(0xffffffffu, ok, 0))
                    return false;
                // the other lanes observe the completed phase too (it cannot
                // move on before this warp releases the slot)
                if (lane != 0)
                    (void)tiled::mbar_try_wait(&accf[slot], (o / RING) & 1);
                tc::fence_after_sync();
                const uint32_t tp = tl + (uint32_t)(NO * (RING - 1 - slot));
                float v[NH];
                if constexpr (NH == 16)
                    tc::tmem_ld16(tp, v);
                else
                    tc::tmem_ld8(tp, v);
                zero_cols(tp);
                if (inside) {
                    if constexpr (EPI == EPI_LINEAR) {
                        // five real output channels, all in the first half
                        if (c0 == 0) {
                            float4 *yo = reinterpret_cast<float4 *>(a.yf + p * 8);
                            yo[0] = make_float4(v[0] + sbias[0], v[1] + sbias[1], v[2] + sbias[2],
                                                v[3] + sbias[3]);
                            yo[1] = make_float4(v[4] + sbias[4], 0.f, 0.f, 0.f);
                        }
                    } else {
                        uint4 out[NH / 8];
#pragma unroll
                        for (int c = 0; c < NH; c += 8) {
                            float2 h[4];
                            if constexpr (EPI == EPI_GELU) {
#pragma unroll
                                for (int j = 0; j < 4; ++j)
                                    h[j] = __fadd2_rn(
                                        make_float2(v[c + 2 * j], v[c + 2 * j + 1]),
                                        *reinterpret_cast<const float2 *>(sbias + c0 + c + 2 * j));
                                if (a.hsave) {
                                    float4 *hs = a.hsave + (c0 + c) / 4 * hq + p;
                                    hs[0] = make_float4(h[0].x, h[0].y, h[1].x, h[1].y);
                                    hs[hq] = make_float4(h[2].x, h[2].y, h[3].x, h[3].y);
                                }
#pragma unroll
                                for (int j = 0; j < 4; ++j)
                                    h[j] = make_float2(gelu(h[j].x), gelu(h[j].y));
                            } else {
                                const float4 h0 = hv[c / 4], h1 = hv[c / 4 + 1];
                                const float hs[8] = {h0.x, h0.y, h0.z, h0.w,
                                                     h1.x, h1.y, h1.z, h1.w};
#pragma unroll
                                for (int j = 0; j < 4; ++j)
                                    h[j] = make_float2(v[c + 2 * j] * gelu_grad(hs[2 * j]),
                                                       v[c + 2 * j + 1] * gelu_grad(hs[2 * j + 1]));
                            }
                            __nv_bfloat162 w[4];
#pragma unroll
                            for (int j = 0; j < 4; ++j)
                                w[j] = __floats2bfloat162_rn(h[j].x, h[j].y);
                            out[c / 8] = *reinterpret_cast<uint4 *>(w);
                        }
                        // the point and its periodic copies in x, y and z
                        auto put = [&](long long i) {
#pragma unroll
                            for (int c = 0; c < NH / 8; ++c)
                                yb[i + c * yc] = out[c];
                        };
                        auto put_xy = [&](long long i) {
                            put(i);
                            if (dx)
                                put(i + dx);
                            if (dy) {
                                put(i + dy);
                                if (dx)
                                    put(i + dy + dx);
                            }
                        };
                        put_xy(col + (z + 1) * m2);
                        if (z == 0)
                            put_xy(col + (n + 1) * m2);
                        else if (z == n - 1)
                            put_xy(col);
                    }
                }
                // the zeroed columns go back to the MMAs
                wait_st();
                tc::fence_before_sync();
                __syncwarp();
                if (lane == 0)
                    mbar_arrive(&acce[slot]);
                if (e % EPI_WARPS == 0 && lane == 0)
                    cnt[4 + group] = o + 1;
            }
            o0 += m;
            return true;
        });
    }
    __syncthreads();
    if (*abort) {
        // a wait gave up: let the copies and MMAs still in flight land
        // before the shared memory and TMEM go away (bounded, abort ignored)
        if (threadIdx.x == 0) {
            atomicExch(a.dev_error, 2);
            volatile int never = 0;
            for (int j = cnt[1]; j < cnt[0]; ++j)
                (void)wait_or_abort(&full[j % NSTAGE], (j / NSTAGE) & 1, &never);
            for (int j = min(cnt[4], cnt[5]); j < cnt[2]; ++j)
                if (j >= cnt[4 + (j & 1)])
                    (void)wait_or_abort(&accf[j % RING], (j / RING) & 1, &never);
            if (cnt[3])
                (void)wait_or_abort(stopped, 0, &never);
        }
        __syncthreads();
    }
    tc::fence_after_sync();
    if (warp == 1)
        tc::tmem_dealloc(tmem, SM::TCOLS);
}

}  // namespace cnn
}  // namespace gbfd

#include "wgrad.cuh"

namespace gbfd {
namespace cnn {

// The 8 channels of chunk 0 of point (b, x, y, z) into a 16-channel padded
// activation, with its periodic copies.  Channels 8 to 15 are padding that stays
// zero from the network's creation on.
__device__ __forceinline__ void put_chunk0(bf16 *dst, const float (&v)[8], int b, int x, int y, int z,
                                           int n, int B)
{
    __nv_bfloat162 o[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
        o[i] = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
    const uint4 c0 = *reinterpret_cast<uint4 *>(o);
    uint4 *d = reinterpret_cast<uint4 *>(dst);
    each_copy(x, y, z, n, [&](int xp, int yp, int zp) { d[aidx(0, b, zp, yp, xp, n, B)] = c0; });
}

// Layer-1 input, normalised, from compact FP32 states [batch][5][n^3] (nf fields
// present).  (Chained kernels read plainly: a read-only load could take the data
// before the wait, while the caller's kernel still writes it.)
__global__ void k_input_compact(const float *xs, int nf, int n, int npts, int B, const float *mean,
                                const float *stdv, bf16 *__restrict__ x0)
{
    // only then may the first convolution start its prologue, which reads the
    // weights that the kernel before this one may have written
    chain_wait();
    chain_next();
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= npts)
        return;
    const int n3 = n * n * n;
    const int b = p / n3, r = p - b * n3;
    float v[8];
#pragma unroll
    for (int c = 0; c < 8; ++c)
        v[c] = (c < nf) ? (xs[((long long)b * NC + c) * n3 + r] - mean[c]) / stdv[c] : 0.f;
    put_chunk0(x0, v, b, r % n, (r / n) % n, r / (n * n), n, B);
}

// Same from a solver context's padded FP32 state (one box, batch 1).
__global__ void k_input_state(const float *st, Layout L, int nf, int B, const float *mean,
                              const float *stdv, bf16 *__restrict__ x0)
{
    chain_wait();
    chain_next();  // (after the wait, as above)
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    const int n = L.nx;
    if (p >= n * n * n)
        return;
    const int z = p / (n * n), y = (p / n) % n, x = p % n;
    float v[8];
#pragma unroll
    for (int c = 0; c < 8; ++c)
        v[c] = (c < nf) ? (st[lidx(L, c, z, y, x)] - mean[c]) / stdv[c] : 0.f;
    put_chunk0(x0, v, 0, x, y, z, n, B);
}

// state += std_out * y (the de-normalised predicted residual), ghosts kept.
__global__ void k_apply(float *st, Layout L, int nf, const float *y, const float *sout)
{
    chain_wait();
    chain_next();
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    const int n = L.nx;
    if (p >= n * n * n)
        return;
    const int z = p / (n * n), yy = (p / n) % n, x = p % n;
    const float4 y4 = *reinterpret_cast<const float4 *>(y + (long long)p * 8);
    const float yv[NC] = {y4.x, y4.y, y4.z, y4.w, y[(long long)p * 8 + 4]};
    float v[NC];  // every load before the first store
#pragma unroll
    for (int f = 0; f < NC; ++f)
        v[f] = f < nf ? st[lidx(L, f, z, yy, x)] + sout[f] * yv[f] : 0.f;
#pragma unroll
    for (int f = 0; f < NC; ++f)
        if (f < nf)
            store_ghosted(st, L, f, z, yy, x, v[f]);
}

// Normalised output [batch][5][n^3] from the layer-3 rows (tests, inference).
__global__ void k_output_compact(const float *__restrict__ y, int n3, int npts,
                                 float *__restrict__ out)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= npts)
        return;
    const int b = p / n3, r = p - b * n3;
    for (int c = 0; c < NC; ++c)
        out[((long long)b * NC + c) * n3 + r] = y[(long long)p * 8 + c];
}

// MSE of the normalised residual: t = (target - x) / std_out; loss partial
// sums per block (FP64) and dY3 = 2 (y - t) / count in BF16, channels-last.  A
// thread takes LOSS_PTS points and sums their squares in float-float (products
// and sums with their rounding errors, about 46 significant bits), one FP64 value
// per thread: converting and adding every square in FP64 kept the narrow FP64
// pipe busy for half of the kernel.
constexpr int LOSS_PTS = 4;
__global__ void __launch_bounds__(256) k_loss(const float *y, const float *xs, const float *ts,
                                              const float *sout, int nf, int n, int npts, int B,
                                              float inv_count, bf16 *__restrict__ dy3,
                                              double *__restrict__ part)
{
    chain_wait();
    chain_next();
    const int n3 = n * n * n;
    __shared__ double sh[256];
    // of channel c at element i of the states, y the network's output there
    auto residual = [&](float yc, int c, long long i) {
        return yc - (c < nf ? (ts[i] - xs[i]) / sout[c] : 0.f);
    };
    float hi = 0.f, lo = 0.f;
#pragma unroll
    for (int k = 0; k < LOSS_PTS; ++k) {
        const int p = (blockIdx.x * LOSS_PTS + k) * 256 + threadIdx.x;
        if (p >= npts)
            break;
        const int b = p / n3, r = p - b * n3;
        const float4 y4 = *reinterpret_cast<const float4 *>(y + (long long)p * 8);
        const float yv[NC] = {y4.x, y4.y, y4.z, y4.w, y[(long long)p * 8 + 4]};
        float d[8];
#pragma unroll
        for (int c = 0; c < 8; ++c)
            d[c] = 0.f;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const float e = residual(yv[c], c, ((long long)b * NC + c) * n3 + r);
            float sq, err, sum, rest;
            two_prod(e, e, sq, err);
            two_sum(hi, sq, sum, rest);
            hi = sum;
            lo = __fadd_rn(lo, __fadd_rn(rest, err));
            d[c] = 2.f * e * inv_count;
        }
        // dY3 into the padded chunk-major layout, with its periodic copies
        put_chunk0(dy3, d, b, r % n, (r / n) % n, r / (n * n), n, B);
    }
    double sum = (double)hi + (double)lo;
    if (!(hi >= 0x1p-100f && hi < INFINITY)) {
        // squares or their error terms outside the FP32 range: again in FP64
        sum = 0.0;
#pragma unroll 1
        for (int k = 0; k < LOSS_PTS; ++k) {
            const int p = (blockIdx.x * LOSS_PTS + k) * 256 + threadIdx.x;
            if (p >= npts)
                break;
            const int b = p / n3, r = p - b * n3;
#pragma unroll 1
            for (int c = 0; c < NC; ++c) {
                const double e = residual(y[(long long)p * 8 + c], c, ((long long)b * NC + c) * n3 + r);
                sum += e * e;
            }
        }
    }
    sh[threadIdx.x] = sum;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (threadIdx.x < s)
            sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0)
        part[blockIdx.x] = sh[0];
}

__global__ void k_sum_double(const double *part, int n, double *__restrict__ out)
{
    chain_wait();
    chain_next();
    __shared__ double sh[256];
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += 256)
        s += part[i];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int k = 128; k > 0; k >>= 1) {
        if (threadIdx.x < k)
            sh[threadIdx.x] += sh[threadIdx.x + k];
        __syncthreads();
    }
    if (threadIdx.x == 0)
        *out = sh[0];
}

struct PackArgs {
    float *w, *m, *v;  // FP32 master parameters and Adam moments [kParams]
    const float *g;    // gradients [kParams] (NULL: pack only)
    float lr, b1, b2, eps, bc1, bc2;
    bf16 *fwd[3];      // forward B operands, layer l: [dz][co][9*ci]
    bf16 *bwd[3];      // input-gradient B operands (layers 2, 3): [dz][ci][9*co]
    float *bias[3];    // FP32 biases [co]
};

// Adam step (Kingma & Ba 2015) on the master weights, then the BF16 GEMM
// copies, tap = (dz, dy, dx) = 9 dz + t: forward B[dz CO + co][t CI + ci];
// input-gradient B'[dz' CI + ci][t' CO + co] for the flipped tap
// (dz', t') of 26 - tap (channels transposed).
__global__ void k_adam_pack(PackArgs a)
{
    chain_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= kParams)
        return;
    float w = a.w[i];
    if (a.g) {
        const float g = a.g[i];
        const float m = a.b1 * a.m[i] + (1.f - a.b1) * g;
        const float v = a.b2 * a.v[i] + (1.f - a.b2) * g * g;
        a.m[i] = m;
        a.v[i] = v;
        w -= a.lr * (m / a.bc1) / (sqrtf(v / a.bc2) + a.eps);
        a.w[i] = w;
    }
    int l = i < poff(1) ? 0 : (i < poff(2) ? 1 : 2);
    const int j = i - poff(l);
    const int CO = dim_co(l), CI = dim_ci(l);
    if (j >= wcount(l)) {
        a.bias[l][j - wcount(l)] = w;
        return;
    }
    const int co = j / (TAPS * CI), tap = (j / CI) % TAPS, ci = j % CI;
    // rows: the three z taps' output channels stacked (dz * CO + co); K:
    // the (dy, dx) tap, then the input channel
    a.fwd[l][core_idx((tap / 9) * CO + co, (tap % 9) * CI + ci, TAPS_XY * CI)] =
        __float2bfloat16_rn(w);
    if (l > 0) {
        const int tf = TAPS - 1 - tap;  // flipped tap
        a.bwd[l][core_idx((tf / 9) * CI + ci, (tf % 9) * CO + co, TAPS_XY * CO)] =
            __float2bfloat16_rn(w);
    }
}

// Centred box filter: coarse vertex I sits on fine vertex r I; per axis the
// weights are (1/2, 1, ..., 1, 1/2) / r over fine offsets -r/2..r/2.  One
// coarse value in FP64.
__device__ float filter_point(const float *__restrict__ fine, const Layout &L, int f, int r, int X,
                              int Y, int Z)
{
    const int h = r / 2;
    double acc = 0.0;
    for (int a = -h; a <= h; ++a) {
        const double wa = (a == -h || a == h) ? 0.5 : 1.0;
        const int z = ((r * Z + a) % L.nz + L.nz) % L.nz;
        for (int b = -h; b <= h; ++b) {
            const double wb = (b == -h || b == h) ? 0.5 : 1.0;
            const int y = ((r * Y + b) % L.ny + L.ny) % L.ny;
            for (int c = -h; c <= h; ++c) {
                const double wc = (c == -h || c == h) ? 0.5 : 1.0;
                const int x = ((r * X + c) % L.nx + L.nx) % L.nx;
                acc += wa * wb * wc * (double)fine[lidx(L, f, z, y, x)];
            }
        }
    }
    return (float)(acc / ((double)r * r * r));
}

// Any even r: one thread per coarse value.
__global__ void k_box_filter(const float *__restrict__ fine, Layout L, int nf, int r,
                             float *__restrict__ out)
{
    const int nc = L.nx / r;
    const long long nc3 = (long long)nc * nc * nc;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nc3 * nf)
        return;
    const int f = (int)(i / nc3);
    const long long q = i - f * nc3;
    const int Z = (int)(q / ((long long)nc * nc)), Y = (int)((q / nc) % nc), X = (int)(q % nc);
    out[i] = filter_point(fine, L, f, r, X, Y, Z);
}

// r = 2, 4, 8: a warp takes 32 x-consecutive coarse values of one row (f, Z, Y)
// and walks the (r + 1)^2 fine rows with 8- and 16-byte loads.  The sums are
// float-float (two_sum: every rounding error kept and added up, about 46
// significant bits) because the FP64 pipe, with its conversions, bounds the
// general kernel: (r + 1)^3 of both per value, 1022 us from 256^3 to 64^3, here
// 79 us (the fine state is 335 MB).  The weights and 1 / r^3 are powers of
// two.  A sum that is not finite is formed again in FP64.
template <int RR>
__global__ void __launch_bounds__(256) k_box_filter_ff(const float *__restrict__ fine, Layout L,
                                                       int nf, float *__restrict__ out)
{
    constexpr int H = RR / 2;
    static_assert(H <= GX, "the x ghosts cover the row ends");
    const int nc = L.nx / RR;
    const int segs = (nc + 31) / 32;  // warps per coarse row
    const long long wid = (long long)blockIdx.x * 8 + threadIdx.x / 32;
    if (wid >= (long long)nf * nc * nc * segs)
        return;
    const int X = (int)(wid % segs) * 32 + threadIdx.x % 32;
    const long long row = wid / segs;
    const int Y = (int)(row % nc), Z = (int)((row / nc) % nc), f = (int)(row / ((long long)nc * nc));
    const bool in = X < nc;
    const int x = RR * (in ? X : nc - 1);
    float hi = 0.f, lo = 0.f;
    auto add = [&](float &s, float &e, float v) {  // s + e += v
        float t, d;
        two_sum(s, v, t, d);
        s = t;
        e = __fadd_rn(e, d);
    };
#pragma unroll(RR <= 4 ? 2 * H + 1 : 1)
    for (int a = -H; a <= H; ++a) {
        int z = RR * Z + a;
        z = z < 0 ? z + L.nz : (z >= L.nz ? z - L.nz : z);
        const float wa = (a == -H || a == H) ? 0.5f : 1.f;
#pragma unroll
        for (int b = -H; b <= H; ++b) {
            int y = RR * Y + b;
            y = y < 0 ? y + L.ny : (y >= L.ny ? y - L.ny : y);
            const float w = (b == -H || b == H) ? 0.5f * wa : wa;
            const float *p = fine + lidx(L, f, z, y, x);
            float v[2 * H + 1];  // offsets -H .. H
            if constexpr (RR == 2) {
                const float2 c = __ldg(reinterpret_cast<const float2 *>(p));
                v[0] = __ldg(p - 1);
                v[1] = c.x;
                v[2] = c.y;
            } else if constexpr (RR == 4) {
                const float2 m = __ldg(reinterpret_cast<const float2 *>(p - 2));
                const float4 c = __ldg(reinterpret_cast<const float4 *>(p));
                v[0] = m.x;
                v[1] = m.y;
                v[2] = c.x;
                v[3] = c.y;
                v[4] = c.z;
            } else {
                const float4 m = __ldg(reinterpret_cast<const float4 *>(p - 4));
                const float4 c = __ldg(reinterpret_cast<const float4 *>(p));
                v[0] = m.x;
                v[1] = m.y;
                v[2] = m.z;
                v[3] = m.w;
                v[4] = c.x;
                v[5] = c.y;
                v[6] = c.z;
                v[7] = c.w;
                v[8] = __ldg(p + 4);
            }
            // the row: ends at half weight, then the others
            float s, e;
            two_sum(v[0], v[2 * H], s, e);
            s *= 0.5f;
            e *= 0.5f;
#pragma unroll
            for (int c = 1; c < 2 * H; ++c)
                add(s, e, v[c]);
            add(hi, lo, w * s);
            lo = __fadd_rn(lo, w * e);
        }
    }
    if (!in)
        return;
    const float sum = __fadd_rn(hi, lo);
    out[(((long long)f * nc + Z) * nc + Y) * nc + X] =
        isfinite(sum) ? sum * (1.f / (RR * RR * RR)) : filter_point(fine, L, f, RR, X, Y, Z);
}

}  // namespace cnn
}  // namespace gbfd

using namespace gbfd;
using namespace gbfd::cnn;

struct gbfd_cnn {
    int n, batch, npts_max;
    cudaStream_t stream;
    char *ws;
    size_t ws_bytes;
    float *w, *m, *v, *g;
    bf16 *fwd[3], *bwd[3];
    float *bias[3];
    float *norm;  // mean_in[5], std_in[5], std_out[5]
    bf16 *x0, *a1, *a2, *dy3, *dh2, *dh1;
    float4 *h1, *h2;  // pre-activations, quads of channels: [8][batch n^3]
    float *y3;
    float *parts;
    int nparts;
    double *lparts, *loss;
    int *derr;
    int adam_t;
    int grid_conv;      // CTAs per convolution launch (each walks its share of the tiles)
    int grid_default;   // one per SM
    // TMA maps of the convolution inputs (padded chunk-major activations)
    CUtensorMap map_x0, map_a1, map_a2, map_dy3, map_dh2;
    // and of the weight gradients' A (32 channels) and B operands
    CUtensorMap wa_a2, wa_dh2, wa_dh1, wb_dy3, wb_a1, wb_x0;
    int64_t launches;
    char err[512];
};

namespace {

thread_local char g_cnn_err[512];

void cerr(gbfd_cnn *c, const char *fmt, ...)
{
    char *buf = c ? c->err : g_cnn_err;
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, 512, fmt, ap);
    va_end(ap);
}

gbfd_status ccuda(gbfd_cnn *c, cudaError_t e, const char *what)
{
    cerr(c, "%s: %s (%s)", what, cudaGetErrorName(e), cudaGetErrorString(e));
    return GBFD_ERR_CUDA;
}

size_t al(size_t v) { return (v + 1023) & ~(size_t)1023; }

struct CnnPlan {
    size_t off[32];
    size_t total;
};

constexpr int kWgradParts = 296;  // most CTAs of the weight-gradient kernels

CnnPlan plan_for(int n, int batch)
{
    CnnPlan pl;
    const size_t np = (size_t)batch * n * n * n;
    const size_t npad = (size_t)batch * (n + 2) * (n + 2) * (n + 2);  // padded activations
    const size_t sizes[] = {
        kParams * 4, kParams * 4, kParams * 4, kParams * 4,  // w m v g
        (size_t)CH * TAPS * C0 * 2, (size_t)CH * TAPS * CH * 2, (size_t)C3 * TAPS * CH * 2,  // fwd
        (size_t)C0 * TAPS * CH * 2, (size_t)CH * TAPS * CH * 2, (size_t)CH * TAPS * C3 * 2,  // bwd
        CH * 4, CH * 4, C3 * 4, 64 * 4,                                   // biases, norm
        npad * C0 * 2, npad * CH * 2, npad * CH * 2, npad * C3 * 2, npad * CH * 2,
        npad * CH * 2,                                                    // bf16 acts
        np * CH * 4, np * CH * 4, np * 8 * 4,                             // h1 h2 y3
        (size_t)kWgradParts * wg::part_floats<true>() * 4,               // parts
        ((np + 255) / 256 + 8) * 8, 64, 256};
    size_t off = 0;
    const int cnt = sizeof(sizes) / sizeof(sizes[0]);
    for (int i = 0; i < cnt; ++i) {
        pl.off[i] = off;
        off = al(off + sizes[i]);
    }
    pl.total = off;
    return pl;
}

// Planes of a run: the length that gives the CTA with most runs the fewest input
// planes (each run reads two more than it writes).
int conv_run(int n, int nb, int ctas)
{
    const long long cols = (long long)nb * ((n + TYT - 1) / TYT) * ((n + TXT - 1) / TXT);
    int best = n;
    long long best_t = 1LL << 60;
    for (int chunks = 1; chunks <= n; ++chunks) {
        const int run = (n + chunks - 1) / chunks;
        const long long t = (cols * ((n + run - 1) / run) + ctas - 1) / ctas * (run + 2);
        if (t < best_t) {
            best_t = t;
            best = run;
        }
    }
    return best;
}

template <int CIN, int N, int EPI>
cudaError_t conv(gbfd_cnn *c, const CUtensorMap &xmap, ConvArgs a)
{
    using SM = ConvSmem<CIN, N, EPI>;
    const int n = a.n;
    const int nb = (int)(a.npts / ((long long)n * n * n));
    a.run = conv_run(n, nb, c->grid_conv);
    const long long runs = (long long)nb * ((n + TYT - 1) / TYT) * ((n + TXT - 1) / TXT) *
                           ((n + a.run - 1) / a.run);
    // persistent: one CTA per SM walking the runs (fewer on request),
    // launched so that its prologue overlaps the previous kernel's tail
    c->launches++;
    return launch_chained<k_conv_tc<CIN, N, EPI>>(
        dim3((unsigned)std::min<long long>(runs, c->grid_conv)), dim3(CONV_THREADS), SM::BYTES, false,
        c->stream, xmap, a);
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    }
    return fn;
}

// TMA map of a padded chunk-major activation of cin channels (B samples on
// an n^3 grid): dims (8 (n + 2) values = x and the 8 channels of a chunk,
// n + 2, (n + 2) B, cin / 8), box = one haloed plane of a conv column, (8 HX, HY,
// 1, cin / 8): 160-byte rows.
bool encode_act_map(CUtensorMap *m, const bf16 *base, int n, int B, int cin)
{
    PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
    if (!fn)
        return false;
    const cuuint64_t np2 = (cuuint64_t)(n + 2);
    const cuuint64_t dims[4] = {8 * np2, np2, np2 * (cuuint64_t)B, (cuuint64_t)(cin / 8)};
    const cuuint64_t strides[3] = {np2 * 16, np2 * np2 * 16, np2 * np2 * np2 * B * 16};
    const cuuint32_t box[4] = {8 * HX, HY, 1, (cuuint32_t)(cin / 8)};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<bf16 *>(base), dims, strides, box,
              estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// TMA maps of the weight gradients' operands (wgrad.cuh), boxes of one tile.
// A, 32 channels: (8 interior x points, chunk, z with its frame, interior y,
// sample).  B wide, 32 channels: (x, chunk, y with their frame, interior z,
// sample).  B narrow, chunk 0 only: (interior x, x shift, y with its frame,
// interior z, sample), the shift dimension one point (16 bytes) apart.
// Outside a map's extents the copy fills zeros.
enum { WG_A, WG_B_WIDE, WG_B_NARROW };
bool encode_wgrad_map(CUtensorMap *m, const bf16 *base, int n, int B, int kind)
{
    PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
    if (!fn)
        return false;
    const cuuint64_t N = (cuuint64_t)n, P = N + 2, row = P * 16, plane = P * row, vol = P * plane;
    const cuuint64_t chunk = vol * (cuuint64_t)B, nb = (cuuint64_t)B;
    const char *p = reinterpret_cast<const char *>(base) + (kind == WG_A ? row + 16 : plane);
    const cuuint64_t dims[3][5] = {
        {8 * N, 4, P, N, nb}, {8 * P, 4, P, N, nb}, {8 * N, 3, P, N, nb}};
    const cuuint64_t strides[3][4] = {
        {chunk, plane, row, vol}, {chunk, row, plane, vol}, {16, row, plane, vol}};
    const cuuint32_t box[3][5] = {{8 * wg::TX, 4, wg::AZ, wg::TY, 1},
                                  {8 * (wg::TX + 2), 4, wg::BY, wg::ZB, 1},
                                  {8 * wg::TX, 3, wg::BY, wg::ZB, 1}};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<char *>(p), dims[kind],
              strides[kind], box[kind], estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

cudaError_t pack(gbfd_cnn *c, const float *g, float lr)
{
    PackArgs a;
    a.w = c->w;
    a.m = c->m;
    a.v = c->v;
    a.g = g;
    a.lr = lr;
    a.b1 = 0.9f;
    a.b2 = 0.999f;
    a.eps = 1e-8f;
    a.bc1 = 1.f - powf(0.9f, (float)c->adam_t);
    a.bc2 = 1.f - powf(0.999f, (float)c->adam_t);
    for (int l = 0; l < 3; ++l) {
        a.fwd[l] = c->fwd[l];
        a.bwd[l] = c->bwd[l];
        a.bias[l] = c->bias[l];
    }
    c->launches++;
    return launch_chained<k_adam_pack>(dim3((kParams + 255) / 256), dim3(256), 0, false, c->stream, a);
}

cudaError_t stage_input(gbfd_cnn *c, const float *xs, int nf, int npts)
{
    return launch_chained<k_input_compact>(dim3((npts + 255) / 256), dim3(256), 0, false, c->stream,
                                           xs, nf, c->n, npts, c->batch, (const float *)c->norm,
                                           (const float *)(c->norm + 5), c->x0);
}

// forward of `npts` points whose layer-1 input is already in x0; `keep`
// saves the pre-activations for the backward pass (training only)
cudaError_t forward(gbfd_cnn *c, int npts, bool keep)
{
    ConvArgs a;
    memset(&a, 0, sizeof a);
    a.n = c->n;
    a.npts = npts;
    a.B = c->batch;
    a.dev_error = c->derr;
    a.wB = c->fwd[0];
    a.bias = c->bias[0];
    a.hsave = keep ? c->h1 : nullptr;
    a.yb = c->a1;
    cudaError_t e = conv<C0, CH, EPI_GELU>(c, c->map_x0, a);
    if (e != cudaSuccess)
        return e;
    a.wB = c->fwd[1];
    a.bias = c->bias[1];
    a.hsave = keep ? c->h2 : nullptr;
    a.yb = c->a2;
    e = conv<CH, CH, EPI_GELU>(c, c->map_a1, a);
    if (e != cudaSuccess)
        return e;
    a.wB = c->fwd[2];
    a.bias = c->bias[2];
    a.hsave = nullptr;
    a.yb = nullptr;
    a.yf = c->y3;
    return conv<CH, C3, EPI_LINEAR>(c, c->map_a2, a);
}

// Weight and bias gradients of one layer: A and B are the staged operands of
// wgrad.cuh (SWAP: A = X, B = dY), one CTA per SM (fewer on request).
template <int CO, int CI, bool WIDE, bool SWAP>
cudaError_t wgrad(gbfd_cnn *c, const CUtensorMap &amap, const CUtensorMap &bmap, int npts, float *g)
{
    const int n = c->n;
    wg::Args a;
    a.n = n;
    a.nb = (int)(npts / ((long long)n * n * n));
    a.bias_b = SWAP;
    a.part = c->parts;
    a.dev_error = c->derr;
    const long long ntiles = (long long)a.nb * ((n + wg::ZB - 1) / wg::ZB) *
                             ((n + wg::TY - 1) / wg::TY) * ((n + wg::TX - 1) / wg::TX);
    const int grid = (int)std::min<long long>(ntiles, c->nparts);
    constexpr int smem = wg::Smem<WIDE>::BYTES;
    cudaError_t e = launch_chained<wg::k_wgrad_tc<WIDE>>(dim3(grid), dim3(wg::THREADS), smem, false,
                                                         c->stream, amap, bmap, a);
    if (e != cudaSuccess)
        return e;
    c->launches += 2;
    return launch_chained<wg::k_wgrad_reduce<CO, CI, WIDE, SWAP>>(
        dim3((wg::part_floats<WIDE>() + 31) / 32), dim3(256), 0, false, c->stream,
        (const float *)c->parts, grid, g);
}

// loss, backward and gradients for `batch` samples (x0 and y3 from forward)
cudaError_t backward(gbfd_cnn *c, const float *xs, const float *ts, int nf, int batch)
{
    const int n3 = c->n * c->n * c->n, npts = batch * n3;
    const int blocks = (npts + 256 * LOSS_PTS - 1) / (256 * LOSS_PTS);
    const float *sout = c->norm + 10;
    c->launches += 2;
    cudaError_t e = launch_chained<k_loss>(dim3(blocks), dim3(256), 0, false, c->stream,
                                           (const float *)c->y3, xs, ts, sout, nf, c->n, npts,
                                           c->batch, 1.0f / ((float)NC * npts), c->dy3, c->lparts);
    if (e != cudaSuccess)
        return e;
    e = launch_chained<k_sum_double>(dim3(1), dim3(256), 0, false, c->stream,
                                     (const double *)c->lparts, blocks, c->loss);
    if (e != cudaSuccess)
        return e;
    // layer 3: weight gradient, then input gradient through GELU'(h2)
    e = wgrad<C3, CH, false, true>(c, c->wa_a2, c->wb_dy3, npts, c->g + poff(2));
    if (e != cudaSuccess)
        return e;
    ConvArgs a;
    memset(&a, 0, sizeof a);
    a.n = c->n;
    a.npts = npts;
    a.dev_error = c->derr;
    a.B = c->batch;
    a.wB = c->bwd[2];
    a.hprev = c->h2;
    a.yb = c->dh2;
    e = conv<C3, CH, EPI_DGELU>(c, c->map_dy3, a);
    if (e != cudaSuccess)
        return e;
    // layer 2
    e = wgrad<CH, CH, true, false>(c, c->wa_dh2, c->wb_a1, npts, c->g + poff(1));
    if (e != cudaSuccess)
        return e;
    a.wB = c->bwd[1];
    a.hprev = c->h1;
    a.yb = c->dh1;
    e = conv<CH, CH, EPI_DGELU>(c, c->map_dh2, a);
    if (e != cudaSuccess)
        return e;
    // layer 1: weight gradient only
    return wgrad<CH, C0, false, false>(c, c->wa_dh1, c->wb_x0, npts, c->g + poff(0));
}

gbfd_status check(gbfd_cnn *c, int batch)
{
    if (!c)
        return GBFD_ERR_INVALID_ARG;
    if (batch < 1 || batch > c->batch) {
        cerr(c, "batch %d outside 1..%d", batch, c->batch);
        return GBFD_ERR_INVALID_ARG;
    }
    return GBFD_OK;
}

}  // namespace

extern "C" {

size_t gbfd_cnn_workspace_bytes(int n, int batch)
{
    if (n < 4 || n > 512 || batch < 1 || (long long)batch * n * n * n > (1LL << 30))
        return 0;
    return plan_for(n, batch).total;
}

gbfd_status gbfd_cnn_init(int n, int batch, void *workspace, size_t workspace_bytes, void *stream,
                          gbfd_cnn **out)
{
    if (!out) {
        cerr(nullptr, "out is NULL");
        return GBFD_ERR_INVALID_ARG;
    }
    *out = nullptr;
    const size_t need = gbfd_cnn_workspace_bytes(n, batch);
    if (need == 0) {
        cerr(nullptr, "cnn: n must be in 4..512, batch >= 1, batch*n^3 <= 2^30");
        return GBFD_ERR_INVALID_ARG;
    }
    if (!workspace || ((uintptr_t)workspace & 1023) || workspace_bytes < need) {
        cerr(nullptr, "cnn: workspace must be 1024-byte aligned with >= %zu bytes", need);
        return GBFD_ERR_WORKSPACE;
    }
    gbfd_cnn *c = new (std::nothrow) gbfd_cnn();
    if (!c) {
        cerr(nullptr, "out of host memory");
        return GBFD_ERR_INVALID_ARG;
    }
    CnnPlan pl = plan_for(n, batch);
    c->n = n;
    c->batch = batch;
    c->npts_max = batch * n * n * n;
    c->stream = (cudaStream_t)stream;
    c->ws = (char *)workspace;
    c->ws_bytes = workspace_bytes;
    char *b = c->ws;
    int k = 0;
    c->w = (float *)(b + pl.off[k++]);
    c->m = (float *)(b + pl.off[k++]);
    c->v = (float *)(b + pl.off[k++]);
    c->g = (float *)(b + pl.off[k++]);
    for (int l = 0; l < 3; ++l)
        c->fwd[l] = (bf16 *)(b + pl.off[k++]);
    for (int l = 0; l < 3; ++l)
        c->bwd[l] = (bf16 *)(b + pl.off[k++]);
    for (int l = 0; l < 3; ++l)
        c->bias[l] = (float *)(b + pl.off[k++]);
    c->norm = (float *)(b + pl.off[k++]);
    c->x0 = (bf16 *)(b + pl.off[k++]);
    c->a1 = (bf16 *)(b + pl.off[k++]);
    c->a2 = (bf16 *)(b + pl.off[k++]);
    c->dy3 = (bf16 *)(b + pl.off[k++]);
    c->dh2 = (bf16 *)(b + pl.off[k++]);
    c->dh1 = (bf16 *)(b + pl.off[k++]);
    c->h1 = (float4 *)(b + pl.off[k++]);
    c->h2 = (float4 *)(b + pl.off[k++]);
    c->y3 = (float *)(b + pl.off[k++]);
    c->parts = (float *)(b + pl.off[k++]);
    c->lparts = (double *)(b + pl.off[k++]);
    c->loss = (double *)(b + pl.off[k++]);
    c->derr = (int *)(b + pl.off[k++]);
    c->adam_t = 0;
    c->launches = 0;
    c->err[0] = 0;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    c->grid_conv = c->grid_default = sms > 0 ? sms : 1;
    c->nparts = std::min(c->grid_default, kWgradParts);
    if (e == cudaSuccess &&
        !(encode_act_map(&c->map_x0, c->x0, n, batch, C0) &&
          encode_act_map(&c->map_a1, c->a1, n, batch, CH) &&
          encode_act_map(&c->map_a2, c->a2, n, batch, CH) &&
          encode_act_map(&c->map_dy3, c->dy3, n, batch, C3) &&
          encode_act_map(&c->map_dh2, c->dh2, n, batch, CH) &&
          encode_wgrad_map(&c->wa_a2, c->a2, n, batch, WG_A) &&
          encode_wgrad_map(&c->wa_dh2, c->dh2, n, batch, WG_A) &&
          encode_wgrad_map(&c->wa_dh1, c->dh1, n, batch, WG_A) &&
          encode_wgrad_map(&c->wb_dy3, c->dy3, n, batch, WG_B_NARROW) &&
          encode_wgrad_map(&c->wb_a1, c->a1, n, batch, WG_B_WIDE) &&
          encode_wgrad_map(&c->wb_x0, c->x0, n, batch, WG_B_NARROW))) {
        cerr(nullptr, "cnn init: TMA descriptor encoding failed");
        delete c;
        return GBFD_ERR_CUDA;
    }
    if (e == cudaSuccess)
        e = cudaMemsetAsync(c->ws, 0, pl.total, c->stream);
    // identity normalisation until set
    std::vector<float> nm(64, 0.f);
    for (int i = 0; i < 5; ++i)
        nm[5 + i] = nm[10 + i] = 1.f;
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(c->norm, nm.data(), 64 * 4, cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess)
        e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) {
        ccuda(nullptr, e, "cnn init");
        delete c;
        return GBFD_ERR_CUDA;
    }
    *out = c;
    return GBFD_OK;
}

gbfd_status gbfd_cnn_destroy(gbfd_cnn *c)
{
    delete c;
    return GBFD_OK;
}

gbfd_status gbfd_cnn_set_option(gbfd_cnn *c, int key, int64_t value)
{
    if (!c)
        return GBFD_ERR_INVALID_ARG;
    switch (key) {
    case GBFD_CNN_OPT_CONV_GRID:
        if (value < 0 || value > (1 << 20))
            break;
        c->grid_conv = value == 0 ? c->grid_default : (int)value;
        return GBFD_OK;
    case GBFD_CNN_OPT_WGRAD_PARTS:
        if (value < 0 || value > kWgradParts)
            break;
        c->nparts = value == 0 ? std::min(c->grid_default, kWgradParts) : (int)value;
        return GBFD_OK;
    default:
        break;
    }
    cerr(c, "cnn set_option: bad key %d or value %lld", key, (long long)value);
    return GBFD_ERR_INVALID_ARG;
}

gbfd_status gbfd_cnn_set_params(gbfd_cnn *c, const float *params)
{
    if (!c || !params) {
        cerr(c, "cnn set_params: NULL argument");
        return GBFD_ERR_INVALID_ARG;
    }
    std::vector<float> packed(kParams, 0.f);
    const float *src = params;
    for (int l = 0; l < 3; ++l) {
        const int CO = dim_co(l), CI = dim_ci(l);
        for (int o = 0; o < kRealOut[l]; ++o)
            for (int ci = 0; ci < kRealIn[l]; ++ci)
                for (int t = 0; t < TAPS; ++t)
                    packed[poff(l) + (o * TAPS + t) * CI + ci] = src[(o * kRealIn[l] + ci) * TAPS + t];
        src += kRealOut[l] * kRealIn[l] * TAPS;
        for (int o = 0; o < kRealOut[l]; ++o)
            packed[poff(l) + CO * TAPS * CI + o] = src[o];
        src += kRealOut[l];
    }
    cudaError_t e =
        cudaMemcpyAsync(c->w, packed.data(), kParams * 4, cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess)
        e = cudaMemsetAsync(c->m, 0, kParams * 4, c->stream);
    if (e == cudaSuccess)
        e = cudaMemsetAsync(c->v, 0, kParams * 4, c->stream);
    c->adam_t = 0;
    if (e == cudaSuccess)
        e = pack(c, nullptr, 0.f);
    if (e == cudaSuccess)
        e = cudaStreamSynchronize(c->stream);
    return e == cudaSuccess ? GBFD_OK : ccuda(c, e, "cnn set_params");
}

// unpack a padded parameter vector (device) into the real-size host layout
static gbfd_status unpack(gbfd_cnn *c, const float *dev, float *host)
{
    std::vector<float> packed(kParams);
    cudaError_t e =
        cudaMemcpyAsync(packed.data(), dev, kParams * 4, cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess)
        e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess)
        return ccuda(c, e, "cnn read parameters");
    float *dst = host;
    for (int l = 0; l < 3; ++l) {
        const int CO = dim_co(l), CI = dim_ci(l);
        for (int o = 0; o < kRealOut[l]; ++o)
            for (int ci = 0; ci < kRealIn[l]; ++ci)
                for (int t = 0; t < TAPS; ++t)
                    dst[(o * kRealIn[l] + ci) * TAPS + t] = packed[poff(l) + (o * TAPS + t) * CI + ci];
        dst += kRealOut[l] * kRealIn[l] * TAPS;
        for (int o = 0; o < kRealOut[l]; ++o)
            dst[o] = packed[poff(l) + CO * TAPS * CI + o];
        dst += kRealOut[l];
    }
    return GBFD_OK;
}

gbfd_status gbfd_cnn_get_params(gbfd_cnn *c, float *params)
{
    if (!c || !params) {
        cerr(c, "cnn get_params: NULL argument");
        return GBFD_ERR_INVALID_ARG;
    }
    return unpack(c, c->w, params);
}

int gbfd_cnn_param_count(void) { return kRealParams; }

gbfd_status gbfd_cnn_set_norm(gbfd_cnn *c, const float *mean_in, const float *std_in,
                              const float *std_out)
{
    if (!c || !mean_in || !std_in || !std_out) {
        cerr(c, "cnn set_norm: NULL argument");
        return GBFD_ERR_INVALID_ARG;
    }
    float nm[64] = {0};
    for (int i = 0; i < 5; ++i) {
        if (!(std_in[i] > 0) || !(std_out[i] > 0)) {
            cerr(c, "cnn set_norm: standard deviations must be > 0");
            return GBFD_ERR_INVALID_ARG;
        }
        nm[i] = mean_in[i];
        nm[5 + i] = std_in[i];
        nm[10 + i] = std_out[i];
    }
    cudaError_t e = cudaMemcpyAsync(c->norm, nm, sizeof nm, cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess)
        e = cudaStreamSynchronize(c->stream);
    return e == cudaSuccess ? GBFD_OK : ccuda(c, e, "cnn set_norm");
}

gbfd_status gbfd_cnn_forward(gbfd_cnn *c, const float *xs, int nf, int batch, float *ys)
{
    gbfd_status st = check(c, batch);
    if (st != GBFD_OK)
        return st;
    if (!xs || !ys || (nf != 4 && nf != 5)) {
        cerr(c, "cnn forward: bad arguments");
        return GBFD_ERR_INVALID_ARG;
    }
    const int n3 = c->n * c->n * c->n, npts = batch * n3;
    cudaError_t e = stage_input(c, xs, nf, npts);
    if (e == cudaSuccess)
        e = forward(c, npts, false);
    if (e == cudaSuccess) {
        k_output_compact<<<(npts + 255) / 256, 256, 0, c->stream>>>(c->y3, n3, npts, ys);
        e = cudaGetLastError();
    }
    c->launches += 2;
    return e == cudaSuccess ? GBFD_OK : ccuda(c, e, "cnn forward");
}

gbfd_status gbfd_cnn_gradients(gbfd_cnn *c, const float *xs, const float *ts, int nf, int batch,
                               float *grads, double *loss)
{
    gbfd_status st = check(c, batch);
    if (st != GBFD_OK)
        return st;
    if (!xs || !ts || (nf != 4 && nf != 5)) {
        cerr(c, "cnn gradients: bad arguments");
        return GBFD_ERR_INVALID_ARG;
    }
    const int n3 = c->n * c->n * c->n, npts = batch * n3;
    cudaError_t e = stage_input(c, xs, nf, npts);
    c->launches++;
    if (e == cudaSuccess)
        e = forward(c, npts, true);
    if (e == cudaSuccess)
        e = backward(c, xs, ts, nf, batch);
    double l = 0;
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(&l, c->loss, 8, cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess)
        e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess)
        return ccuda(c, e, "cnn gradients");
    if (loss)
        *loss = l / ((double)NC * npts);
    return grads ? unpack(c, c->g, grads) : GBFD_OK;
}

gbfd_status gbfd_cnn_train_step(gbfd_cnn *c, const float *xs, const float *ts, int nf, int batch,
                                float lr, double *loss)
{
    gbfd_status st = check(c, batch);
    if (st != GBFD_OK)
        return st;
    if (!xs || !ts || (nf != 4 && nf != 5) || !(lr >= 0)) {
        cerr(c, "cnn train_step: bad arguments");
        return GBFD_ERR_INVALID_ARG;
    }
    const int n3 = c->n * c->n * c->n, npts = batch * n3;
    cudaError_t e = stage_input(c, xs, nf, npts);
    c->launches++;
    if (e == cudaSuccess)
        e = forward(c, npts, true);
    if (e == cudaSuccess)
        e = backward(c, xs, ts, nf, batch);
    c->adam_t++;
    if (e == cudaSuccess)
        e = pack(c, c->g, lr);
    if (e == cudaSuccess && loss) {
        double l = 0;
        e = cudaMemcpyAsync(&l, c->loss, 8, cudaMemcpyDeviceToHost, c->stream);
        if (e == cudaSuccess)
            e = cudaStreamSynchronize(c->stream);
        *loss = l / ((double)NC * npts);
    }
    return e == cudaSuccess ? GBFD_OK : ccuda(c, e, "cnn train_step");
}

gbfd_status gbfd_cnn_apply(gbfd_cnn *c, gbfd_ctx *ctx)
{
    if (!c || !ctx)
        return GBFD_ERR_INVALID_ARG;
    float *st = nullptr;
    Layout L;
    int nf = 0;
    cudaStream_t s;
    if (!ctx_view(ctx, &st, &L, &nf, &s)) {
        cerr(c, "cnn apply: context must be FP32 with a cubic grid");
        return GBFD_ERR_UNSUPPORTED;
    }
    if (L.nx != c->n) {
        cerr(c, "cnn apply: grid %d does not match the network's %d", L.nx, c->n);
        return GBFD_ERR_INVALID_ARG;
    }
    const int n3 = c->n * c->n * c->n;
    // run on the solver's stream so the correction is ordered with its steps
    const cudaStream_t saved = c->stream;
    c->stream = s;
    cudaError_t e = launch_chained<k_input_state>(dim3((n3 + 255) / 256), dim3(256), 0, false, s,
                                                  (const float *)st, L, nf, c->batch,
                                                  (const float *)c->norm,
                                                  (const float *)(c->norm + 5), c->x0);
    if (e == cudaSuccess)
        e = forward(c, n3, false);
    if (e == cudaSuccess)
        e = launch_chained<k_apply>(dim3((n3 + 255) / 256), dim3(256), 0, false, s, st, L, nf,
                                    (const float *)c->y3, (const float *)(c->norm + 10));
    c->stream = saved;
    c->launches += 2;
    return e == cudaSuccess ? GBFD_OK : ccuda(c, e, "cnn apply");
}

gbfd_status gbfd_step_corrected(gbfd_ctx *ctx, gbfd_cnn *c, double dt, int nsteps)
{
    if (!ctx || !c || nsteps < 0)
        return GBFD_ERR_INVALID_ARG;
    for (int i = 0; i < nsteps; ++i) {
        gbfd_status st = gbfd_rk3_step(ctx, dt, 1);
        if (st != GBFD_OK)
            return st;
        st = gbfd_cnn_apply(c, ctx);
        if (st != GBFD_OK)
            return st;
    }
    return GBFD_OK;
}

gbfd_status gbfd_box_filter(gbfd_ctx *fine, int r, float *out)
{
    float *st = nullptr;
    Layout L;
    int nf = 0;
    cudaStream_t s;
    if (!fine || !out || r < 2 || r % 2)
        return GBFD_ERR_INVALID_ARG;
    if (!ctx_view(fine, &st, &L, &nf, &s) || L.nx % r)
        return GBFD_ERR_UNSUPPORTED;
    const int nc = L.nx / r;
    const long long cnt = (long long)nc * nc * nc * nf;
    const long long warps = (long long)nf * nc * nc * ((nc + 31) / 32);
    const unsigned wblocks = (unsigned)((warps + 7) / 8);
    if (r == 2)
        k_box_filter_ff<2><<<wblocks, 256, 0, s>>>(st, L, nf, out);
    else if (r == 4)
        k_box_filter_ff<4><<<wblocks, 256, 0, s>>>(st, L, nf, out);
    else if (r == 8)
        k_box_filter_ff<8><<<wblocks, 256, 0, s>>>(st, L, nf, out);
    else
        k_box_filter<<<(unsigned)((cnt + 255) / 256), 256, 0, s>>>(st, L, nf, r, out);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? GBFD_OK : GBFD_ERR_CUDA;
}

int64_t gbfd_cnn_launch_count(const gbfd_cnn *c) { return c ? c->launches : 0; }

const char *gbfd_cnn_last_error(const gbfd_cnn *c) { return c ? c->err : g_cnn_err; }

}  // extern "C"
