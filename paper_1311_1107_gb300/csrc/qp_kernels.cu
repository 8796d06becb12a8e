// Auxiliary kernels of libqedpic (sm_103a): initial optical depths,
// diagnostics, the bounded-wait self-test, and the launchers of all kernels
// (the step kernel itself is in qp_step.cuh).
#include <cuda_runtime.h>
#include <math.h>

#include "qp_kernels.h"
#include "qp_step.cuh"

namespace qp {

// -------------------------------------------------------------------- wait self-test

// Tile 1 of a chain whose tile 0 never publishes: the bounded wait must
// give up, raise QP_ERR_TIMEOUT and return.
__global__ void k_wait_selftest(unsigned long long *words, unsigned spin_limit, int *status)
{
    if (threadIdx.x < 32 && blockIdx.x == 0) {
        if (threadIdx.x == 0) words[0] = 0ull;
        __syncwarp();
        (void)chain_prefix(words, 1u, 0, 7u, spin_limit, status);
    }
}

cudaError_t launch_wait_selftest(unsigned long long *words, unsigned spin_limit, int *status,
                                 cudaStream_t st)
{
    k_wait_selftest<<<1, 32, 0, st>>>(words, spin_limit, status);
    return cudaGetLastError();
}

// The ends of a launch of three steps, one thread a block.  late 1: block 0 comes
// to the end of the first step only after another block's wait for it ran out;
// late 2: it counts as started only then.  Every other wait of a block is for
// blocks that do not wait for it (bounded all the same).
__global__ void k_step_end_selftest(StepCtl *ctl, int late, unsigned spin_limit, int *status)
{
    constexpr int kSteps = 3;
    const bool is_late = late && blockIdx.x == 0;
    unsigned epoch = __ldcg(&ctl->epoch);
    if (is_late)
        for (unsigned k = 0; k < (1u << 22) && !*(volatile unsigned *)&ctl->abandoned; ++k)
            __nanosleep(256);
    if (late == 2) (void)spread_ticket(ctl, spin_limit, status);
    for (int step = 0;; ++step) {
        if (last_block(ctl, step, kSteps)) end_step(ctl, epoch, step + 1 == kSteps);
        if (step + 1 == kSteps || !next_step(ctl, epoch, spin_limit, status)) return;
        ++epoch;
    }
}

// More blocks than groups of counters; all resident (a cooperative launch).
cudaError_t launch_step_end_selftest(StepCtl *ctl, int late, unsigned spin_limit, int *status,
                                     cudaStream_t st)
{
    void *args[] = {(void *)&ctl, (void *)&late, (void *)&spin_limit, (void *)&status};
    return cudaLaunchCooperativeKernel((const void *)k_step_end_selftest, dim3(2 * kDoneGroups + 3),
                                       dim3(1), args, 0, st);
}

// -------------------------------------------------------------------- initial optical depth

__global__ void k_init_tau(double *tau, int64_t first, int64_t count, int64_t id_base,
                           int64_t id_split, int64_t id_append, uint64_t seed, int species)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < count; k += stride) {
        const int64_t i = first + k;
        const uint4 r =
            draw(seed, species, kRngInit, particle_id(id_base, id_split, id_append, i), 0, 0);
        tau[i] = -log(u53(r.x, r.y));
    }
}

// -------------------------------------------------------------------- diagnostics

// Fixed-order reduction: block b takes tiles b, b + G, ...; every thread sums
// its own elements in order, every warp its histogram slot after slot, and the
// sums over lanes, warps and blocks have a fixed shape, so the result is
// independent of timing.  A second launch sums the blocks' partials and puts
// everything the host reads side by side.
//   Bound by the FP64 pipe (an instruction of a warp takes it 20 cycles), so
// the live count is an integer, the bin of log10(gamma) comes from an FP32
// logarithm except next to a bin's edge, the root is a Newton iteration, the
// weights of distinct bins are added by one instruction, and the threads' sums
// are added scalar by scalar with every lane at work (a butterfly of all of
// them is four times the adds).  Before, one thread a bin walked the tile's
// 256 slots and one thread an output the 256 blocks: 31 + 15 us for the
// species of a cascade of 16384 electrons, now 10 + 4.
constexpr int kDiagScalars = 8;  // n_alive, weight, energy, px, py, pz, w chi, (spare)
constexpr int kDiagSums = 6;     // those of them that threads sum in FP64
constexpr int kDiagWarps = kDiagTile / 32;
static_assert(kDiagScalars + QP_HIST_BINS == kDiagWords, "words of a partial");
static_assert(kDiagTile == 32 * kDiagSums + QP_HIST_BINS, "a warp a sum, a thread a bin");

// The bin of g = sqrt(g2), gamma or |u|, in the spectrum: log10 over its range,
// values outside it in the first and the last bin.
__device__ __forceinline__ int hist_bin(double g, double g2)
{
    constexpr double kScale = QP_HIST_BINS / (QP_HIST_LOG10_MAX - QP_HIST_LOG10_MIN);
    if (!(g > 0.0)) return 0;
    if (in_fp32_range(g)) {
        // a few 1e-6 off: sure away from the edges
        const float f = (log10f(hi_d(g)) - (float)QP_HIST_LOG10_MIN) * (float)kScale;
        if (fabsf(f - rintf(f)) > 1e-3f && f > 0.0f && f < (float)QP_HIST_BINS) return (int)f;
    }
    double b = (log10(sqrt(g2)) - QP_HIST_LOG10_MIN) * kScale;
    b = b < 0.0 ? 0.0 : (b > QP_HIST_BINS - 1 ? QP_HIST_BINS - 1 : b);
    return (int)b;
}

__global__ void __launch_bounds__(kDiagTile) k_diag_partial(SpeciesDev S, int is_photon,
                                                            double *partials)
{
    __shared__ double s_hist[kDiagWarps][QP_HIST_BINS];
    __shared__ double s_sum[kDiagSums][kDiagTile];
    __shared__ unsigned s_alive[kDiagWarps];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int64_t n = *S.n_live;
    n = n < 0 ? 0 : (n > S.cap ? S.cap : n);
    if ((int64_t)blockIdx.x * kDiagTile >= n) return;  // k_diag_final knows
    for (int k = lane; k < QP_HIST_BINS; k += 32) s_hist[warp][k] = 0.0;
    __syncwarp();
    double acc[kDiagSums] = {0, 0, 0, 0, 0, 0};
    unsigned alive = 0u;  // the warp's
    for (int64_t base = (int64_t)blockIdx.x * kDiagTile; base < n; base += (int64_t)gridDim.x * kDiagTile) {
        const int64_t i = base + tid;
        int bin = -1;
        double w = 0.0;
        if (i < n) {
            const double tau = S.tau[i];
            const double ux = S.ux[i], uy = S.uy[i], uz = S.uz[i], wi = S.w[i];
            if (!is_photon || tau >= 0.0) {
                const double p2 = ux * ux + uy * uy + uz * uz;
                const double g2 = is_photon ? p2 : 1.0 + p2;
                const double g = root_of(g2, rsqrt64(g2));
                w = wi;
                acc[0] += w;
                acc[1] += w * g;
                acc[2] += w * ux;
                acc[3] += w * uy;
                acc[4] += w * uz;
                if (S.chi) acc[5] += w * S.chi[i];
                bin = hist_bin(g, g2);
            }
        }
        alive += __popc(__ballot_sync(0xFFFFFFFFu, bin >= 0));
        // the lanes that share a bin in turn, those of distinct bins together
        const unsigned peers = __match_any_sync(0xFFFFFFFFu, bin);
        int turn = bin >= 0 ? __popc(peers & ((1u << lane) - 1u)) : 32;
        while (__any_sync(0xFFFFFFFFu, turn < 32)) {
            if (turn == 0) s_hist[warp][bin] += w;
            turn = turn > 0 && turn < 32 ? turn - 1 : 32;
            __syncwarp();
        }
    }
#pragma unroll
    for (int k = 0; k < kDiagSums; ++k) s_sum[k][tid] = acc[k];
    if (lane == 0) s_alive[warp] = alive;
    __syncthreads();
    double *out = partials + (size_t)blockIdx.x * kDiagWords;
    if (warp < kDiagSums) {
        double v = 0.0;
#pragma unroll
        for (int m = 0; m < kDiagWarps; ++m) v += s_sum[warp][32 * m + lane];
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, d);
        if (lane == 0) out[1 + warp] = v;
    } else {
        const int b = tid - 32 * kDiagSums;
        double v = 0.0;
#pragma unroll
        for (int m = 0; m < kDiagWarps; ++m) v += s_hist[m][b];
        out[kDiagScalars + b] = v;
    }
    if (tid == 0) {
        int64_t c = 0;
        for (int m = 0; m < kDiagWarps; ++m) c += s_alive[m];
        out[0] = (double)c;
        out[kDiagScalars - 1] = 0.0;
    }
}

// A block sums kFinalWords words of the partials of the blocks that had a
// tile: 32 threads a word, then over the lanes and warps of the word.  (One
// block for all words spends 11 us in its SM's FP64 pipe.)
constexpr int kFinalWords = 8, kFinalThreads = 256, kFinalRows = kFinalThreads / kFinalWords;
static_assert(kDiagWords % kFinalWords == 0, "blocks of whole words");

__global__ void __launch_bounds__(kFinalThreads) k_diag_final(SpeciesDev S, int blocks, DiagOut o)
{
    __shared__ double s_sum[kFinalThreads / 32][kFinalWords];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int word = tid % kFinalWords, k = blockIdx.x * kFinalWords + word;
    int64_t n = *S.n_live;
    if (blockIdx.x == 0 && tid == 0) {
        if (o.stats) o.out->stats = *o.stats;
        o.out->n_live = n;
        o.out->status = o.status ? *o.status : 0;
    }
    n = n < 0 ? 0 : (n > S.cap ? S.cap : n);
    const int64_t tiles = (n + kDiagTile - 1) / kDiagTile;
    const int used = tiles < blocks ? (int)tiles : blocks;
    double v = 0.0;
#pragma unroll 4
    for (int b = tid / kFinalWords; b < used; b += kFinalRows) v += o.partials[(size_t)b * kDiagWords + k];
#pragma unroll
    for (int d = 16; d >= kFinalWords; d >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, d);
    if (lane < kFinalWords) s_sum[warp][word] = v;
    __syncthreads();
    if (tid < kFinalWords) {
        v = 0.0;
#pragma unroll
        for (int w = 0; w < kFinalThreads / 32; ++w) v += s_sum[w][tid];
        o.out->sums[k] = v;
    }
}

// -------------------------------------------------------------------- launchers

static const void *step_fn(int precision, int fk, bool batch)
{
    return precision == QP_MIXED ? step_kernel_mixed(fk, batch) : step_kernel_fp64(fk, batch);
}

size_t step_smem_bytes(int precision, int field_kind)
{
    return precision == QP_MIXED ? step_smem_mixed(field_kind) : step_smem_fp64(field_kind);
}

int step_blocks_per_sm(int precision, int field_kind, bool batch)
{
    const void *fn = step_fn(precision, field_kind, batch);
    if (!fn) return 1;
    const size_t smem = step_smem_bytes(precision, field_kind);
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
        cudaSuccess)
        return 1;
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, kTile, smem) != cudaSuccess)
        return 1;
    return nb < 1 ? 1 : nb;
}

cudaError_t launch_step(const StepArgs &a, int precision, int field_kind, bool batch, int grid,
                        cudaStream_t st)
{
    const void *fn = step_fn(precision, field_kind, batch);
    if (!fn) return cudaErrorInvalidValue;
    const size_t smem = step_smem_bytes(precision, field_kind);
    void *args[] = {(void *)&a};
    // a single problem on the mixed path takes fixed first tiles, and a launch
    // of several steps meets at their ends: both need every block resident at
    // once, which a cooperative launch guarantees (or fails to launch)
    if (!batch && (precision == QP_MIXED || single_steps(a.launch) > 1))
        return cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(kTile), args, smem, st);
    return cudaLaunchKernel(fn, dim3(grid), dim3(kTile), args, smem, st);
}

static int bits_of(unsigned long long v)
{
    int b = 0;
    while (v) {
        ++b;
        v >>= 1;
    }
    return b;
}

int fused_key_bits(int K, long long tiles, int *ordinal_bits)
{
    const int ob = bits_of((unsigned long long)(tiles > 0 ? tiles : 1) * 32ull - 1ull);
    if (ordinal_bits) *ordinal_bits = ob;
    return bits_of((unsigned long long)(K > 1 ? K - 1 : 0)) + ob + kEmitBits;
}

// Warps an SM up to which a fused window's tiles of 32 leptons are split into
// warps of fewer lanes.  A window is a chain of K steps a warp, each as long as
// the emission loops of its slowest lane, and a few thousand leptons leave most
// of the chip idle: fewer lanes a warp meet fewer of them.  On the FP64 path a
// warp's instruction takes the pipe 20 cycles however few its lanes, so the
// line lies lower.  Measured, us a window, whole tiles and split up to 2 / 4 /
// 8 / 16 warps an SM:
//   mixed  4096 leptons x 250 steps 1519: 1265 / 1024 /  935 /  988
//          9000 x 100                723:  714 /  631 /  564 /  585
//         20000 x 100                793:  787 /  792 /  788 /  739
//   FP64   1500 x 200               3011: 2083 / 1755 / 1814 / 1809
//          4096 x 250               3811: 3263 / 2655 / 3235 / 5222
//          9000 x 100               1638: 1634 / 1500 / 1871 / 2724
constexpr int kFusedWarpsMixed = 8, kFusedWarpsFp64 = 4;

cudaError_t launch_fused(const StepArgs &a, int precision, int field_kind, int K,
                         long long tiles_e, long long tiles, void *scratch, int order_grid,
                         long long *win, int num_sms, cudaStream_t st)
{
    const bool mixed = precision == QP_MIXED;
    const void *lep = mixed ? fused_kernel_mixed(field_kind) : fused_kernel_fp64(field_kind);
    const void *photons = mixed ? fused_photons_mixed() : fused_photons_fp64();
    if (!lep) return cudaErrorInvalidValue;
    const SpeciesDev &Ph = a.single.sp[2];
    FusedArgs f{};
    f.a = a;
    f.K = K;
    const int key_bits = fused_key_bits(K, tiles, &f.ob);
    f.tiles_e = tiles_e;
    f.tiles = tiles;
    f.fs = fused_scratch(scratch, Ph.present ? Ph.cap : 0, order_grid, key_bits);
    f.win = win;
    void *args[] = {(void *)&f};
    const long long resident = (long long)num_sms * 32;
    const int most = mixed ? kFusedWarpsMixed : kFusedWarpsFp64;
    while (f.split < 5 && (tiles << (f.split + 1)) <= (long long)most * num_sms) ++f.split;
    const long long warps = tiles << f.split;
    const unsigned grid = (unsigned)(warps < resident ? (warps > 0 ? warps : 1) : resident);
    cudaError_t e = cudaMemsetAsync(f.fs.alloc, 0, sizeof(long long), st);
    if (e == cudaSuccess) e = cudaLaunchKernel(lep, dim3(grid), dim3(32), args, 0, st);
    if (e == cudaSuccess) e = launch_fused_order(Ph, scratch, order_grid, key_bits, win, a.status, st);
    const long long cap = Ph.present ? Ph.cap : 0;
    if (e == cudaSuccess && cap > 0) {
        long long pb = (cap + 255) / 256;
        if (pb > (long long)num_sms * 8) pb = (long long)num_sms * 8;
        e = cudaLaunchKernel(photons, dim3((unsigned)pb), dim3(256), args, 0, st);
    }
    return e;
}

cudaError_t launch_init_tau(double *tau, int64_t first, int64_t count, int64_t id_base,
                            int64_t id_split, int64_t id_append, uint64_t seed, int species,
                            cudaStream_t st)
{
    if (count <= 0) return cudaSuccess;
    int64_t blocks = (count + kDiagTile - 1) / kDiagTile;
    if (blocks > 4096) blocks = 4096;
    k_init_tau<<<(int)blocks, kDiagTile, 0, st>>>(tau, first, count, id_base, id_split,
                                                  id_append, seed, species);
    return cudaGetLastError();
}

cudaError_t launch_diag(const SpeciesDev &S, int is_photon, const DiagOut &o, cudaStream_t st)
{
    // no more blocks than tiles of the capacity
    const int64_t tiles = (S.cap + kDiagTile - 1) / kDiagTile;
    const int blocks = (int)(tiles < 1 ? 1 : tiles < kDiagBlocks ? tiles : kDiagBlocks);
    k_diag_partial<<<blocks, kDiagTile, 0, st>>>(S, is_photon, o.partials);
    k_diag_final<<<kDiagWords / kFinalWords, kFinalThreads, 0, st>>>(S, blocks, o);
    return cudaGetLastError();
}

// -------------------------------------------------------------------- pulse refill

// One launch: each block fills a tile of 32 columns x kPulseRows rows.  Its
// column factors (for the E_y and the B_z staggering) and row radii go to
// shared memory first: E = A exp(-c r^2) cos(phi + kappa r^2) with
// A = a0 (1 + q^2)^(-1/4) exp(-2 ln2 eta^2/tau^2), c = 1/(w0^2 (1 + q^2)),
// kappa = xi / (2 (xi^2 + zr^2)), phi = -eta - atan(q)/2.  Only eta and the
// phase reduction modulo 2 pi are FP64 (the phase is hundreds of radians);
// the factors and the nodes are FP32.
constexpr int kPulseRows = 64;

__global__ void __launch_bounds__(256) k_pulse_fill(Pulse2DDev p, int64_t nx, int64_t ny,
                                                    double dx, double dy, double x0, double y0,
                                                    double t, float *ey, float *bz)
{
    __shared__ float4 s_col[64];
    __shared__ float s_r2[kPulseRows];
    const int tid = threadIdx.x;
    const int64_t i0 = (int64_t)blockIdx.x * 32, j0 = (int64_t)blockIdx.y * kPulseRows;
    if (tid < 64) {
        const int s = tid >> 5;  // 0: E_y column, 1: B_z column (half a cell further)
        const int64_t i = i0 + (tid & 31);
        const double xi = x0 + ((double)i + 0.5 * s) * dx - p.x_focus;
        const double eta = (t - p.t_focus) - xi;
        const float zr = (float)(0.5 * p.w0 * p.w0);
        const float xf = (float)xi, ef = (float)eta;
        const float q = xf / zr, wr2 = 1.0f + q * q;
        const float tau = (float)p.tau_fwhm;
        const float A = (float)p.a0 * rsqrtf(sqrtf(wr2)) *
                        expf(-1.3862943611198906f * ef * ef / (tau * tau));
        // -eta reduced modulo 2 pi in FP64, then the Gouy phase
        const double red = -eta - 6.283185307179586477 * rint(-eta * 0.15915494309189533577);
        const float phi = (float)red - 0.5f * atanf(q);
        s_col[tid] = make_float4(A, 1.0f / ((float)(p.w0 * p.w0) * wr2),
                                 xf / (2.0f * (xf * xf + zr * zr)), phi);
    } else if (tid < 64 + kPulseRows) {
        const int64_t j = j0 + (tid - 64);
        const double r = y0 + ((double)j + 0.5) * dy - p.y_axis;
        s_r2[tid - 64] = (float)(r * r);
    }
    __syncthreads();
    const int c = tid & 31;
    const int64_t i = i0 + c;
    if (i >= nx) return;
    const float4 e = s_col[c], b = s_col[32 + c];
    for (int r = tid >> 5; r < kPulseRows; r += 8) {
        const int64_t j = j0 + r;
        if (j >= ny) break;
        const float r2 = s_r2[r];
        const int64_t k = j * nx + i;
        ey[k] = e.x * expf(-e.y * r2) * cosf(fmaf(e.z, r2, e.w));
        bz[k] = b.x * expf(-b.y * r2) * cosf(fmaf(b.z, r2, b.w));
    }
}

cudaError_t launch_pulse_fill(const Pulse2DDev &p, int64_t nx, int64_t ny, double dx, double dy,
                              double x0, double y0, double t, float *ey, float *bz,
                              cudaStream_t st)
{
    if (nx <= 0 || ny <= 0) return cudaSuccess;
    const dim3 grid((unsigned)((nx + 31) / 32), (unsigned)((ny + kPulseRows - 1) / kPulseRows));
    k_pulse_fill<<<grid, 256, 0, st>>>(p, nx, ny, dx, dy, x0, y0, t, ey, bz);
    return cudaGetLastError();
}

}  // namespace qp
