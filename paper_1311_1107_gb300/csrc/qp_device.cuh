// Device building blocks of libqedpic: kernel argument layout, Philox,
// field models, chi, table lookups and inverse-CDF sampling.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "qp_df.h"
#include "qp_internal.h"

namespace qp {

enum Prec { kFP64 = 0, kMixed = 1 };
constexpr int kTile = QP_STEP_TILE;  // particles per step tile = threads per block
constexpr int kWarps = kTile / 32;
constexpr int kDiagTile = 256;  // slots per block tile of the diagnostics

// ------------------------------------------------------------------ layout

struct SpeciesDev {
    double *x, *y, *z, *ux, *uy, *uz, *tau, *w, *chi;
    int32_t *nemit;
    int64_t *n_live;
    int64_t cap;
    int64_t id_base;     // global number of slot 0: particle id = id_base + slot
    int64_t id_split;    // > 0: slots from here on are id_append + (slot - id_split)
    int64_t id_append;
    int32_t present;
    int32_t slot_stats;  // index of this species' counter block
};

// The particle id of a slot: the counter of its random streams.
__device__ __forceinline__ int64_t particle_id(int64_t id_base, int64_t id_split,
                                               int64_t id_append, int64_t slot)
{
    return (id_split > 0 && slot >= id_split) ? id_append + (slot - id_split) : id_base + slot;
}
__device__ __forceinline__ int64_t particle_id(const SpeciesDev &S, int64_t slot)
{
    return particle_id(S.id_base, S.id_split, S.id_append, slot);
}

// Per-species event counters (device; atomics aggregated per block).
struct DevStats {
    unsigned long long n_emit, n_photon, n_photon_drop, n_subthreshold, n_pair, n_pair_drop,
        n_saturated, n_clamped, n_continuous;
    double e_subthreshold, e_dropped;
};

struct FieldDev {
    int32_t kind;
    double a0, w0, tau_fwhm, x_focus, t_focus, b0;
    const float *yee[6];
    int64_t nx, ny;
    double dx, dy, x0, y0;
    // YEE2D: 1/dx, 1/dy, x0/dx, y0/dy; GAUSSIAN, with zr = w0^2/2: 1/zr, 1/w0^2,
    // 2 ln2 / tau_fwhm^2, 1/(2 zr^2)
    double c[4];
};

struct TablesDev {
    const double *H, *Gs, *Ts, *Cg, *Cp;       // FP64
    const float *Hf, *Gsf, *Tsf;               // FP32 copies of the rate rows
    // CDF rows C and their complements Q = 1 - C as hi + lo float pairs
    const float2 *Cg2, *Cp2, *Qg2, *Qp2;
    const float *Eg, *Ep;                      // e^(-s_j) at the logit nodes
    // guide tables of the CDF rows (see guide_bucket): [half][row][bucket]
    const unsigned char *Gg, *Gp;
};

// Step constants of the mixed path as FP32 values or double-float pairs
// (split on the host), so the kernel needs no FP64 arithmetic for them.
struct MixedConsts {
    float xf_hi, xf_lo;         // x_focus
    float idx_hi, idx_lo, idy_hi, idy_lo;  // 1/dx, 1/dy (Yee grid)
    float x0s_hi, x0s_lo, y0s_hi, y0s_lo;  // x0/dx, y0/dy
    float h[2];                 // 0.5 q dt for electrons, positrons
    float dt, C_rate, inv_aS, tau0w, chi_th, gmin;
    float inv_aS_lo;            // 1/a_S - inv_aS: chi is scaled by the pair, so
                                // that no rounding of the constant biases every chi
    float a0, b0, zr, inv_zr, inv_w0sq, k_env;  // field shape (k_env = 2 ln2 / tau_fwhm^2)
    float nxf, nyf;                            // Yee grid size
};

// The step being taken: its index and time t = step dt, and the mixed path's
// constants of it.
struct StepTime {
    double t;
    uint64_t step;
    float t_hi, t_lo;           // t
    float tr_hi, tr_lo;         // t - t_focus (Gaussian pulse)
};

// Device-resident control block of a launch sequence: the tile ticket, the
// epoch that tags look-back words (it advances with every step), whether the
// launch has been given up (see abandon_launch), and the counts of blocks that
// have ended a step.  Blocks count in kDoneGroups group counters (one 32-byte
// sector each) and the last of each group in `done`: no counter sees more than
// a few tens of atomics at once.  Row 1 counts the end of a launch's last step,
// where every block comes by, row 0 the ends of the steps before it.  Between
// launches everything but the epoch is 0.
constexpr int kDoneGroups = 32;
// The spread of a launch's first tiles (spread_ticket): blocks met on each SM
// (SM ids modulo kSpreadSms) and as each SM's n-th, and blocks counted.
constexpr int kSpreadSms = 256, kSpreadRanks = 32;
struct StepCtl {
    unsigned ticket, epoch, abandoned, arrived;
    unsigned done[2];
    unsigned grp[2][kDoneGroups][8];
    unsigned sm_blocks[kSpreadSms], rank_blocks[kSpreadRanks];
};

constexpr int kMaxProblems = 64;  // problems (independent runs) per launch
// doubles of one append record (see the stash of qp_step.cuh), tiles a block
// has in flight, sub-tiles of 32 slots in a warp's part of a long tile
constexpr int kStashFieldsHost = 9 + QP_MAX_EMISSIONS;
constexpr int kStashBufs = 4;
constexpr int kSubTiles = 8;

// A launch of `subs` sub-tiles of 32 slots on `grid` blocks takes long tiles
// once every warp has about four of their parts of kSubTiles sub-tiles (below
// that the last parts leave warps idle), else short ones (see qp_step.cuh).
constexpr int kPartsPerWarp = 4;
__host__ __device__ inline bool long_tiles(long long subs, int grid)
{
    return subs >= (long long)kSubTiles * kPartsPerWarp * kWarps * grid;
}

// Steps of a launch of a single problem, and whether its stash has room for
// long tiles, in one word of the launch parameters (a word more there cost the
// shortest launches 5 %).
__host__ __device__ inline int32_t single_launch(int steps, bool long_ok)
{
    return steps * 2 + (long_ok ? 1 : 0);
}
__host__ __device__ inline int single_steps(int32_t launch) { return launch >> 1; }
__host__ __device__ inline bool single_long(int32_t launch) { return (launch & 1) != 0; }
// Steps a launch takes at most: other streams' kernels wait for it.
constexpr int kStepsPerLaunch = 8;

// Field kinds whose step kernel has the loop over long tiles (see kEmitInPlace).
__host__ __device__ constexpr bool has_long_tiles(int field_kind)
{
    return field_kind != QP_FIELD_YEE2D;
}

// Doubles of a block's stash: kStashBufs short tiles, or the three parts each
// warp has in flight of long ones.
__host__ __device__ inline size_t stash_words(bool long_ok)
{
    return (size_t)kStashFieldsHost * kTile * (long_ok ? 3 * kSubTiles : kStashBufs);
}

// One independent run stepped by a launch: its species, field, step
// constants, look-back scratch and control words.  A launch steps either a
// single problem passed by value (qp_step) or a device table of problems
// (a batch); the kernel copies the problem of each tile to shared memory.
struct Problem {
    SpeciesDev sp[3];                 // electron, positron, photon
    FieldDev f;
    MixedConsts mc;
    unsigned long long *lep_words;    // look-back words of the lepton chain
    unsigned long long *pho_words;    // look-back words of the photon chain
    long long *pending;               // [3] new live counts, applied by the last block
    long long *step_ctr;              // device-stepped: next step index
    long long *left_ctr;              // device-stepped: launches still to run (0 = idle)
    long long *work_ctr;              // device-stepped: live slots stepped so far
    double dt;
    uint64_t step, seed;              // step: the launch's first (a batch: step_ctr)
    double chi_th, gmin;
    int32_t pairs, max_emit;
    int32_t device_step;              // 1: step and activity from step_ctr/left_ctr
    int32_t pad;
};

// The append records of a batch's launches, and whether they have room for long
// tiles.  On the device: a captured launch takes what the batch has when it runs.
struct BatchStash {
    double *stash;
    unsigned long_ok, pad;
};

struct StepArgs {
    TablesDev tab;
    StepCtl *ctl;
    DevStats *stats;                  // counters, indexed by species handle
    int *status;                      // sticky status word
    double inv_aS, C_rate, tau0w;     // 1/a_S
    unsigned int spin_limit;          // bound of every device-side wait
    int32_t launch;                   // batch: problems in the table; single problem: see
                                      // single_launch
    const Problem *problems;          // a batch's device table
    union {
        double *stash;                // append records: stash_words() a block
        const BatchStash *batch;      // a batch's
    };
    Problem single;
};

// ------------------------------------------------------------------ status

__device__ __forceinline__ void raise_status(int *status, int code)
{
    // first error wins; a warning never overwrites an error
    int old = *((volatile int *)status);
    if (old < 0) return;
    if (code < 0)
        atomicCAS(status, old, code);
    else if (old == 0)
        atomicCAS(status, 0, code);
}

// ------------------------------------------------------------------ TMA bulk copies

__device__ __forceinline__ unsigned smem_addr(const void *p)
{
    return (unsigned)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(unsigned long long *bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count)
                 : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(unsigned long long *bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
                 "r"(bytes)
                 : "memory");
}

// Global -> shared bulk copy completing on `bar`; both addresses 16-byte
// aligned, bytes a multiple of 16.
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, unsigned bytes,
                                         unsigned long long *bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
            "r"(smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(unsigned long long *bar, unsigned parity)
{
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait for phase `parity` of `bar`; false on time-out.
__device__ __forceinline__ bool mbar_wait_bounded(unsigned long long *bar, unsigned parity,
                                                  unsigned limit)
{
#pragma unroll 1
    for (unsigned k = 0; k < limit; ++k)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

// ------------------------------------------------------------------ Philox4x32-10

__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k)
{
    // two rounds per iteration: a short loop body keeps the several inlined
    // draws of the step kernel small in the instruction cache
#pragma unroll 1
    for (int r = 0; r < 10; r += 2) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const unsigned hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
            const unsigned hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
            c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
            k.x += 0x9E3779B9u;
            k.y += 0xBB67AE85u;
        }
    }
    return c;
}

enum RngPurpose { kRngInit = 0, kRngEmit = 1, kRngPhotonTau = 2, kRngPair = 3, kRngPairPos = 4 };

// counter (slot lo, slot hi, step, species<<24 | purpose<<16 | k), key = seed
__device__ __forceinline__ uint4 draw(uint64_t seed, int species, int purpose, int64_t slot,
                                      uint64_t step, int k)
{
    const uint4 c = make_uint4((unsigned)((uint64_t)slot & 0xFFFFFFFFu),
                               (unsigned)((uint64_t)slot >> 32), (unsigned)(step & 0xFFFFFFFFu),
                               ((unsigned)species << 24) | ((unsigned)purpose << 16) |
                                   ((unsigned)k & 0xFFFFu));
    return philox4x32_10(c, make_uint2((unsigned)(seed & 0xFFFFFFFFu), (unsigned)(seed >> 32)));
}

// uniform in ]0,1] with 53 random bits
__device__ __forceinline__ double u53(unsigned a, unsigned b)
{
    const unsigned long long m = ((unsigned long long)(a >> 5) << 26) | (unsigned long long)(b >> 6);
    return (double)(m + 1ull) * 0x1.0p-53;
}

// ------------------------------------------------------------------ FP64 roots and reciprocals

// The FP64 pipe issues one warp instruction in about 20 cycles of an SM, so
// the FP64 path is bound by their number.  An IEEE square root or division
// takes about ten; here a Newton iteration of third order (Householder's
// method) from an FP32 seed takes three for a reciprocal and nine for a root
// with its reciprocal, the conversions of the seed being integer
// instructions.  Results are within one unit of the last place.  Arguments
// outside FP32's range go to the IEEE operations.  (With the gather's integer
// conversions and one sampling copy for both CDF rows: 2D foil 209 -> 119 us a
// step of 131072 e-, the 2e5-electron collision 316 -> 205 us.)

__device__ __forceinline__ bool in_fp32_range(double x)
{
    const unsigned e = ((unsigned)__double2hiint(x) >> 20) & 0x7FFu;
    return e - 903u <= 1143u - 903u;  // 2^-120 <= |x| < 2^121
}

static __device__ __noinline__ double rcp64_ieee(double x) { return 1.0 / x; }

__device__ __forceinline__ double rcp64(double x)
{
    if (!in_fp32_range(x)) return rcp64_ieee(x);
    const double y = finite_to_d(__fdividef(1.0f, hi_d(x)));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// 1/sqrt(x) for x > 0.
static __device__ __noinline__ double rsqrt64_ieee(double x) { return 1.0 / sqrt(x); }

__device__ __forceinline__ double rsqrt64(double x)
{
    if (!in_fp32_range(x)) return rsqrt64_ieee(x);
    const double y = finite_to_d(rsqrtf(hi_d(x)));
    const double e = fma(-(x * y), y, 1.0);
    return fma(y * e, fma(e, 0.375, 0.5), y);
}

// sqrt(x) from r = 1/sqrt(x) (x >= 0; 0 and infinity pass through).
__device__ __forceinline__ double root_of(double x, double r)
{
    if (!in_fp32_range(x)) return sqrt(x);
    const double s = x * r;
    return fma(fma(-s, s, x), 0.5 * r, s);
}

// ------------------------------------------------------------------ fields

template <typename R>
struct Vec3 {
    R x, y, z;
};

// Linear interpolation of the Yee components on their four staggered
// stencils (node/half-node in x and y): stencil (hx, hy) serves
// (0,0) Ez, (1,0) Ex and By, (0,1) Ey and Bx, (1,1) Bz.  Each stencil is
// bounds-checked once; nodes outside the grid contribute zero field.  The
// sum over the four nodes runs in the order (i,j), (i+1,j), (i,j+1),
// (i+1,j+1).
template <typename R>
struct YeeStencil {
    int base;      // index of node (i, j)
    int ix, iy;
    bool inside;   // all four nodes inside the grid
    R wx, wy;
};

template <typename R>
__device__ __forceinline__ R yee_interp(const float *__restrict__ F, const YeeStencil<R> &st,
                                        int nx, int ny)
{
    const R w00 = (R(1) - st.wx) * (R(1) - st.wy), w10 = st.wx * (R(1) - st.wy);
    const R w01 = (R(1) - st.wx) * st.wy, w11 = st.wx * st.wy;
    if (st.inside) {
        const float *p = F + st.base;
        R acc = R(0);
        acc += w00 * (R)__ldg(p);
        acc += w10 * (R)__ldg(p + 1);
        acc += w01 * (R)__ldg(p + nx);
        acc += w11 * (R)__ldg(p + nx + 1);
        return acc;
    }
    R acc = R(0);
    const R w[4] = {w00, w10, w01, w11};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int ii = st.ix + (k & 1), jj = st.iy + (k >> 1);
        if (ii < 0 || jj < 0 || ii >= nx || jj >= ny) continue;
        acc += w[k] * (R)__ldg(F + jj * nx + ii);
    }
    return acc;
}

// A node's value in the gather's type; to FP64 by integer instructions (the
// conversion unit is the FP64 pipe) unless it is denormal, infinite or NaN.
template <typename R>
__device__ __forceinline__ R node_value(float v)
{
    if constexpr (sizeof(R) == 8) {
        // exponents 255 and 0 become the lowest two; 0x01000000 is a zero
        const unsigned u = (__float_as_uint(v) << 1) + 0x01000000u;
        if (u < 0x02000000u && u != 0x01000000u) return (double)v;
        return finite_to_d(v);
    } else {
        return v;
    }
}

template <typename R>
__device__ __forceinline__ void yee_gather(const FieldDev &f, const int ix[2], const int iy[2],
                                           const R wx[2], const R wy[2], Vec3<R> &E, Vec3<R> &B)
{
    const int nx = (int)f.nx, ny = (int)f.ny;
    // one check for all four stencils (their nodes span min(ix)..max(ix)+1)
    const bool all_inside = min(ix[0], ix[1]) >= 0 && min(iy[0], iy[1]) >= 0 &&
                            max(ix[0], ix[1]) + 1 < nx && max(iy[0], iy[1]) + 1 < ny;
    YeeStencil<R> st[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int hx = k & 1, hy = k >> 1;
        st[k].ix = ix[hx];
        st[k].iy = iy[hy];
        st[k].wx = wx[hx];
        st[k].wy = wy[hy];
        st[k].inside = all_inside || (ix[hx] >= 0 && iy[hy] >= 0 && ix[hx] + 1 < nx &&
                                      iy[hy] + 1 < ny);
        st[k].base = iy[hy] * nx + ix[hx];
    }
    if (all_inside) {
        // the common case: the 24 loads of the six components are issued
        // together (one round trip to memory), then combined in the order
        // of yee_interp
        const int comp_st[6] = {1, 2, 0, 2, 1, 3};  // stencil of Ex Ey Ez Bx By Bz
        float v[6][4];
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            const float *p = f.yee[c] + st[comp_st[c]].base;
            v[c][0] = __ldg(p);
            v[c][1] = __ldg(p + 1);
            v[c][2] = __ldg(p + nx);
            v[c][3] = __ldg(p + nx + 1);
        }
        R out[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            const YeeStencil<R> &q = st[comp_st[c]];
            if constexpr (sizeof(R) == 8) {
                // a component that is zero around the particle (four of a
                // wave's six, for a whole warp) costs no FP64 instruction
                const unsigned any = __float_as_uint(v[c][0]) | __float_as_uint(v[c][1]) |
                                     __float_as_uint(v[c][2]) | __float_as_uint(v[c][3]);
                out[c] = R(0);
                if ((any << 1) == 0u) continue;
            }
            const R w00 = (R(1) - q.wx) * (R(1) - q.wy), w10 = q.wx * (R(1) - q.wy);
            const R w01 = (R(1) - q.wx) * q.wy, w11 = q.wx * q.wy;
            R acc = R(0);
            acc += w00 * node_value<R>(v[c][0]);
            acc += w10 * node_value<R>(v[c][1]);
            acc += w01 * node_value<R>(v[c][2]);
            acc += w11 * node_value<R>(v[c][3]);
            out[c] = acc;
        }
        E = {out[0], out[1], out[2]};
        B = {out[3], out[4], out[5]};
        return;
    }
    E.x = yee_interp<R>(f.yee[0], st[1], nx, ny);
    E.y = yee_interp<R>(f.yee[1], st[2], nx, ny);
    E.z = yee_interp<R>(f.yee[2], st[0], nx, ny);
    B.x = yee_interp<R>(f.yee[3], st[2], nx, ny);
    B.y = yee_interp<R>(f.yee[4], st[1], nx, ny);
    B.z = yee_interp<R>(f.yee[5], st[3], nx, ny);
}

// a / b rounded to nearest, from r = 1/b rounded to nearest (Markstein's
// correction): the last bit of a cell coordinate of a thousand is 1e-13 of a
// weight, far above the rounding of anything else in a step.
__device__ __forceinline__ double quotient64(double a, double b, double r)
{
    const double q = a * r;
    return fma(fma(-q, b, a), r, q);
}

// The cell index i of a coordinate a and its weight a - i, for the node grid
// (h = 0) and the half-node grid (h = 1, floor(a - 1/2)); i clamped to
// -2 .. n + 1, NaN to n + 1 (outside: no field).
__device__ __forceinline__ void cell64(double a, int n, int i[2], double w[2])
{
    const double f = floor(a);
    const bool nan = (__double_as_longlong(a) & 0x7FFFFFFFFFFFFFFFll) > 0x7FF0000000000000ll;
    const int c = nan ? n + 1 : __double2int_rz(f);  // saturates
    w[0] = a - f;
    const bool upper = __double2hiint(w[0]) >= 0x3FE00000;  // w >= 1/2
    w[1] = w[0] + (upper ? -0.5 : 0.5);  // exact
    i[0] = max(-2, min(n + 1, c));
    i[1] = max(-2, min(n + 1, nan ? n + 1 : upper ? c : max(c, -2) - 1));
}

// Fields of the FP64 path at (x, y, z, t).
template <int FK>
__device__ __forceinline__ void eval_field(const FieldDev &f, double x, double y, double z,
                                           double t, Vec3<double> &E, Vec3<double> &B)
{
    E = {0.0, 0.0, 0.0};
    B = {0.0, 0.0, 0.0};
    if constexpr (FK == QP_FIELD_PLANE) {
        const double v = f.a0 * cos(t - x);
        E.y = v;
        B.z = v;
    } else if constexpr (FK == QP_FIELD_GAUSSIAN) {
        const double xi = x - f.x_focus;
        const double eta = (t - f.t_focus) - xi;
        const double q = xi * f.c[0];
        const double ir = rsqrt64(1.0 + q * q), iwr2 = ir * ir;  // 1/sqrt(1 + q^2)
        const double r2w = (y * y + z * z) * iwr2;
        const double env = -r2w * f.c[1] - f.c[2] * eta * eta;
        const double phase = -eta + r2w * xi * f.c[3] - atan(q);
        const double v = f.a0 * ir * exp(env) * cos(phase);
        E.y = v;
        B.z = v;
    } else if constexpr (FK == QP_FIELD_UNIFORM_B) {
        B.z = f.b0;
    } else if constexpr (FK == QP_FIELD_YEE2D) {
        // linear interpolation of the six staggered components
        //   Ex(i+1/2,j) Ey(i,j+1/2) Ez(i,j) Bx(i,j+1/2) By(i+1/2,j) Bz(i+1/2,j+1/2);
        // nodes outside the grid contribute zero field
        int ix[2], iy[2];
        double wx[2], wy[2];
        cell64(quotient64(x - f.x0, f.dx, f.c[0]), (int)f.nx, ix, wx);
        cell64(quotient64(y - f.y0, f.dy, f.c[1]), (int)f.ny, iy, wy);
        yee_gather<double>(f, ix, iy, wx, wy, E, B);
    }
}

// ------------------------------------------------------------------ chi (Eq. 1)

// chi_e = sqrt(|gamma E + u x B|^2 - (u.E)^2) / a_S, in FP64
__device__ __forceinline__ double chi_e64(double Ex, double Ey, double Ez, double Bx, double By,
                                          double Bz, double ux, double uy, double uz, double g,
                                          double inv_aS)
{
    const double ax = g * Ex + (uy * Bz - uz * By);
    const double ay = g * Ey + (uz * Bx - ux * Bz);
    const double az = g * Ez + (ux * By - uy * Bx);
    const double ue = ux * Ex + uy * Ey + uz * Ez;
    const double s = ax * ax + ay * ay + az * az - ue * ue;
    return s > 0.0 ? root_of(s, rsqrt64(s)) * inv_aS : 0.0;
}

// ------------------------------------------------------------------ rate tables

// Index and exact interpolation weight of chi on a grid of 2^k nodes per
// octave starting at 2^-14, from the bits of chi (no logarithm): the node is
// 2^e (1 + m/2^k) with m the top k mantissa bits; the weight is the rest of
// the mantissa.  Requires 2^-14 <= chi < 2^10.
template <int KBITS>
__device__ __forceinline__ int grid_index64(double chi, double &f)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(chi);
    const int e = (int)((b >> 52) & 0x7FF) - 1023;
    const int m = (int)((b >> (52 - KBITS)) & ((1u << KBITS) - 1));
    // the rest of the mantissa, as 1.rest - 1
    const unsigned long long rest = (b << KBITS) & ((1ull << 52) - 1);
    f = __longlong_as_double((long long)((1023ull << 52) | rest)) - 1.0;
    return ((e - kChiExp0) << KBITS) + m;
}

template <int KBITS>
__device__ __forceinline__ int grid_index32(float chi, float &f)
{
    const unsigned b = __float_as_uint(chi);
    const int e = (int)((b >> 23) & 0xFF) - 127;
    const int m = (int)((b >> (23 - KBITS)) & ((1u << KBITS) - 1));
    f = (float)(b & ((1u << (23 - KBITS)) - 1)) * (1.0f / (float)(1u << (23 - KBITS)));
    return ((e - kChiExp0) << KBITS) + m;
}

constexpr double kChiLo = 0x1.0p-14, kChiHi = 0x1.0p10;
constexpr double kPi = 3.14159265358979323846;

// which: 0 H, 1 G (table holds G/chi), 2 T (table holds T exp(8/(3 chi)))
// V points at the (shared-memory) table of that quantity.
template <int WHICH>
__device__ __forceinline__ double rate64(const double *V, double chi, bool &clamped)
{
    if (WHICH == 2 && !(chi >= kPairChiMin)) return 0.0;
    if (!(chi >= kChiLo)) {
        if (WHICH == 0) return __dmul_rn(2.5 * kPi, chi);
        return __dmul_rn(__dmul_rn(2.0 * kPi / 1.7320508075688772, chi), chi);
    }
    double v, c = chi;
    if (chi >= kChiHi) {
        clamped = true;
        v = V[kNRate - 1];
        c = kChiHi;
    } else {
        double f;
        const int j = grid_index64<5>(chi, f);
        const double a = V[j], d = __dsub_rn(V[j + 1], a);
        v = __dadd_rn(a, __dmul_rn(f, d));
    }
    if (WHICH == 1) return __dmul_rn(v, c);
    if (WHICH == 2) return __dmul_rn(v, exp(-8.0 / 3.0 * rcp64(c)));
    return v;
}

template <int WHICH>
__device__ __forceinline__ float rate32(const float *V, float chi, bool &clamped)
{
    if (WHICH == 2 && !(chi >= (float)kPairChiMin)) return 0.0f;
    if (!(chi >= (float)kChiLo)) {
        if (WHICH == 0) return (float)(2.5 * kPi) * chi;
        return (float)(2.0 * kPi / 1.7320508075688772) * chi * chi;
    }
    float v, c = chi;
    if (chi >= (float)kChiHi) {
        clamped = true;
        v = V[kNRate - 1];
        c = (float)kChiHi;
    } else {
        float f;
        const int j = grid_index32<5>(chi, f);
        const float a = V[j];
        v = fmaf(f, V[j + 1] - a, a);
    }
    if (WHICH == 1) return v * c;
    if (WHICH == 2) return v * __expf(-8.0f / (3.0f * c));
    return v;
}

// ------------------------------------------------------------------ inverse CDF (Eq. 7)

// Guide tables: the search of a CDF row for xi starts from a node read from
// a small table instead of bisecting the row (8 dependent loads on the rare
// emission branch, which every later tile of the launch waits for through
// the look-back).  xi <= 1/2 is located in the row by xi itself, xi > 1/2 by
// eta = 1 - xi; the bucket of a value in (0, 1/2] is four per octave, from
// its exponent and two leading mantissa bits.  Lower-half entry: the last
// node with C < the bucket's lower edge; upper-half entry: the last node
// with 1 - C > the bucket's upper edge.  A forward scan then finds the same
// interval as a bisection would (the last node below xi).
constexpr int kGuideBuckets = 224;

__device__ __forceinline__ int guide_bucket(double x)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int e = (int)((b >> 52) & 0x7FF) - 1023;
    const int m = ((-1 - e) << 2) | (int)((b >> 50) & 3u);
    return min(max(m, 0), kGuideBuckets - 1);
}

__device__ __forceinline__ int guide_bucket(float x)
{
    const unsigned b = __float_as_uint(x);
    const int e = (int)((b >> 23) & 0xFF) - 127;
    const int m = ((-1 - e) << 2) | (int)((b >> 21) & 3u);
    return min(max(m, 0), kGuideBuckets - 1);
}

// Invert one CDF row C (kNNode logit nodes s_i = smin + ds i) at xi, in FP64.
// Emission rows follow u^(1/3) below the first node; pair rows clamp.
__device__ __forceinline__ double row_invert(const double *__restrict__ C,
                                             const unsigned char *__restrict__ guide, double xi,
                                             double smin, double ds, bool power_tail)
{
    const double c0 = __ldg(C);
    // the last node below xi: guide entry, then a forward scan (past the ends:
    // the first or the last node)
    double pos = 0.0, tail = 1.0;
    if (xi <= c0) {
        if (power_tail && c0 > 0.0) {
            const double r = xi * rcp64(c0);
            tail = r * r * r;
        }
    } else if (xi >= __ldg(C + kNNode - 1)) {
        pos = (double)(kNNode - 1);
    } else {
        int lo = xi <= 0.5 ? (int)__ldg(guide + guide_bucket(xi))
                           : (int)__ldg(guide + kNCdf * kGuideBuckets + guide_bucket(1.0 - xi));
#pragma unroll 1
        while (lo < kNNode - 2 && __ldg(C + lo + 1) < xi) ++lo;
        const double clo = __ldg(C + lo), chi_ = __ldg(C + lo + 1);
        pos = (double)lo + (xi - clo) * rcp64(chi_ - clo);
    }
    return tail * rcp64(1.0 + exp(-fma(ds, pos, smin)));
}

// Photon fraction u = chi_gamma / chi_e for chi_e (rows j, j+1 interpolated
// linearly in chi; below the grid the classical scaling u ~ chi).  One copy of
// the row inversion serves both rows.
__device__ __forceinline__ double sample_cdf(const double *__restrict__ rows,
                                             const unsigned char *__restrict__ guide, double chi,
                                             double xi, double smin, double span, bool emission,
                                             bool &clamped)
{
    const double ds = span / (kNNode - 1);
    const bool below = !(chi >= kChiLo);
    double f = 0.0;
    int j = 0, nrow = 1;
    if (!below) {
        if (chi >= kChiHi) {
            clamped = true;
            j = kNCdf - 1;
        } else {
            j = grid_index64<2>(chi, f);
            nrow = 2;
        }
    }
    double a = 0.0, b = 0.0;
#pragma unroll 1
    for (int k = 0; k < nrow; ++k, ++j) {
        b = row_invert(rows + j * kNNode, guide + j * kGuideBuckets, xi, smin, ds, emission);
        if (k == 0) a = b;
    }
    if (nrow == 2) return a + f * (b - a);
    return below && emission ? chi * (1.0 / kChiLo) * a : a;
}

// ------------------------------------------------------------------ FP32 inverse CDF with complement

// Mixed path: the same inversion in FP32, returning x and 1 - x, both
// accurate (1 - x from the logit, not by subtraction), so that the recoil
// (|p| - u gamma) and the pair split (1 - v) keep their precision when the
// photon or the electron takes nearly everything.
}  // namespace qp
