// The step kernel of libqedpic (sm_103a), instantiated per precision in
// qp_step_fp64.cu and qp_step_mixed.cu.
//
// One launch of the persistent kernel k_step takes one or several QED particle
// steps.  Its blocks take tiles from one atomic ticket over a single tile
// space: per problem, first the electron tiles, then the positron tiles
// (together: the lepton chain), then the photon tiles (the photon chain).
//   lepton tile : gather, Boris, chi_e, Sokolov or optical depth + emission,
//                 position update; new photons appended in slot order;
//   photon tile : chi_gamma, pair optical depth, decay into an e-/e+ pair
//                 appended in slot order, ballistic motion.
// Lepton tiles only append photons at slots >= the photon count of the step
// start and photon tiles only append leptons at slots >= the lepton counts,
// so the two chains never touch the same slots and both run in the same
// step.  The live counts are read-only during a step; the last block to
// finish it applies the new counts, resets the ticket and advances the epoch
// (device memory), which tags the look-back words: no memset and no host-side
// state between steps, so a step can be replayed in a CUDA graph.  Where a
// launch takes several steps the others wait for that epoch: it saves the gap
// between two launches and the tables' staging (256-electron plane wave: 42 ->
// 37 us a step).
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include <stddef.h>

#include <type_traits>

#include "qp_device.cuh"
#include "qp_kernels.h"
#include "qp_mixed.cuh"

namespace qp {

namespace {

// Look-back word: epoch (24 bits) | flag (2 bits) | value (38 bits).
constexpr int kEpochShift = 40, kFlagShift = 38;
constexpr unsigned long long kValMask = (1ull << kFlagShift) - 1;
constexpr unsigned kEpochMask = 0xFFFFFFu;
constexpr unsigned kFlagAgg = 1u, kFlagPre = 2u;

__device__ __forceinline__ unsigned long long make_word(unsigned epoch, unsigned flag,
                                                        long long value)
{
    return ((unsigned long long)(epoch & kEpochMask) << kEpochShift) |
           ((unsigned long long)flag << kFlagShift) | ((unsigned long long)value & kValMask);
}

__device__ __forceinline__ unsigned long long ld_volatile(const unsigned long long *p)
{
    return *((const volatile unsigned long long *)p);
}

// *p += v at GPU scope with acquire-release semantics; returns the old value
__device__ __forceinline__ unsigned atom_add_acq_rel(unsigned *p, unsigned v)
{
    unsigned old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;"
                 : "=r"(old)
                 : "l"(p), "r"(v)
                 : "memory");
    return old;
}

__device__ __forceinline__ void st_release(unsigned *p, unsigned v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// The control block as a launch finds it, its epoch past every tag that a step
// of this launch has used; one thread, once every block has counted its end.
__device__ __noinline__ void clear_ctl(StepCtl *ctl)
{
    const unsigned epoch = *(volatile unsigned *)&ctl->epoch;
    unsigned *const w = reinterpret_cast<unsigned *>(ctl);
#pragma unroll 1
    for (int k = 0; k < (int)(sizeof(StepCtl) / sizeof(unsigned)); ++k)
        *(volatile unsigned *)(w + k) = w + k == &ctl->epoch ? epoch + 1u : 0u;
}

// One thread counts its block's end of a step (of a launch's last step: fin);
// true in the last block.  The counts are acquire-release atomics: a count
// releases the block's writes (every thread's: the barrier that closed its last
// flush orders them before this thread's count) and the group's last count
// acquires the group's, so the last block sees every block's pending counts.
__device__ __forceinline__ bool count_block(StepCtl *ctl, bool fin)
{
    const unsigned g = blockIdx.x % kDoneGroups;
    const unsigned in_group = (gridDim.x - 1 - g) / kDoneGroups + 1;
    const unsigned groups = gridDim.x < kDoneGroups ? gridDim.x : kDoneGroups;
    bool last = false;
    if (atom_add_acq_rel(&ctl->grp[fin][g][0], 1u) == in_group - 1) {
        ctl->grp[fin][g][0] = 0u;  // every block of the group has counted
        last = atom_add_acq_rel(&ctl->done[fin], 1u) == groups - 1;
    }
    return last;
}

// The last block of a launch of several steps finds whether it was abandoned
// (one thread): it then has no whole step to publish, and leaves the control
// block clean, as no block has anything left to count: each has ended the
// launch's last step or abandoned.
__device__ __forceinline__ bool was_abandoned(StepCtl *ctl)
{
    if (!*(volatile unsigned *)&ctl->abandoned) return false;
    clear_ctl(ctl);
    return true;
}

// One thread ends its block's step `step`: true in the last block, which
// publishes the step.
__device__ __noinline__ bool last_block(StepCtl *ctl, int step, int n_steps)
{
    const bool fin = step + 1 == n_steps;
    bool last = count_block(ctl, fin);
    if (last && n_steps > 1 && fin) last = !was_abandoned(ctl);
    return last;
}

// A block whose wait for the others ran out leaves a launch of several steps;
// one thread.  The others see it at their next wait and leave too (this
// block's tiles are missing), and the last to come by, here or at the end of
// the last step, clears the control block.
__device__ __noinline__ void abandon_launch(StepCtl *ctl)
{
    atomicExch(&ctl->abandoned, 1u);
    if (count_block(ctl, true)) clear_ctl(ctl);
}

// The last block's end of a step, one thread: the next launch reads the control
// block after this one has ended, the next step of this one once it has
// acquired the epoch.
__device__ __forceinline__ void end_step(StepCtl *ctl, unsigned epoch, bool fin)
{
    *(volatile unsigned *)&ctl->ticket = 0u;
    *(volatile unsigned *)&ctl->done[fin] = 0u;
    if (!fin)
        st_release(&ctl->epoch, epoch + 1u);
    else
        *(volatile unsigned *)&ctl->epoch = epoch + 1u;
}

// One thread waits until the launch's epoch has left `epoch` (bounded; false
// and the status on a time-out, false when another block gave the launch up).
__device__ __forceinline__ bool await_epoch(const StepCtl *ctl, unsigned epoch, unsigned limit,
                                            int *status)
{
    unsigned spins = 0;
    while (ld_acquire(&ctl->epoch) == epoch) {
        if (++spins % 256u == 0u && *(const volatile unsigned *)&ctl->abandoned) return false;
        if (spins > limit) {
            raise_status(status, QP_ERR_TIMEOUT);
            return false;
        }
        __nanosleep(64);
    }
    return true;
}

// One thread waits for the launch's next step; false if it was given up.  (This
// and last_block are called: their values would take registers from the tile
// loops, 4.2e6-slot steps 1 % longer.)
__device__ __noinline__ bool next_step(StepCtl *ctl, unsigned epoch, unsigned limit, int *status)
{
    const bool go = await_epoch(ctl, epoch, limit, status);
    if (!go) abandon_launch(ctl);
    return go;
}

// The first ticket of a block of a cooperative launch of several steps: 0 ..
// grid - 1, those of the blocks that came first on their SM before those that
// came second, and so on.  Blocks that follow one another share an SM, and so
// did the few tiles of a small step, whose warps then queue for one SM's pipes.
// Us for 20 steps of a plane wave, block b taking tile b / this:
//   FP64   4096 electrons 1124 / 761, 8000 1131 / 821, 20000 1135 / 970, a
//          cascade of 16384 with diagnostics 1554 / 1441;
//   mixed  4096 458 / 424, 8000 556 / 472, 20000 and 40000 photons 570 / 510.
// One thread a block; every block is resident, so the wait for all of them ends.
// It is bounded: a block whose wait runs out abandons the launch and takes no
// tile in it.  It costs some 2 us, so a launch of one step does without.
__device__ __noinline__ long long spread_ticket(StepCtl *ctl, unsigned limit, int *status)
{
    unsigned sm;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(sm));
    const unsigned seen = atomicAdd(&ctl->sm_blocks[sm % kSpreadSms], 1u);
    const unsigned rank = seen < kSpreadRanks ? seen : kSpreadRanks - 1;
    long long t = atom_add_acq_rel(&ctl->rank_blocks[rank], 1u);
    atom_add_acq_rel(&ctl->arrived, 1u);
    unsigned spins = 0;
    while (ld_acquire(&ctl->arrived) < gridDim.x) {
        if (++spins > limit) {
            raise_status(status, QP_ERR_TIMEOUT);
            atomicExch(&ctl->abandoned, 1u);
            return 1ll << 62;
        }
        __nanosleep(32);
    }
    for (unsigned q = 0; q < rank; ++q) t += __ldcg(&ctl->rank_blocks[q]);
    return t;
}

// Decoupled look-back over a chain of tiles.  A tile first publishes its
// aggregate (the number of particles it appends); the exclusive prefix is
// then computed by one full warp with a 32-tile window: lane l inspects tile
// base - l; a word counts only if it carries this step's epoch.  The
// window is consumed up to the nearest tile that published its inclusive
// prefix, summing the aggregates in between.  Waits are bounded by
// spin_limit; on time-out the status is raised and the prefix is what was
// summed so far (the output is then wrong, the status says so, and the
// kernel still terminates).  Returns the prefix in every lane.

// Publish a tile's aggregate (tile 0: its inclusive prefix); one thread.
__device__ __forceinline__ void publish_aggregate(unsigned long long *words, unsigned tile,
                                                  long long aggregate, unsigned epoch)
{
    atomicExch(words + tile, make_word(epoch, tile == 0 ? kFlagPre : kFlagAgg, aggregate));
}

// The exclusive prefix of a tile whose aggregate is published: one full
// warp; publishes the tile's inclusive prefix.
__device__ long long resolve_prefix(unsigned long long *words, unsigned tile, long long aggregate,
                                    unsigned epoch, unsigned spin_limit, int *status)
{
    const int lane = threadIdx.x & 31;
    if (tile == 0) return 0;
    long long excl = 0;
    long long base = (long long)tile - 1;
    unsigned spins = 0, nap = 32;
    for (;;) {
        const long long idx = base - lane;
        // before tile 0 the chain is complete: read as "prefix 0"
        const unsigned long long w =
            idx >= 0 ? ld_volatile(words + idx) : make_word(epoch, kFlagPre, 0);
        const bool current = (unsigned)(w >> kEpochShift) == (epoch & kEpochMask);
        const unsigned flag = current ? (unsigned)(w >> kFlagShift) & 3u : 0u;
        const unsigned pre = __ballot_sync(0xFFFFFFFFu, flag == kFlagPre);
        const unsigned empty = __ballot_sync(0xFFFFFFFFu, flag == 0u);
        const int first = pre ? __ffs(pre) - 1 : 32;  // nearest inclusive prefix
        const unsigned need = first == 32 ? 0xFFFFFFFFu : (2u << first) - 1u;
        if (empty & need) {
            if (++spins > spin_limit) {
                if (lane == 0) raise_status(status, QP_ERR_TIMEOUT);
                break;
            }
            // back off (32 ns doubling to 256 ns): a waiting warp takes few
            // issue slots from the warps still computing their tiles, and
            // wakes soon after the tile it waits on publishes (a 1 us cap:
            // foil 30.5 us per step, 256 ns: 30.1)
            __nanosleep(nap);
            if (nap < 256) nap <<= 1;
            continue;
        }
        long long v = lane <= first ? (long long)(w & kValMask) : 0;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, d);
        excl += v;
        if (first < 32) break;
        base -= 32;
    }
    if (lane == 0) atomicExch(words + tile, make_word(epoch, kFlagPre, excl + aggregate));
    return excl;
}

__device__ long long chain_prefix(unsigned long long *words, unsigned tile, long long aggregate,
                                  unsigned epoch, unsigned spin_limit, int *status)
{
    if ((threadIdx.x & 31) == 0) publish_aggregate(words, tile, aggregate, epoch);
    __syncwarp();
    return resolve_prefix(words, tile, aggregate, epoch, spin_limit, status);
}

// Counters kept in shared memory per block and species, flushed with one
// atomic per counter when the block leaves.  The counts are 32-bit (shared
// memory adds them natively; a block never counts 2^32 events in a launch),
// summed over a warp before one lane adds them.
struct BlockStats {
    unsigned c[3][9];
    double e[3][2];
};
enum { cEmit, cPhoton, cPhotonDrop, cSub, cPair, cPairDrop, cSat, cClamp, cCont };

__device__ __forceinline__ void warp_count(unsigned *ctr, bool pred)
{
    const unsigned m = __ballot_sync(0xFFFFFFFFu, pred);
    if ((threadIdx.x & 31) == 0 && m) atomicAdd(ctr, (unsigned)__popc(m));
}

// Sum of v over the (converged) warp, added by one lane.
__device__ __forceinline__ void warp_add(unsigned *ctr, unsigned v)
{
    const unsigned s = __reduce_add_sync(0xFFFFFFFFu, v);
    if ((threadIdx.x & 31) == 0 && s) atomicAdd(ctr, s);
}

__device__ __forceinline__ void warp_add(double *ctr, double v)
{
    if (!__any_sync(0xFFFFFFFFu, v != 0.0)) return;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, d);
    if ((threadIdx.x & 31) == 0) atomicAdd(ctr, v);
}

__device__ __forceinline__ void clear_stats(BlockStats &bs)
{
    const int t = threadIdx.x;
    if (t < 27) (&bs.c[0][0])[t] = 0u;
    if (t < 6) (&bs.e[0][0])[t] = 0.0;
}

__device__ void flush_stats(const BlockStats &bs, const StepArgs &a, const Problem &P)
{
    __syncthreads();
    const int t = threadIdx.x;
    if (t < 27) {
        const int s = t / 9, k = t % 9;
        if (bs.c[s][k] && P.sp[s].present)
            atomicAdd(&a.stats[P.sp[s].slot_stats].n_emit + k, (unsigned long long)bs.c[s][k]);
    } else if (t >= 32 && t < 38) {
        const int s = (t - 32) / 2, k = (t - 32) % 2;
        if (bs.e[s][k] != 0.0 && P.sp[s].present)
            atomicAdd(&a.stats[P.sp[s].slot_stats].e_subthreshold + k, bs.e[s][k]);
    }
    if (t == 0 && (bs.c[0][cClamp] | bs.c[1][cClamp] | bs.c[2][cClamp]))
        raise_status(a.status, QP_WARN_TABLE_CLAMPED);
}

// Append records of a tile (short tiles) or of a warp's part of one (long
// parts), [field][record], in device memory; written with the events, read
// when the slots are known.  Leptons, one record an emitter in slot order:
// x, y, z, direction kx, ky, kz, weight, its slot, what its photons are (their
// number, and 4 bits each for the emission that made it) and the energies of
// up to QP_MAX_EMISSIONS of them; their optical depths are drawn when they are
// written.  Photons, one record a decayed photon: chi and the slot; the rest
// is still in its slot.
constexpr int kStashSlot = 7, kStashWhat = 8, kStashGg = 9;
static_assert(kStashGg + QP_MAX_EMISSIONS == kStashFieldsHost, "stash layout");
static_assert(QP_MAX_EMISSIONS <= 8, "emission indices and the count take 4 bits each");

// The optical depth of the photon of a lepton's emission k in this step.
template <int PREC>
__device__ __forceinline__ double photon_depth(const Problem &P, const StepTime &tm, int sp,
                                               int64_t i, int k)
{
    const uint4 r = draw(P.seed, sp, kRngPhotonTau, particle_id(P.sp[sp], i), tm.step, k);
    if constexpr (PREC == kFP64)
        return -log(u53(r.x, r.y));
    else
        return finite_to_d(-logf(u53f(r.x, r.y)));
}

// Entries of a warp's queue of emitters: long parts, fewer than 32 wait while
// a sub-tile adds up to 32; short tiles, two halves of 32 for two tiles.
constexpr int kQueue = 64;

// What a lepton carries out of its push: momentum after it (mixed path: the
// FP32 increment of the FP64 momentum), gamma, chi_e, W dt and the fields; a lepton
// without an event needs no fields any more: E holds delta v, chi the
// decrement of its optical depth (FP64: the new one), gam 1/gamma in FP64 and B
// the FP32 momentum.
template <typename R>
struct LeptonMid {
    R ux, uy, uz, gam, chi, wdt;
    Vec3<R> E, B;
};

// The same queued in shared memory, [field][entry]: a wave along x polarised
// in y has one independent field component, a constant B none.
template <int FK>
constexpr int mid_words()
{
    return FK == QP_FIELD_YEE2D ? 12 : (FK == QP_FIELD_PLANE || FK == QP_FIELD_GAUSSIAN) ? 7 : 6;
}

template <int FK, typename R>
__device__ __forceinline__ void mid_put(R (*w)[kQueue], int t, const LeptonMid<R> &m)
{
    w[0][t] = m.ux;
    w[1][t] = m.uy;
    w[2][t] = m.uz;
    w[3][t] = m.gam;
    w[4][t] = m.chi;
    w[5][t] = m.wdt;
    if constexpr (FK == QP_FIELD_PLANE || FK == QP_FIELD_GAUSSIAN) w[6][t] = m.E.y;
    if constexpr (FK == QP_FIELD_YEE2D) {
        w[6][t] = m.E.x;
        w[7][t] = m.E.y;
        w[8][t] = m.E.z;
        w[9][t] = m.B.x;
        w[10][t] = m.B.y;
        w[11][t] = m.B.z;
    }
}

template <int FK, typename R>
__device__ __forceinline__ void mid_get(const R (*w)[kQueue], int t, R b0, LeptonMid<R> &m)
{
    m.ux = w[0][t];
    m.uy = w[1][t];
    m.uz = w[2][t];
    m.gam = w[3][t];
    m.chi = w[4][t];
    m.wdt = w[5][t];
    m.E = {R(0), R(0), R(0)};
    m.B = {R(0), R(0), R(0)};
    if constexpr (FK == QP_FIELD_PLANE || FK == QP_FIELD_GAUSSIAN) m.E.y = m.B.z = w[6][t];
    if constexpr (FK == QP_FIELD_UNIFORM_B) m.B.z = b0;
    if constexpr (FK == QP_FIELD_YEE2D) {
        m.E = {w[6][t], w[7][t], w[8][t]};
        m.B = {w[9][t], w[10][t], w[11][t]};
    }
}

// Short tiles of the mixed path on a 2D grid run their emitters in place: a
// lepton there carries six field components to them, and a push whose gather
// keeps 24 loads in flight has no registers for it (2D foil: 36 us a step in
// place, 38.5 packed).  The kernels of 2D grids have no long tiles either
// (has_long_tiles): the call alone costs them registers (39.5 us).
template <int FK, typename R>
constexpr bool kEmitInPlace = sizeof(R) == 4 && FK == QP_FIELD_YEE2D;

// Shared-memory layout of k_step (dynamic part).  Where emitters run in place
// nothing is queued: the 12 KB a block are left to the L1 cache, which serves
// the gather.
template <int FK, typename R>
struct Smem {
    static constexpr bool kQueued = !kEmitInPlace<FK, R>;
    R H[kNRatePad];                          // rate tables (TMA-staged)
    R G[kNRatePad];
    R T[kNRatePad];
    // each warp's emitters
    R mid[kQueued ? kWarps : 1][kQueued ? mid_words<FK>() : 1][kQueue];
};

__device__ __forceinline__ void wait_tables(unsigned long long *bar, const StepArgs &a)
{
    if (!mbar_wait_bounded(bar, 0, a.spin_limit)) {
        // the step's results are flagged invalid from here on; a second
        // bounded wait gives the copy more time to land before the block
        // reads the tables or leaves.  If it runs out too, the tile reads
        // tables that may be incomplete (the raised status says so) and the
        // kernel still terminates.
        raise_status(a.status, QP_ERR_TIMEOUT);
        (void)mbar_wait_bounded(bar, 0, a.spin_limit);
    }
}

// -------------------------------------------------------------------- lepton tile

// Issue the copy of the rate tables H and G into shared memory (one TMA
// bulk copy each, completing on `bar`); one thread, before a barrier that
// makes the barrier's initialisation visible to the block.
template <int PREC, int FK, typename R>
__device__ __forceinline__ void stage_rate_tables(const StepArgs &a, Smem<FK, R> &sm,
                                                  unsigned long long *bar)
{
    const unsigned bytes = kNRatePad * sizeof(R);
    mbar_init(bar, 1);
    mbar_expect_tx(bar, 2 * bytes);
    if constexpr (PREC == kFP64) {
        bulk_g2s(sm.H, a.tab.H, bytes, bar);
        bulk_g2s(sm.G, a.tab.Gs, bytes, bar);
    } else {
        bulk_g2s(sm.H, a.tab.Hf, bytes, bar);
        bulk_g2s(sm.G, a.tab.Gsf, bytes, bar);
    }
}

// The same for the pair rate T.
template <int PREC, int FK, typename R>
__device__ __forceinline__ void stage_pair_table(const StepArgs &a, Smem<FK, R> &sm,
                                                 unsigned long long *bar)
{
    const unsigned bytes = kNRatePad * sizeof(R);
    mbar_init(bar, 1);
    mbar_expect_tx(bar, bytes);
    if constexpr (PREC == kFP64)
        bulk_g2s(sm.T, a.tab.Ts, bytes, bar);
    else
        bulk_g2s(sm.T, a.tab.Tsf, bytes, bar);
}

// State of one lepton at the start of a step (the FP64 storage of both
// paths; component c of the new state goes to the sink's put<c> as soon as
// it is formed, c = x y z ux uy uz tau, tau only when it changed).
struct LeptonState {
    double x, y, z, ux, uy, uz, tau;
};

// What one lepton's step produced besides its new state.
struct LeptonOut {
    int n_emit, nph, n_sub;
    double e_sub;   // sum of gamma_gamma of the photons below the cut
    bool cont, sat, clamped;
};

// One step of one lepton (a1..a8 of the hot path) in three parts.
//   lepton_push: fields at (x, t), Boris push, chi_e, then Sokolov damping
//     below chi_th or the first optical-depth decision (Eq. 6); true if the
//     lepton has an event;
//   lepton_finish: the position (Eq. 4) of a lepton without one;
//   lepton_events: of one with an event, the emission sub-loop from its first
//     emission on (Eq. 6-8), then the position.
// A few leptons of a warp emit in a step, so the step kernel queues them and
// runs the second part on 32 at a time; inside the first part every warp paid
// a round of it for its three or four emitters.
// The sink receives the new state (put<c>, see LeptonState) and what an
// append needs: tables() before the rate tables H and G are first read,
// chi(c) with chi_e after the push, direction(k) with the momentum direction
// before the first recoil, photon(j, gamma, k) for the j-th stored photon, of
// emission k (its optical depth: photon_depth),
// origin(x) with the position at the start of the step when photons were
// stored.  S, i: the particle's species and slot (its id keys the random
// streams).
template <int PREC, int FK, typename R, class Sink>
__device__ __forceinline__ bool lepton_push(const StepArgs &a, const Problem &P,
                                            const StepTime &tm, const R *H, const R *G, int sp, const LeptonState &s,
                                            LeptonMid<R> &mid, LeptonOut &o, Sink &sink)
{
    o.n_emit = o.nph = o.n_sub = 0;
    o.e_sub = 0.0;
    o.cont = o.sat = o.clamped = false;
    bool clamped = false;
    if constexpr (PREC == kFP64) {
        const double q = sp == 0 ? -1.0 : 1.0;
        const double dt = P.dt;
        const double x0 = s.x, y0 = s.y, z0 = s.z;
        double ux = s.ux, uy = s.uy, uz = s.uz;
        double tau = s.tau;
        Vec3<R> E, B;
        eval_field<FK>(P.f, x0, y0, z0, tm.t, E, B);

        // ---- Boris push of the Lorentz force (f_l of Eq. 4)
        {
            const double h = 0.5 * q * dt;
            const double mx = ux + h * E.x, my = uy + h * E.y, mz = uz + h * E.z;
            const double hig = h * rsqrt64(1.0 + mx * mx + my * my + mz * mz);
            const double tx = hig * B.x, ty = hig * B.y, tz = hig * B.z;
            const double k2 = 2.0 * rcp64(1.0 + tx * tx + ty * ty + tz * tz);
            const double sx = k2 * tx, sy = k2 * ty, sz = k2 * tz;
            const double px = mx + (my * tz - mz * ty), py = my + (mz * tx - mx * tz),
                         pz = mz + (mx * ty - my * tx);
            ux = mx + (py * sz - pz * sy) + h * E.x;
            uy = my + (pz * sx - px * sz) + h * E.y;
            uz = mz + (px * sy - py * sx) + h * E.z;
        }
        double g2 = 1.0 + ux * ux + uy * uy + uz * uz;
        double ig = rsqrt64(g2);
        const double gam = root_of(g2, ig);
        const double Ex = E.x, Ey = E.y, Ez = E.z, Bx = B.x, By = B.y, Bz = B.z;
        sink.tables();  // tables are needed from here on
        const double chi = chi_e64(Ex, Ey, Ez, Bx, By, Bz, ux, uy, uz, gam, a.inv_aS);
        sink.chi(chi);
        double dvx = 0.0, dvy = 0.0, dvz = 0.0;

        if (chi < P.chi_th) {
            // ---- Sokolov continuous regime (Eq. 4, P_rad of Eq. 5)
            o.cont = true;
            const double vx = ux * ig, vy = uy * ig, vz = uz * ig;
            const double fx = q * (Ex + (vy * Bz - vz * By));
            const double fy = q * (Ey + (vz * Bx - vx * Bz));
            const double fz = q * (Ez + (vx * By - vy * Bx));
            const double vf = vx * fx + vy * fy + vz * fz;
            const double k = a.tau0w * rcp64(1.0 + a.tau0w * vf);
            dvx = k * (fx - vx * vf);
            dvy = k * (fy - vy * vf);
            dvz = k * (fz - vz * vf);
            const double prad = a.C_rate * rate64<1>(G, chi, clamped);
            ux = ux + dt * (q * (dvy * Bz - dvz * By) - prad * vx);
            uy = uy + dt * (q * (dvz * Bx - dvx * Bz) - prad * vy);
            uz = uz + dt * (q * (dvx * By - dvy * Bx) - prad * vz);
            ig = rsqrt64(1.0 + ux * ux + uy * uy + uz * uz);
        } else {
            // ---- optical depth (Eq. 6)
            const double Hv = rate64<0>(H, chi, clamped);
            const double dtau = a.C_rate * Hv * ig * dt;
            if (dtau > 0.0 && !(tau > dtau)) {
                o.clamped = clamped;
                mid = {ux, uy, uz, gam, chi, dtau, E, B};
                return true;
            }
            tau = tau - dtau;
        }
        o.clamped = clamped;
        mid = {ux, uy, uz, ig, tau, 0.0, {dvx, dvy, dvz}, {0.0, 0.0, 0.0}};
    } else {
        // ---- mixed precision: FP32 physics; the FP64 state is read once,
        // increments are formed in FP32 and added back by integer
        // instructions; chi_e falls back to double-float where FP32 cancels
        const MixedConsts &m = P.mc;
        const double xd = s.x, yd = s.y, zd = s.z;
        const double uxd = s.ux, uyd = s.uy, uzd = s.uz;
        const double taud = s.tau;
        Vec3<float> E, B;
        eval_field_mixed<FK>(P.f, m, tm, xd, yd, zd, E, B);

        // Boris on the leading FP32 parts; the increment is kept in FP32
        const float u0x = hi_d(uxd), u0y = hi_d(uyd), u0z = hi_d(uzd);
        const float h = m.h[sp];
        const float hx = h * E.x, hy = h * E.y, hz = h * E.z;
        const float mx = u0x + hx, my = u0y + hy, mz = u0z + hz;
        const float ig = rsqrtf(1.0f + mx * mx + my * my + mz * mz);
        const float tx = h * B.x * ig, ty = h * B.y * ig, tz = h * B.z * ig;
        const float k2 = 2.0f / (1.0f + tx * tx + ty * ty + tz * tz);
        const float sx = k2 * tx, sy = k2 * ty, sz = k2 * tz;
        const float px = mx + (my * tz - mz * ty), py = my + (mz * tx - mx * tz),
                    pz = mz + (mx * ty - my * tx);
        float dux = (py * sz - pz * sy) + 2.0f * hx, duy = (pz * sx - px * sz) + 2.0f * hy,
              duz = (px * sy - py * sx) + 2.0f * hz;
        float ux = u0x + dux, uy = u0y + duy, uz = u0z + duz;
        float gam = sqrtf(1.0f + ux * ux + uy * uy + uz * uz);
        sink.tables();  // tables are needed from here on
        const float chi = chi_mixed_auto(uxd, uyd, uzd, dux, duy, duz, ux, uy, uz, gam, E, B,
                                         m.inv_aS, m.inv_aS_lo);
        sink.chi(finite_to_d(chi));
        float dvx = 0.0f, dvy = 0.0f, dvz = 0.0f;
        float dtau = 0.0f;

        if (chi < m.chi_th) {
            // ---- Sokolov (Eq. 4, 5); denominator 1 + tau0 v.f_l in double-float
            o.cont = true;
            const float q = sp == 0 ? -1.0f : 1.0f;
            const float gi = 1.0f / gam;
            const float vx = ux * gi, vy = uy * gi, vz = uz * gi;
            const float fx = q * (E.x + (vy * B.z - vz * B.y));
            const float fy = q * (E.y + (vz * B.x - vx * B.z));
            const float fz = q * (E.z + (vx * B.y - vy * B.x));
            const float vf = vx * fx + vy * fy + vz * fz;
            const df2 den = two_sum(1.0f, m.tau0w * vf);
            const float c = m.tau0w / den.hi * (1.0f - den.lo / den.hi);
            dvx = c * (fx - vx * vf);
            dvy = c * (fy - vy * vf);
            dvz = c * (fz - vz * vf);
            const float prad = m.C_rate * rate32<1>(G, chi, clamped);
            const float sx_ = m.dt * (q * (dvy * B.z - dvz * B.y) - prad * vx);
            const float sy_ = m.dt * (q * (dvz * B.x - dvx * B.z) - prad * vy);
            const float sz_ = m.dt * (q * (dvx * B.y - dvy * B.x) - prad * vz);
            dux += sx_;
            duy += sy_;
            duz += sz_;
            ux += sx_;
            uy += sy_;
            uz += sz_;
            gam = sqrtf(1.0f + ux * ux + uy * uy + uz * uz);
        } else {
            // ---- optical depth (Eq. 6); tau > dtau decided on the
            // double-float optical depth
            const df2 TAU = split_d(taud);
            const float Hv = rate32<0>(H, chi, clamped);
            const float wdt = m.C_rate * Hv / gam * m.dt;
            dtau = wdt;
            if (dtau > 0.0f && !(TAU.hi > dtau || (TAU.hi == dtau && TAU.lo > 0.0f))) {
                o.clamped = clamped;
                mid = {dux, duy, duz, gam, chi, wdt, E, B};
                return true;
            }
        }
        o.clamped = clamped;
        mid = {dux, duy, duz, gam, dtau, 0.0f, {dvx, dvy, dvz}, {ux, uy, uz}};
    }
    return false;
}

// The position (Eq. 4: dx/dt = v + delta v) and the new state of a lepton whose
// push had no event.
template <int PREC, typename R, class Sink>
__device__ __forceinline__ void lepton_finish(const Problem &P, const LeptonState &s,
                                              const LeptonMid<R> &mid, Sink &sink)
{
    const Vec3<R> &dv = mid.E;
    if constexpr (PREC == kFP64) {
        sink.template put<0>(s.x + P.dt * (mid.ux * mid.gam + dv.x));
        sink.template put<1>(s.y + P.dt * (mid.uy * mid.gam + dv.y));
        if (sink.has_z()) sink.template put<2>(s.z + P.dt * (mid.uz * mid.gam + dv.z));
        sink.template put<3>(mid.ux);
        sink.template put<4>(mid.uy);
        sink.template put<5>(mid.uz);
        sink.template put<6>(mid.chi);
    } else {
        // FP64 accumulation of FP32 increments
        const float gi = 1.0f / mid.gam, dt = P.mc.dt;
        const Vec3<float> &u = mid.B;
        sink.template put<0>(add_fd(s.x, dt * (u.x * gi + dv.x)));
        sink.template put<1>(add_fd(s.y, dt * (u.y * gi + dv.y)));
        if (sink.has_z()) sink.template put<2>(add_fd(s.z, dt * (u.z * gi + dv.z)));
        sink.template put<3>(add_fd(s.ux, mid.ux));
        sink.template put<4>(add_fd(s.uy, mid.uy));
        // a wave polarised in y leaves the momentum along z alone
        if (mid.uz != 0.0f) sink.template put<5>(add_fd(s.uz, mid.uz));
        if (mid.chi != 0.0f) sink.template put<6>(add_fd(s.tau, -mid.chi));
    }
}

// Nodes of a CDF row that a sample loads at once (mixed path): on a 2D grid the
// gather's values leave registers for fewer.
template <int FK>
constexpr int kWindowNodes = FK == QP_FIELD_YEE2D ? 3 : 4;

template <int PREC, int FK, typename R, class Sink>
__device__ __forceinline__ void lepton_events(const StepArgs &a, const Problem &P,
                                              const StepTime &tm, const R *H, int sp, const SpeciesDev &S, int64_t i,
                                              const LeptonState &s, const LeptonMid<R> &mid,
                                              LeptonOut &o, Sink &sink)
{
    bool clamped = false, sat = false;
    int nph = 0, n_emit = 0, n_sub = 0;
    const Vec3<R> &E = mid.E, &B = mid.B;
    if constexpr (PREC == kFP64) {
        const double dt = P.dt;
        double ux = mid.ux, uy = mid.uy, uz = mid.uz, gam = mid.gam, chi = mid.chi;
        double tau = s.tau, e_sub = 0.0;
        double r = 1.0, wdt = mid.wdt, ig = 0.0;
        for (int k = 0;;) {
            r = r - tau * rcp64(wdt);
            // ---- emission: Eq. 7 sampling, Eq. 8 recoil
            const uint4 rr = draw(P.seed, sp, kRngEmit, particle_id(S, i), tm.step, k);
            const double xi_p = u53(rr.x, rr.y), xi = u53(rr.z, rr.w);
            const double ufrac = sample_cdf(a.tab.Cg, a.tab.Gg, chi, xi_p, kSgMin, kSgSpan,
                                                    true, clamped);
            const double p2 = ux * ux + uy * uy + uz * uz;
            const double ip = p2 > 0.0 ? rsqrt64(p2) : 0.0, pmag = root_of(p2, ip);
            double gg = ufrac * gam;
            if (gg > pmag) gg = pmag;
            if (n_emit == 0 && pmag > 0.0) sink.direction(ux * ip, uy * ip, uz * ip);
            ++n_emit;
            if (gg > P.gmin) {
                sink.photon(nph, gg, k);
                ++nph;
            } else {
                ++n_sub;
                e_sub += gg;
            }
            if (pmag > 0.0) {
                const double scale = (pmag - gg) * ip;
                ux *= scale;
                uy *= scale;
                uz *= scale;
            }
            tau = -log(xi);
            const double g2 = 1.0 + ux * ux + uy * uy + uz * uz;
            ig = rsqrt64(g2);
            gam = root_of(g2, ig);
            chi = chi_e64(E.x, E.y, E.z, B.x, B.y, B.z, ux, uy, uz, gam, a.inv_aS);
            // ---- the rest of the step (Eq. 6)
            const double Hv = rate64<0>(H, chi, clamped);
            wdt = a.C_rate * Hv * ig * dt;
            const double dtau = wdt * r;
            const bool more = dtau > 0.0 && !(tau > dtau);
            sat = more && ++k == P.max_emit;
            if (!more || sat) {
                tau = tau - dtau;
                break;
            }
        }
        // ---- position (Eq. 4)
        if (nph) sink.origin(s.x, s.y, s.z);
        sink.template put<0>(s.x + dt * (ux * ig));
        sink.template put<1>(s.y + dt * (uy * ig));
        if (sink.has_z()) sink.template put<2>(s.z + dt * (uz * ig));
        sink.template put<3>(ux);
        sink.template put<4>(uy);
        sink.template put<5>(uz);
        sink.template put<6>(tau);
        o.e_sub = e_sub;
    } else {
        const MixedConsts &m = P.mc;
        float dux = mid.ux, duy = mid.uy, duz = mid.uz, gam = mid.gam, chi = mid.chi;
        float ux = hi_d(s.ux) + dux, uy = hi_d(s.uy) + duy, uz = hi_d(s.uz) + duz;
        df2 TAU = split_d(s.tau);
        float r = 1.0f, esub_f = 0.0f, wdt = mid.wdt;
        for (int k = 0;;) {
            r = r - df_to_f(TAU) / wdt;
            // ---- emission: Eq. 7 sampling, Eq. 8 recoil
            const uint4 rr = draw(P.seed, sp, kRngEmit, particle_id(S, i), tm.step, k);
            const float xi = u53f(rr.z, rr.w);
            const FracPair uf = sample_cdf_f<kWindowNodes<FK>>(
                a.tab.Cg2, a.tab.Qg2, a.tab.Gg, a.tab.Eg, chi, u53_pair(rr.x, rr.y),
                u53_pair_complement(rr.x, rr.y), (float)(kSgSpan / (kNNode - 1)), true, clamped);
            const float pmag = sqrtf(ux * ux + uy * uy + uz * uz);
            float gg = uf.x * gam;
            // what the electron keeps, |p| - u gamma = (1-u) gamma - 1/(gamma + |p|),
            // formed without cancellation
            float keep = uf.omx * gam - 1.0f / (gam + pmag);
            if (gg > pmag || keep < 0.0f) {
                gg = pmag;
                keep = 0.0f;
            }
            if (n_emit == 0) {
                // the photons' direction goes to the append record now
                // (fewer values live through the loop)
                const float ip = pmag > 0.0f ? 1.0f / pmag : 0.0f;
                sink.direction(finite_to_d(ux * ip), finite_to_d(uy * ip), finite_to_d(uz * ip));
            }
            ++n_emit;
            if (gg > m.gmin) {
                sink.photon(nph, finite_to_d(gg), k);
                ++nph;
            } else {
                ++n_sub;
                esub_f += gg;
            }
            if (pmag > 0.0f) {
                const float s1 = keep / pmag;
                const float s1m = s1 - 1.0f;  // exact (Sterbenz) for s1 in [1/2, 1]
                dux = fmaf(ux, s1m, dux);
                duy = fmaf(uy, s1m, duy);
                duz = fmaf(uz, s1m, duz);
                ux *= s1;
                uy *= s1;
                uz *= s1;
            }
            TAU = {-logf(xi), 0.0f};
            gam = sqrtf(1.0f + ux * ux + uy * uy + uz * uz);
            chi = chi_mixed_auto(s.ux, s.uy, s.uz, dux, duy, duz, ux, uy, uz, gam, E, B, m.inv_aS,
                                 m.inv_aS_lo);
            // ---- the rest of the step (Eq. 6); tau > dtau decided on the
            // double-float optical depth
            const float Hv = rate32<0>(H, chi, clamped);
            wdt = m.C_rate * Hv / gam * m.dt;
            const float dtau = wdt * r;
            const bool more = dtau > 0.0f && !(TAU.hi > dtau || (TAU.hi == dtau && TAU.lo > 0.0f));
            sat = more && ++k == P.max_emit;
            if (!more || sat) {
                TAU = df_add_f(TAU, -dtau);
                break;
            }
        }
        // ---- position and state: FP64 accumulation of FP32 increments
        if (nph) sink.origin(s.x, s.y, s.z);
        const float gi = 1.0f / gam;
        sink.template put<0>(add_fd(s.x, m.dt * (ux * gi)));
        sink.template put<1>(add_fd(s.y, m.dt * (uy * gi)));
        if (sink.has_z()) sink.template put<2>(add_fd(s.z, m.dt * (uz * gi)));
        sink.template put<3>(add_fd(s.ux, dux));
        sink.template put<4>(add_fd(s.uy, duy));
        if (duz != 0.0f) sink.template put<5>(add_fd(s.uz, duz));
        sink.template put<6>(merge_df(TAU));
        if (n_sub) o.e_sub = finite_to_d(esub_f);
    }
    o.n_emit = n_emit;
    o.nph = nph;
    o.n_sub = n_sub;
    o.sat = sat;
    // a step above the table's range is counted once, with the push if it was
    // there already
    if (clamped && !(mid.chi >= (R)kChiHi)) o.clamped = true;
}

// The append sink of a step tile: new state to the particle's slot, append
// records to the warp's stash.
struct StashSink {
    const StepArgs &a;
    unsigned long long *bar;  // the rate tables' copy, NULL once it has landed
    double *st;
    int cap;           // records of each field
    int e;             // the emitter's number in its warp's part
    double *chi_slot;  // the particle's chi, or NULL
    const SpeciesDev &S;
    int64_t i;
    unsigned long long what;  // emission indices of the stored photons
    // each component is stored as soon as it is formed (a value kept across
    // the called write-back helpers would have to be saved and restored)
    template <int C>
    __device__ __forceinline__ void put(double v)
    {
        if constexpr (C == 0) S.x[i] = v;
        if constexpr (C == 1) S.y[i] = v;
        if constexpr (C == 2) S.z[i] = v;
        if constexpr (C == 3) S.ux[i] = v;
        if constexpr (C == 4) S.uy[i] = v;
        if constexpr (C == 5) S.uz[i] = v;
        if constexpr (C == 6) S.tau[i] = v;
    }
    __device__ __forceinline__ bool has_z() const { return S.z != nullptr; }
    __device__ __forceinline__ void tables()
    {
        if (bar) wait_tables(bar, a);
    }
    __device__ __forceinline__ void chi(double c)
    {
        if (chi_slot) *chi_slot = c;
    }
    __device__ __forceinline__ void direction(double kx, double ky, double kz)
    {
        st[3 * cap + e] = kx;
        st[4 * cap + e] = ky;
        st[5 * cap + e] = kz;
    }
    __device__ __forceinline__ void photon(int j, double gg, int k)
    {
        st[(kStashGg + j) * cap + e] = gg;
        what |= (unsigned long long)k << (4 + 4 * j);
    }
    __device__ __forceinline__ void origin(double x, double y, double z)
    {
        st[0 * cap + e] = x;
        st[1 * cap + e] = y;
        st[2 * cap + e] = z;
    }
};

// -------------------------------------------------------------------- a block's tiles
//
// Emission loops and pair samplings are long and rare: 3 to 15 % of the slots
// of a step, so in place a warp pays a round of them for its two to four
// lanes that need one (16 of 32 lanes active over the 4.2e6-lepton collision
// step, 498 M warp instructions).  Both kinds of tile run them on packed
// lanes; which one a launch takes follows from the slots it steps
// (long_tiles), and the results are the same: slots are assigned in slot
// order.
//   Short tiles (128 slots, a sub-tile of 32 a warp, one barrier a tile):
//     tile q      physics of every slot; slots with an event are listed;
//     tile q - 1  its emitters, 32 at a time in whichever warps are free; the
//                 last chunk publishes the tile's aggregate (photon tiles
//                 publish theirs with their physics: a decay is one pair);
//     tile q - 3  its prefix is resolved and its particles are written, by
//                 the first warp to come there.
//   Long tiles (256 slots a warp, no barrier): each warp goes over its part,
//     queueing emitters and running 32 of them together, and counts what it
//     appends; the last warp of the tile to do so publishes its aggregate.
//     kLag tiles later the first warp to come there resolves the tile's
//     prefix and every warp writes its own part.  A warp waits for no other
//     warp's emission rounds (short tiles: barrier 6.6 of 17.6 cycles between
//     two issues of a warp), the lanes are fuller, and there are an eighth of
//     the look-backs; but a launch needs some 1024 slots a block and more to
//     keep every warp busy.
// Measured, us a step with short / long tiles: the collision of 4.2e6 leptons
// 660 / 465, its photon-dominated steps 607 / 480.
constexpr int kRing = kStashBufs;  // tiles in flight in a block
constexpr int kLag = 2;            // a long tile is written kLag tiles after its physics
static_assert((kRing & (kRing - 1)) == 0 && kLag < kRing, "ring of tiles");

// Slots of a warp's part of a long tile, slots of the tile.
constexpr int kPart = 32 * kSubTiles, kLongTile = kPart * kWarps;
constexpr int kShortShift = 7, kLongShift = 10;
static_assert((1 << kShortShift) == kTile && (1 << kLongShift) == kLongTile, "tile sizes");
constexpr int kTickets = 2 * kRing;

// The emission loop of the lepton in slot i, its record number e of the stash;
// wgt: its weight.
template <int PREC, int FK, typename R>
__device__ __forceinline__ void run_emitter(const StepArgs &a, const Problem &P,
                                            const StepTime &tm, const R *H, int sp, int64_t i,
                                            const LeptonState &s, const LeptonMid<R> &mid,
                                            double *st, int cap, int e, LeptonOut &o, double &wgt)
{
    const SpeciesDev &S = P.sp[sp];
    StashSink sink{a, nullptr, st, cap, e, nullptr, S, i, 0ull};
    lepton_events<PREC, FK, R>(a, P, tm, H, sp, S, i, s, mid, o, sink);
    wgt = S.w[i];
    double *const r = st + e;
    if (o.nph) {
        r[6 * cap] = wgt;
        r[kStashSlot * cap] = __longlong_as_double((long long)i);
    }
    r[kStashWhat * cap] = __longlong_as_double((long long)(sink.what | (unsigned long long)o.nph));
    if (S.nemit) S.nemit[i] += o.n_emit;
}

// The counters of a warp's emitters; returns the photons they append.
__device__ __forceinline__ int count_emitters(BlockStats &bs, int sp, const LeptonOut &o,
                                              double wgt)
{
    warp_count(&bs.c[sp][cSat], o.sat);
    warp_add(&bs.c[sp][cEmit], (unsigned)o.n_emit);
    warp_add(&bs.c[sp][cSub], (unsigned)o.n_sub);
    warp_add(&bs.e[sp][0], o.n_sub ? wgt * o.e_sub : 0.0);
    return (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned)o.nph);
}

// The emission loops of `ne` listed leptons (at most 32, one warp, lane e of
// it the entry t of the queue `mids`, slot i).  Their records go to the stash
// from number e0 on; returns the photons they append.
template <int PREC, int FK, typename R>
__device__ __forceinline__ int run_emitters(const StepArgs &a, const Problem &P,
                                            const StepTime &tm, const R *H,
                                            const R (*mids)[kQueue], int t, int ne, int sp,
                                            int64_t i, int e0, double *st, int cap,
                                            BlockStats &bs)
{
    const int lane = threadIdx.x & 31;
    const SpeciesDev &S = P.sp[sp];
    LeptonOut o{};
    double wgt = 0.0;
    if (lane < ne) {
        const LeptonState s{S.x[i],  S.y[i],  S.z ? S.z[i] : 0.0, S.ux[i],
                            S.uy[i], S.uz[i], S.tau[i]};
        LeptonMid<R> mid;
        if constexpr (PREC == kFP64)
            mid_get<FK, R>(mids, t, P.f.b0, mid);
        else
            mid_get<FK, R>(mids, t, P.mc.b0, mid);
        run_emitter<PREC, FK, R>(a, P, tm, H, sp, i, s, mid, st, cap, e0 + lane, o, wgt);
    }
    warp_count(&bs.c[sp][cClamp], o.clamped);
    return count_emitters(bs, sp, o, wgt);
}

// One sub-tile of 32 leptons pushed by a warp, lane l the slot i (below n);
// those with an event are queued in slot order from entry `tail` on, with their
// place `at` in the tile or part.  Returns their number.
template <int PREC, int FK, typename R>
__device__ __forceinline__ int push_leptons(const StepArgs &a, const Problem &P,
                                            const StepTime &tm, Smem<FK, R> &sm,
                                            unsigned long long *bar, bool &loaded, int sp,
                                            int64_t i, int64_t n, R (*mids)[kQueue],
                                            unsigned *slots, unsigned tail, unsigned at,
                                            BlockStats &bs)
{
    const SpeciesDev &S = P.sp[sp];
    LeptonOut o{};
    bool event = false;
    LeptonMid<R> mid;
    LeptonState s;
    StashSink sink{a, loaded ? nullptr : bar, nullptr, 0, 0, S.chi ? S.chi + i : nullptr, S, i,
                       0ull};
    if (i < n) {
        s = {S.x[i], S.y[i], S.z ? S.z[i] : 0.0, S.ux[i], S.uy[i], S.uz[i], S.tau[i]};
        event = lepton_push<PREC, FK, R>(a, P, tm, sm.H, sm.G, sp, s, mid, o, sink);
    }
    if (!loaded) {
        // the rate tables' copy was issued in the kernel's prologue
        // (stage_rate_tables); every thread waits once: later tiles read the
        // tables without a wait, and the block never leaves with the copy in
        // flight
        wait_tables(bar, a);
        loaded = true;
    }
    const unsigned m = __ballot_sync(0xFFFFFFFFu, event);
    if (event) {
        const unsigned lt = (1u << (threadIdx.x & 31)) - 1u;
        const unsigned t = (tail + (unsigned)__popc(m & lt)) % (unsigned)kQueue;
        mid_put<FK, R>(mids, (int)t, mid);
        slots[t] = at;
    } else if (i < n) {
        lepton_finish<PREC, R>(P, s, mid, sink);
    }
    warp_count(&bs.c[sp][cCont], o.cont);
    warp_count(&bs.c[sp][cClamp], o.clamped);
    return __popc(m);
}

// Photons of ne recorded emitters whose first slot is known (one warp;
// record(e): the stash record of emitter e): emitter after emitter; those beyond the capacity are counted as dropped with
// their energy.
template <int PREC, class Record>
__device__ __forceinline__ void write_photons(const Problem &P, const StepTime &tm, int sp, int ne,
                                              const double *st, int cap, Record record,
                                              long long base, BlockStats &bs)
{
    const int lane = threadIdx.x & 31;
    const SpeciesDev &Ph = P.sp[2];
    const bool photons = Ph.present != 0;
    unsigned stored = 0, dropped = 0;
    double e_drop = 0.0;
#pragma unroll 1
    for (int e0 = 0; e0 < ne; e0 += 32) {
        const double *r = st + (e0 + lane < ne ? record(e0 + lane) : 0);
        unsigned long long what =
            e0 + lane < ne ? (unsigned long long)__double_as_longlong(r[kStashWhat * cap]) : 0ull;
        const int n = (int)(what & 15ull);
        int inc = n;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, inc, d);
            if (lane >= d) inc += y;
        }
        if (n) {
            const double x = r[0], y = r[cap], z = r[2 * cap];
            const double kx = r[3 * cap], ky = r[4 * cap], kz = r[5 * cap], wgt = r[6 * cap];
            const int64_t i = __double_as_longlong(r[kStashSlot * cap]);
            int64_t slot = base + (inc - n);
            r += kStashGg * cap;
#pragma unroll 1
            for (int k = 0; k < n; ++k, ++slot, r += cap) {
                const double gg = *r;
                what >>= 4;
                if (photons && slot < Ph.cap) {
                    Ph.x[slot] = x;
                    Ph.y[slot] = y;
                    if (Ph.z) Ph.z[slot] = z;
                    Ph.ux[slot] = gg * kx;
                    Ph.uy[slot] = gg * ky;
                    Ph.uz[slot] = gg * kz;
                    Ph.tau[slot] = photon_depth<PREC>(P, tm, sp, i, (int)(what & 15ull));
                    Ph.w[slot] = wgt;
                    if (Ph.chi) Ph.chi[slot] = 0.0;
                    if (Ph.nemit) Ph.nemit[slot] = 0;
                    ++stored;
                } else {
                    ++dropped;
                    e_drop += wgt * gg;
                }
            }
        }
        base += __shfl_sync(0xFFFFFFFFu, inc, 31);
    }
    warp_add(&bs.c[sp][cPhoton], stored);
    if (__any_sync(0xFFFFFFFFu, dropped != 0)) {
        warp_add(&bs.c[sp][cPhotonDrop], dropped);
        warp_add(&bs.e[sp][1], e_drop);
    }
}

// Ballistic motion of a photon over one step, x += c k^ dt: one copy of the
// arithmetic for every place a photon moves (the step's photon tiles and
// the fused steps), with every rounding explicit (a product left to the
// compiler could be fused into the add in one place and hoisted out of a
// loop in the other), so both give the same bits.
__device__ __forceinline__ double photon_u64(double ux, double uy, double uz)
{
    return __fma_rn(uz, uz, __fma_rn(uy, uy, __dmul_rn(ux, ux)));  // |u|^2
}
__device__ __forceinline__ double photon_move64(double x, double u, double ig, double dt)
{
    return __fma_rn(dt, __dmul_rn(u, ig), x);  // ig = 1/|u|
}
__device__ __forceinline__ float photon_speed32(float fx, float fy, float fz)
{
    return sqrtf(fx * fx + fy * fy + fz * fz);
}
__device__ __forceinline__ double photon_move32(double x, float f, float c)
{
    return add_fd(x, c * f);
}

// -------------------------------------------------------------------- photon step

// One step of the photon in slot i: chi_gamma, pair optical depth, motion.
// True if it decays: it is marked dead and chi_d is its chi.
template <int PREC, int FK, typename R>
__device__ __forceinline__ bool photon_step(const StepArgs &a, const Problem &P,
                                            const StepTime &tm, const R *T,
                                            int64_t i, bool &clamped, double &chi_d)
{
    const SpeciesDev &Ph = P.sp[2];
    const bool pairs = P.pairs != 0;
    bool decayed = false;
    // all loads before the test: decayed photons lie among live ones, whose
    // sectors are read anyway, and a load after the test waits once more
    const double taud = Ph.tau[i];
    const double px = Ph.x[i], py = Ph.y[i], pz = Ph.z ? Ph.z[i] : 0.0;
    const double gux = Ph.ux[i], guy = Ph.uy[i], guz = Ph.uz[i];
    if (!(taud >= 0.0)) return false;
    if constexpr (PREC == kFP64) {
        const double u2 = photon_u64(gux, guy, guz);
        const double ig = u2 > 0.0 ? rsqrt64(u2) : 0.0;
        const double dt = P.dt;
        if (pairs && u2 > 4.0) {
            Vec3<R> E, B;
            eval_field<FK>(P.f, px, py, pz, tm.t, E, B);
            const double kx = gux * ig, ky = guy * ig, kz = guz * ig;
            const double ax = E.x + (ky * B.z - kz * B.y);
            const double ay = E.y + (kz * B.x - kx * B.z);
            const double az = E.z + (kx * B.y - ky * B.x);
            const double ke = kx * E.x + ky * E.y + kz * E.z;
            const double s = ax * ax + ay * ay + az * az - ke * ke;
            // |u| sqrt(s) as one root
            const double us = u2 * s;
            const double chi = us > 0.0 ? root_of(us, rsqrt64(us)) * a.inv_aS : 0.0;
            const double Tr = rate64<2>(T, chi, clamped);
            const double dtau = a.C_rate * Tr * ig * dt;
            if (Ph.chi) Ph.chi[i] = chi;
            if (dtau > 0.0 && !(taud > dtau)) {
                decayed = true;
                chi_d = chi;
                Ph.tau[i] = -1.0;
            } else {
                Ph.tau[i] = taud - dtau;
            }
        }
        if (!decayed && u2 > 0.0) {
            Ph.x[i] = photon_move64(px, gux, ig, dt);
            Ph.y[i] = photon_move64(py, guy, ig, dt);
            if (Ph.z) Ph.z[i] = photon_move64(pz, guz, ig, dt);
        }
    } else {
        // ---- mixed precision: FP32 physics, FP64 accumulation by
        // integer instructions
        const MixedConsts &m = P.mc;
        const float fx = hi_d(gux), fy = hi_d(guy), fz = hi_d(guz);
        const float g = photon_speed32(fx, fy, fz);
        if (pairs && g > 2.0f) {
            Vec3<float> E, B;
            eval_field_mixed<FK>(P.f, m, tm, px, py, pz, E, B);
            const float ig = 1.0f / g;
            const float kx = fx * ig, ky = fy * ig, kz = fz * ig;
            const float ax = E.x + (ky * B.z - kz * B.y);
            const float ay = E.y + (kz * B.x - kx * B.z);
            const float az = E.z + (kx * B.y - ky * B.x);
            const float ke = kx * E.x + ky * E.y + kz * E.z;
            const float s2 = ax * ax + ay * ay + az * az - ke * ke;
            const float chi =
                s2 > 0.0f ? over_aS(g * sqrtf(s2), m.inv_aS, m.inv_aS_lo) : 0.0f;
            const float Tr = rate32<2>(T, chi, clamped);
            const float dtau = m.C_rate * Tr / g * m.dt;
            if (Ph.chi) Ph.chi[i] = finite_to_d(chi);
            const df2 TAU = split_d(taud);
            if (dtau > 0.0f && !(TAU.hi > dtau || (TAU.hi == dtau && TAU.lo > 0.0f))) {
                decayed = true;
                chi_d = finite_to_d(chi);
                Ph.tau[i] = -1.0;
            } else if (dtau != 0.0f) {
                Ph.tau[i] = add_fd(taud, -dtau);
            }
        }
        if (!decayed && g > 0.0f) {
            const float c = m.dt / g;
            Ph.x[i] = photon_move32(px, fx, c);
            Ph.y[i] = photon_move32(py, fy, c);
            if (Ph.z) Ph.z[i] = photon_move32(pz, fz, c);
        }
    }
    if (decayed && Ph.nemit) Ph.nemit[i] += 1;
    return decayed;
}

// The e-/e+ pairs of n decayed photons whose first pair number is known (one
// warp, a lane a pair; record(e, i): chi and slot i of pair e): pair e goes to
// slots be + excl + e and bp + excl + e while excl + e is below `room`;
// beyond it the pair is dropped and its energy counted.  The energies and
// optical depths are sampled here (Eq. 7), on packed lanes, from the chi in
// the stash and the photon's slot, which nothing has touched since it
// decayed.
template <int PREC, int NODES, class Record>
__device__ __forceinline__ void write_pairs(const StepArgs &a, const Problem &P,
                                            const StepTime &tm, int n,
                                            Record record, long long excl, long long be,
                                            long long bp, long long room, BlockStats &bs)
{
    const SpeciesDev &El = P.sp[0], &Po = P.sp[1], &Ph = P.sp[2];
    const bool leptons = El.present && Po.present;
#pragma unroll 1
    for (int e = threadIdx.x & 31; e < n; e += 32) {
        int64_t i;
        const double chi = record(e, i);
        const double gux = Ph.ux[i], guy = Ph.uy[i], guz = Ph.uz[i];
        const double wg = Ph.w[i];
        const int64_t ord = excl + e;
        if (leptons && ord < room) {
            const double px = Ph.x[i], py = Ph.y[i], pz = Ph.z ? Ph.z[i] : 0.0;
            const uint4 r1 = draw(P.seed, QP_PHOTON, kRngPair, particle_id(Ph, i), tm.step, 0);
            const uint4 r2 = draw(P.seed, QP_PHOTON, kRngPairPos, particle_id(Ph, i), tm.step, 0);
            double v, om, tm, tp;
            bool clamped = false;  // counted with the rate, at the same chi
            if constexpr (PREC == kFP64) {
                v = sample_cdf(a.tab.Cp, a.tab.Gp, chi, u53(r1.x, r1.y), kSpMin, kSpSpan,
                                       false, clamped);
                om = 1.0 - v;
                tm = -log(u53(r1.z, r1.w));
                tp = -log(u53(r2.x, r2.y));
            } else {
                const FracPair vf = sample_cdf_f<NODES>(
                    a.tab.Cp2, a.tab.Qp2, a.tab.Gp, a.tab.Ep, hi_d(chi), u53_pair(r1.x, r1.y),
                    u53_pair_complement(r1.x, r1.y), (float)(kSpSpan / (kNNode - 1)), false,
                    clamped);
                v = finite_to_d(vf.x);
                om = finite_to_d(vf.omx);
                tm = finite_to_d(-logf(u53f(r1.z, r1.w)));
                tp = finite_to_d(-logf(u53f(r2.x, r2.y)));
            }
            const int64_t se = be + ord, spo = bp + ord;
            El.x[se] = px;
            El.y[se] = py;
            if (El.z) El.z[se] = pz;
            El.ux[se] = v * gux;
            El.uy[se] = v * guy;
            El.uz[se] = v * guz;
            El.tau[se] = tm;
            El.w[se] = wg;
            if (El.chi) El.chi[se] = 0.0;
            if (El.nemit) El.nemit[se] = 0;
            Po.x[spo] = px;
            Po.y[spo] = py;
            if (Po.z) Po.z[spo] = pz;
            Po.ux[spo] = om * gux;
            Po.uy[spo] = om * guy;
            Po.uz[spo] = om * guz;
            Po.tau[spo] = tp;
            Po.w[spo] = wg;
            if (Po.chi) Po.chi[spo] = 0.0;
            if (Po.nemit) Po.nemit[spo] = 0;
        } else {
            atomicAdd(&bs.c[2][cPairDrop], 1u);
            atomicAdd(&bs.e[2][1], wg * sqrt(gux * gux + guy * guy + guz * guz));
        }
    }
}

// One sub-tile of 32 photons stepped by a warp, lane l the slot i (below n);
// the records of those that decay go to st in slot order.  Returns their
// number.
template <int PREC, int FK, typename R>
__device__ __forceinline__ int step_photons(const StepArgs &a, const Problem &P,
                                            const StepTime &tm, const R *T,
                                            int64_t i, int64_t n, double *st, int cap,
                                            BlockStats &bs)
{
    bool decayed = false, clamped = false;
    double chi = 0.0;
    if (i < n) decayed = photon_step<PREC, FK, R>(a, P, tm, T, i, clamped, chi);
    warp_count(&bs.c[2][cClamp], clamped);
    const unsigned m = __ballot_sync(0xFFFFFFFFu, decayed);
    if (decayed) {
        double *r = st + __popc(m & ((1u << (threadIdx.x & 31)) - 1u));
        r[0] = chi;
        r[kStashSlot * cap] = __longlong_as_double((long long)i);
    }
    const int total = __popc(m);
    if ((threadIdx.x & 31) == 0 && total) atomicAdd(&bs.c[2][cPair], (unsigned)total);
    return total;
}

// -------------------------------------------------------------------- the step

// Live slots of one problem in this step, and its long or short tiles.  Live
// counts and step counters change only at the end of a step (last block),
// so every block sees the same values.  Counts outside [0, capacity] are
// clamped (and reported).
struct ProbCounts {
    long long n[3];
    long long tiles_e, tiles_l, tiles_g;
    bool active, bad;
    __device__ __forceinline__ void set_tiles(bool lng)
    {
        const int s = lng ? kLongShift : kShortShift;
        const long long m = (1ll << s) - 1;
        tiles_e = (n[0] + m) >> s;
        tiles_l = tiles_e + ((n[1] + m) >> s);
        tiles_g = (n[2] + m) >> s;
    }
};

__device__ __forceinline__ ProbCounts problem_counts(const Problem &P)
{
    ProbCounts c{};
    // every counter is loaded before any is tested, so the (uncached) reads
    // overlap instead of following each other
    long long v[3], left = 1;
#pragma unroll
    for (int s = 0; s < 3; ++s) v[s] = P.sp[s].present ? __ldcg(P.sp[s].n_live) : 0;
    if (P.device_step) left = __ldcg(P.left_ctr);
    c.active = left > 0;
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        long long x = c.active ? v[s] : 0;
        if (x < 0 || x > P.sp[s].cap) {
            c.bad = true;
            x = x < 0 ? 0 : P.sp[s].cap;
        }
        c.n[s] = x;
    }
    return c;
}

// The step's index, and its time as the field reads it: FP64, or the mixed path's
// double-float constants (a 2D grid and a constant field need none).
template <int PREC, int FK>
__device__ __forceinline__ void set_time(StepTime &tm, const Problem &P, long long step)
{
    tm.step = (uint64_t)step;
    if constexpr (FK == QP_FIELD_PLANE || FK == QP_FIELD_GAUSSIAN) {
        const double t = __dmul_rn((double)step, P.dt);  // (rounded: no sum may take it in)
        if constexpr (PREC == kFP64) {
            tm.t = t;
        } else if constexpr (FK == QP_FIELD_PLANE) {
            tm.t_hi = __double2float_rn(t);
            tm.t_lo = __double2float_rn(t - (double)tm.t_hi);
        } else {
            const double tr = t - P.f.t_focus;
            tm.tr_hi = __double2float_rn(tr);
            tm.tr_lo = __double2float_rn(tr - (double)tm.tr_hi);
        }
    }
}

// Block-wide inclusive scan of v[0..n) in place (n <= 2 kTile).
__device__ void scan_offsets(long long *v, int n, long long *s_tmp)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long a = 2 * tid < n ? v[2 * tid] : 0, b = 2 * tid + 1 < n ? v[2 * tid + 1] : 0;
    long long inc = a + b;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const long long y = __shfl_up_sync(0xFFFFFFFFu, inc, d);
        if (lane >= d) inc += y;
    }
    if (lane == 31) s_tmp[warp] = inc;
    __syncthreads();
    long long before = 0;
    for (int w = 0; w < warp; ++w) before += s_tmp[w];
    const long long excl = before + inc - (a + b);
    __syncthreads();
    if (2 * tid < n) v[2 * tid] = excl + a;
    if (2 * tid + 1 < n) v[2 * tid + 1] = excl + a + b;
    __syncthreads();
}

// -------------------------------------------------------------------- short tiles

struct ShortRec {
    int chain, last, sp, total;
    unsigned tile;
    unsigned arrived;              // warps past the tile's physics (never reset)
    unsigned claimed, resolved;    // chunks of 32 emitters taken, done
    int made;                      // emitters run in place: photons they append
    int count[kWarps];             // listed slots of each warp
    long long first;               // the tile's first slot
    unsigned char list[kTile];     // warp w's listed threads, in order, from 32 w on
};

// The index in the list of the tile's listed slot number e (slot order).
__device__ __forceinline__ int listed_entry(const ShortRec &r, int e)
{
    int w = 0;
#pragma unroll
    for (int k = 0; k < kWarps - 1; ++k)
        if (w == k && e >= r.count[k]) {
            e -= r.count[k];
            ++w;
        }
    return 32 * w + e;
}

__device__ __forceinline__ int listed_total(const ShortRec &r)
{
    int n = 0;
#pragma unroll
    for (int k = 0; k < kWarps; ++k) n += r.count[k];
    return n;
}

// One warp's listed slots go to the tile's record; true in the warp that
// comes last (it sees every warp's list).
__device__ __forceinline__ bool list_slots(ShortRec &r, bool listed)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned m = __ballot_sync(0xFFFFFFFFu, listed);
    if (listed) r.list[32 * warp + __popc(m & ((1u << lane) - 1u))] = (unsigned char)threadIdx.x;
    __syncwarp();
    unsigned old = 0u;
    if (lane == 0) {
        r.count[warp] = __popc(m);
        __threadfence_block();
        old = atomicAdd(&r.arrived, 1u);
        __threadfence_block();
    }
    old = __shfl_sync(0xFFFFFFFFu, old, 0);
    return old % (unsigned)kWarps == (unsigned)(kWarps - 1);
}

// The physics of a lepton tile; emitters are listed, what they carry stays in
// entry `half` + lane of the warps' queues.  Or they run in place (see
// kEmitInPlace), the record of thread t at t.  True in the warp that came last.
template <int PREC, int FK, typename R>
__device__ __forceinline__ bool short_leptons(const StepArgs &a, const Problem &P,
                                              const StepTime &tm, Smem<FK, R> &sm,
                                              unsigned long long *bar, bool &loaded, ShortRec &rec,
                                              unsigned half, int sp, int64_t first, int64_t n,
                                              BlockStats &bs, double *st)
{
    const int tid = threadIdx.x;
    const SpeciesDev &S = P.sp[sp];
    const int64_t i = first + tid;
    LeptonOut o{};
    bool event = false;
    double wgt = 0.0;
    if (i < n) {
        const LeptonState s{S.x[i],  S.y[i],  S.z ? S.z[i] : 0.0, S.ux[i],
                            S.uy[i], S.uz[i], S.tau[i]};
        StashSink sink{a, loaded ? nullptr : bar, nullptr, 0, 0, S.chi ? S.chi + i : nullptr, S, i,
                       0ull};
        LeptonMid<R> mid;
        event = lepton_push<PREC, FK, R>(a, P, tm, sm.H, sm.G, sp, s, mid, o, sink);
        if (!event)
            lepton_finish<PREC, R>(P, s, mid, sink);
        else if constexpr (kEmitInPlace<FK, R>)
            run_emitter<PREC, FK, R>(a, P, tm, sm.H, sp, i, s, mid, st, kTile, tid, o, wgt);
        else
            mid_put<FK, R>(sm.mid[tid >> 5], (int)half + (tid & 31), mid);
    }
    if (!loaded) {
        // the rate tables' copy was issued in the kernel's prologue
        // (stage_rate_tables); every thread waits once: later tiles read the
        // tables without a wait, and the block never leaves with the copy in
        // flight
        wait_tables(bar, a);
        loaded = true;
    }
    warp_count(&bs.c[sp][cCont], o.cont);
    warp_count(&bs.c[sp][cClamp], o.clamped);
    if (kEmitInPlace<FK, R> && __any_sync(0xFFFFFFFFu, event)) {
        const int photons = count_emitters(bs, sp, o, wgt);
        if ((tid & 31) == 0) atomicAdd(&rec.made, photons);
    }
    return list_slots(rec, event);
}

// The physics of a photon tile; decaying photons are listed, their records in
// entry 32 w + k of the stash for warp w's k-th.  True in the warp that came
// last.
template <int PREC, int FK, typename R>
__device__ __forceinline__ bool short_photons(const StepArgs &a, const Problem &P,
                                              const StepTime &tm, const R *T,
                                              ShortRec &rec, int64_t first, int64_t n,
                                              BlockStats &bs, double *st)
{
    const int tid = threadIdx.x;
    const int64_t i = first + tid;
    bool decayed = false, clamped = false;
    if (i < n) {
        double chi = 0.0;
        decayed = photon_step<PREC, FK, R>(a, P, tm, T, i, clamped, chi);
        if (decayed) st[tid] = chi;
    }
    warp_count(&bs.c[2][cClamp], clamped);
    warp_count(&bs.c[2][cPair], decayed);
    return P.pairs && list_slots(rec, decayed);
}

// The emitters of a lepton tile, in chunks of 32 that the warps of the block
// claim as they come free, or spread over all of them when the block has no
// other tile (fewer lanes take fewer of the branches).  True in the warp that finished the last chunk (it
// published the aggregate and sees the whole stash).
template <int PREC, int FK, typename R>
__device__ __forceinline__ bool resolve_emitters(const StepArgs &a, const Problem &P,
                                                 const StepTime &tm, const Smem<FK, R> &sm, ShortRec &rec,
                                                 unsigned half, bool spread, unsigned epoch,
                                                 BlockStats &bs, double *st)
{
    const int lane = threadIdx.x & 31;
    const int ne = listed_total(rec);
    const int size = spread ? min(32, max(4, (ne + kWarps - 1) / kWarps)) : 32;
    const unsigned chunks = (unsigned)(ne + size - 1) / (unsigned)size;
    const int sp = rec.sp;
    bool last = false;
#pragma unroll 1
    for (;;) {
        unsigned c = 0u;
        if (lane == 0) c = atomicAdd(&rec.claimed, 1u);
        c = __shfl_sync(0xFFFFFFFFu, c, 0);
        if (c >= chunks) return last;
        const int e0 = (int)c * size, n = min(size, ne - e0);
        const int t = lane < n ? rec.list[listed_entry(rec, e0 + lane)] : 0;
        const int tot = run_emitters<PREC, FK, R>(a, P, tm, sm.H, sm.mid[t >> 5],
                                                  (int)half + (t & 31), n, sp, rec.first + t, e0,
                                                  st, kTile, bs);
        // every lane's records before the chunk counts as done
        __threadfence_block();
        __syncwarp();
        unsigned d = 0u;
        if (lane == 0) {
            if (tot) atomicAdd(&rec.total, tot);
            __threadfence_block();
            d = atomicAdd(&rec.resolved, 1u);
            __threadfence_block();
        }
        d = __shfl_sync(0xFFFFFFFFu, d, 0);
        if (d == chunks - 1u) {
            if (lane == 0)
                publish_aggregate(P.lep_words, rec.tile, *(volatile int *)&rec.total, epoch);
            last = true;
        }
    }
}

// Pairs there is room for beside the live leptons.
__device__ __forceinline__ long long pair_room(const Problem &P, const ProbCounts &pc)
{
    if (!P.sp[0].present || !P.sp[1].present) return 0;
    const long long e = P.sp[0].cap - pc.n[0], p = P.sp[1].cap - pc.n[1];
    const long long room = e < p ? e : p;
    return room < 0 ? 0 : room;
}

// The live counts after the last tile of a chain, whose particles are number
// excl .. excl + total - 1 (applied at the end of the step).
__device__ __forceinline__ void set_pending(const StepArgs &a, const Problem &P,
                                            const ProbCounts &pc, int chain, long long excl,
                                            int total)
{
    if (chain == 0) {
        const long long tot = pc.n[2] + excl + total;
        if (P.sp[2].present) {
            P.pending[2] = tot < P.sp[2].cap ? tot : P.sp[2].cap;
            if (tot > P.sp[2].cap) raise_status(a.status, QP_WARN_BUFFER_FULL);
        } else if (tot > pc.n[2]) {
            raise_status(a.status, QP_WARN_BUFFER_FULL);
        }
    } else {
        const long long room = pair_room(P, pc), tot = excl + total;
        const long long add = tot < room ? tot : room;
        P.pending[0] = pc.n[0] + add;
        P.pending[1] = pc.n[1] + add;
        if (tot > add) raise_status(a.status, QP_WARN_BUFFER_FULL);
    }
}

// A tile's prefix is resolved (its predecessors are, by now, almost always
// published) and its photons or pairs are written, by one warp.  HERE: its
// emitters ran in place.
template <int PREC, int FK, bool HERE>
__device__ __forceinline__ void flush_short(const StepArgs &a, const Problem &P,
                                            const ProbCounts &pc, const ShortRec &rec,
                                            const StepTime &tm, unsigned epoch, BlockStats &bs, const double *st)
{
    const int total = *(const volatile int *)&rec.total, chain = rec.chain;
    const long long excl = resolve_prefix(chain ? P.pho_words : P.lep_words, rec.tile, total,
                                          epoch, a.spin_limit, a.status);
    if (rec.last && (threadIdx.x & 31) == 0) set_pending(a, P, pc, chain, excl, total);
    if (!total) return;
    if (chain == 0)
        write_photons<PREC>(
            P, tm, rec.sp, listed_total(rec), st, kTile,
            [&](int e) { return HERE ? (int)rec.list[listed_entry(rec, e)] : e; },
            pc.n[2] + excl, bs);
    else
        write_pairs<PREC, kWindowNodes<FK>>(
            a, P, tm, total,
            [&](int e, int64_t &i) {
                const int t = rec.list[listed_entry(rec, e)];
                i = rec.first + t;
                return st[t];
            },
            excl, pc.n[0], pc.n[1], pair_room(P, pc), bs);
}

// -------------------------------------------------------------------- long tiles

// One tile in flight, shared by the block's warps (counts never reset: the
// use u of a record is complete when they reach warps x (u + 1)).
struct TileRec {
    unsigned arrived;         // warps that have counted their part
    unsigned flushed;         // warps that have written their part
    unsigned claim, ready;    // 1 + the tile whose prefix a warp looks up, has looked up
    int count[kWarps];        // particles each part appends
    long long excl;           // the tile's prefix
};

// A warp's part of a tile in flight (read by that warp only).
struct PartRec {
    int chain;                // 0 leptons, 1 photons, 2 nothing to append
    int last, sp, n;          // last tile of its chain; species; records of the stash
    unsigned tile;
};

// Wait until *p reaches `target` (shared memory, one warp; bounded).
__device__ __noinline__ void await_count(const unsigned *p, unsigned target, unsigned limit,
                                         int *status)
{
    unsigned spins = 0;
    while ((int)(*(const volatile unsigned *)p - target) < 0) {
        if (++spins > limit) {
            if ((threadIdx.x & 31) == 0) raise_status(status, QP_ERR_TIMEOUT);
            break;
        }
        __nanosleep(64);
    }
    __threadfence_block();
    __syncwarp();
}

// A photon part of a problem without pairs: nothing to append.
__device__ __forceinline__ void count_part_empty(TileRec &rec)
{
    __syncwarp();
    if ((threadIdx.x & 31) == 0) atomicAdd(&rec.arrived, 1u);
}

// The ticket of the next tile: the first warp of the block to start tile n
// takes it from the counter and hands it over once it has come back (after
// the warp's first sub-tile), so that no warp stalls on the atomic.
struct NextTicket {
    long long *slot;      // s_ticket entry, NULL when another warp fetches
    unsigned *done;       // s_tdone
    unsigned n_done;      // its value with this ticket
    long long t;
    __device__ __forceinline__ void hand_over()
    {
        if (slot) {
            *(volatile long long *)slot = t;
            __threadfence_block();
            *(volatile unsigned *)done = n_done;
            slot = nullptr;
        }
    }
};

// One warp's part of tile `rec` appends `total` particles (the use of the
// record ends when `target` warps have counted); the last warp publishes.
__device__ __forceinline__ void count_part(TileRec &rec, int warp, unsigned target,
                                           int total, unsigned long long *words, unsigned tile,
                                           unsigned epoch)
{
    __syncwarp();
    if ((threadIdx.x & 31) == 0) {
        rec.count[warp] = total;
        __threadfence_block();
        if (atomicAdd(&rec.arrived, 1u) + 1u == target) {
            __threadfence_block();
            int sum = 0;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) sum += *(volatile int *)&rec.count[w];
            publish_aggregate(words, tile, sum, epoch);
        }
    }
}

// The physics of a warp's part of a lepton tile: slots [first, first + 32 S)
// below n.  `records`: emitters of the part; returns the photons it appends.
template <int PREC, int FK, typename R>
__device__ __forceinline__ int lepton_part(const StepArgs &a, const Problem &P,
                                           const StepTime &tm, Smem<FK, R> &sm,
                                           unsigned long long *bar, bool &loaded, int warp, int sp,
                                           int64_t first, int64_t n, unsigned *slots, double *st,
                                           BlockStats &bs, int &records, NextTicket &next)
{
    const int lane = threadIdx.x & 31;
    R(*mids)[kQueue] = sm.mid[warp];
    unsigned head = 0u, tail = 0u;
    int total = 0;
#pragma unroll 1
    for (int sub = 0; sub < kSubTiles;) {
        tail += (unsigned)push_leptons<PREC, FK, R>(a, P, tm, sm, bar, loaded, sp,
                                                    first + 32 * sub + lane, n, mids, slots, tail,
                                                    (unsigned)(32 * sub + lane), bs);
        __syncwarp();
        next.hand_over();
        ++sub;
        if (first + 32 * sub >= n) sub = kSubTiles;  // no slot left
        // 32 emitters run as they come, the rest at the end of the part (two
        // rounds at most: fewer than 32 waited and 32 came)
#pragma unroll 1
        while (tail - head >= 32u || (sub == kSubTiles && tail != head)) {
            const int ne = min(32, (int)(tail - head));
            const int t = (int)((head + (unsigned)lane) % (unsigned)kQueue);
            total += run_emitters<PREC, FK, R>(a, P, tm, sm.H, mids, t, ne, sp,
                                               first + (lane < ne ? slots[t] : 0u), (int)head, st,
                                               kPart, bs);
            head += (unsigned)ne;
            __syncwarp();
        }
    }
    records = (int)head;
    return total;
}

// The physics of a warp's part of a photon tile.  Returns its pairs, their
// records in slot order.
template <int PREC, int FK, typename R>
__device__ __forceinline__ int photon_part(const StepArgs &a, const Problem &P,
                                           const StepTime &tm, const R *T,
                                           int64_t first, int64_t n, double *st, BlockStats &bs,
                                           NextTicket &next)
{
    int total = 0;
#pragma unroll 1
    for (int sub = 0; sub < kSubTiles && first + 32 * sub < n; ++sub) {
        total += step_photons<PREC, FK, R>(a, P, tm, T, first + 32 * sub + (threadIdx.x & 31), n,
                                           st + total, kPart, bs);
        next.hand_over();
    }
    return total;
}

// A warp's part of a tile in flight is written: the tile's prefix is looked up
// by the first warp of the block to come here (its predecessors are, by now,
// almost always published), then every warp writes its own photons or pairs
// behind the parts before it.
template <int PREC, int FK>
__device__ __forceinline__ void flush_part(const StepArgs &a, const Problem &P,
                                           const StepTime &tm,
                                           const ProbCounts &pc, const PartRec &part,
                                           TileRec &rec, unsigned tile_no, int warp, unsigned epoch,
                                           BlockStats &bs, const double *st)
{
    const int lane = threadIdx.x & 31;
    const int chain = part.chain;
    if (chain != 2) {
        await_count(&rec.arrived, (tile_no / (unsigned)kRing + 1u) * (unsigned)kWarps,
                    a.spin_limit, a.status);
        unsigned first = 0u;
        if (lane == 0) first = atomicMax(&rec.claim, tile_no + 1u) <= tile_no;
        first = __shfl_sync(0xFFFFFFFFu, first, 0);
        int total = 0, before = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            if (w == warp) before = total;
            total += *(const volatile int *)&rec.count[w];
        }
        long long excl;
        if (first) {
            excl = resolve_prefix(chain ? P.pho_words : P.lep_words, part.tile, total, epoch,
                                  a.spin_limit, a.status);
            if (lane == 0) {
                rec.excl = excl;
                __threadfence_block();
                *(volatile unsigned *)&rec.ready = tile_no + 1u;
                if (part.last) set_pending(a, P, pc, chain, excl, total);
            }
        } else {
            await_count(&rec.ready, tile_no + 1u, a.spin_limit, a.status);
            excl = *(const volatile long long *)&rec.excl;
        }
        excl += before;
        if (part.n) {
            if (chain == 0)
                write_photons<PREC>(P, tm, part.sp, part.n, st, kPart, [](int e) { return e; },
                                    pc.n[2] + excl, bs);
            else
                write_pairs<PREC, kWindowNodes<FK>>(
                    a, P, tm, part.n,
                    [&](int e, int64_t &i) {
                        i = __double_as_longlong(st[kStashSlot * kPart + e]);
                        return st[e];
                    },
                    excl, pc.n[0], pc.n[1], pair_room(P, pc), bs);
        }
    }
    __syncwarp();
    if (lane == 0) {
        __threadfence_block();
        atomicAdd(&rec.flushed, 1u);
    }
}

// Everything a block keeps in shared memory (dynamic, so that the loop over
// long tiles, a function of its own, addresses it directly).
template <int FK, typename R>
struct StepShared {
    Smem<FK, R> sm;
    unsigned long long bar[2];        // TMA: lepton, photon tables
    long long ticket[kTickets];       // ticket of tile n at n % kTickets
    unsigned tdone, tclaim;           // long: tiles with a ticket; being fetched
    unsigned claim;                   // short: warps that asked to flush
    int last, go;                     // the step's last block; the next step has begun
    long long tmp[kWarps];
    unsigned long long subs;          // 32-slot sub-tiles of the step
    BlockStats bs;
    StepTime tm;                      // of the current problem's step
    ProbCounts pc;                    // of the current problem
    long long off[kMaxProblems + 1];  // tickets of problems 0..b
    int tl[kMaxProblems], tg[kMaxProblems];
    union {
        ShortRec shrt[kRing];
        struct {
            TileRec rec[kRing];
            PartRec part[kWarps][kRing];
        } lng;
    } ring;
    // long: slots of the queued emitters
    unsigned slots[has_long_tiles(FK) ? kWarps : 1][has_long_tiles(FK) ? kQueue : 1];
    alignas(16) Problem prob;         // batch, or long: the problem of the current tile
};

// The problem of ticket t in a batch: the first b with off[b] > t.
__device__ __forceinline__ int problem_of(const long long *off, int np, long long t)
{
    int lo = 0, hi = np - 1;
#pragma unroll 1
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] > t)
            hi = mid;
        else
            lo = mid + 1;
    }
    return lo;
}

// All threads of a block leave the problem `cur` (P; -1: none): its counters
// are added to the species'.
__device__ __forceinline__ void leave_problem(const StepArgs &a, const Problem &P, int cur,
                                              BlockStats &bs)
{
    if (cur < 0) return;
    flush_stats(bs, a, P);  // begins with a barrier
    __syncthreads();
    clear_stats(bs);
}

// Problem b takes its place in shared memory, cut into long or short tiles.
template <int PREC, int FK, typename R>
__device__ __forceinline__ void enter_problem(StepShared<FK, R> &sh, const Problem &src, bool lng)
{
    const int *from = reinterpret_cast<const int *>(&src);
    int *to = reinterpret_cast<int *>(&sh.prob);
#pragma unroll 1
    for (int k = threadIdx.x; k < (int)(sizeof(Problem) / sizeof(int)); k += kTile)
        to[k] = from[k];
    __syncthreads();
    if (threadIdx.x == 0) {
        sh.pc = problem_counts(sh.prob);
        sh.pc.set_tiles(lng);
        if (sh.prob.device_step)
            set_time<PREC, FK>(sh.tm, sh.prob, *((volatile long long *)sh.prob.step_ctr));
    }
    __syncthreads();
}

// A block's long tiles.  A function of its own, with the problem in shared
// memory: beside the loop over short tiles in one function the registers of
// both spilled (serving steps 38 -> 42 ms a stream).
template <int PREC, int FK, bool BATCH>
__device__ __noinline__ void long_tile_loop(const StepArgs &a, const Problem *table, int np,
                                            unsigned tbase, unsigned epoch, double *stash)
{
    using R = typename std::conditional<PREC == kFP64, double, float>::type;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    StepShared<FK, R> &sh = *reinterpret_cast<StepShared<FK, R> *>(smem_raw);
    Smem<FK, R> &sm = sh.sm;
    BlockStats &bs = sh.bs;
    const Problem &P = sh.prob;
    const StepTime &tm = sh.tm;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long n_tickets = sh.off[np - 1];
    bool lep_loaded = false, ph_loaded = false;
    int cur = -1;  // the problem in shared memory
    double *const parts = stash + (size_t)warp * (kLag + 1) * kStashFieldsHost * kPart;
    auto part_stash = [&](unsigned n) {
        return parts + (size_t)(n % (unsigned)(kLag + 1)) * kStashFieldsHost * kPart;
    };
    unsigned n = 0u;   // the block's tiles before this one (the same in every warp)
    unsigned lo = 0u;  // tiles this warp has written
    for (;;) {
        // the ticket of tile n
        if (n) await_count(&sh.tdone, n + 1u, a.spin_limit, a.status);
        const long long t = *(const volatile long long *)&sh.ticket[n % kTickets];
        const bool more = t < n_tickets;
        const int b = BATCH && more ? problem_of(sh.off, np, t) : 0;
        const bool leave = !more || b != cur;  // the problem's last tile is done
        if (!leave) {
            TileRec &rec = sh.ring.lng.rec[n % kRing];
            PartRec &part = sh.ring.lng.part[warp][n % kRing];
            // the record's previous tile has left every warp
            if (n >= (unsigned)kRing)
                await_count(&rec.flushed, n / (unsigned)kRing * (unsigned)kWarps,
                            a.spin_limit, a.status);
            NextTicket next{nullptr, &sh.tdone, n + 2u, 0};
            if (lane == 0 && atomicMax(&sh.tclaim, n + 1u) <= n) {
                next.slot = &sh.ticket[(n + 1u) % kTickets];
                next.t = (long long)tbase + atomicAdd(&a.ctl->ticket, 1u);
            }
            const ProbCounts &pc = sh.pc;
            const long long lt = t - (b > 0 ? sh.off[b - 1] : 0);  // tile within the problem
            const bool lepton = lt < pc.tiles_l;
            const int sp = !lepton ? 2 : lt < pc.tiles_e ? 0 : 1;
            const long long tile = lepton ? lt : lt - pc.tiles_l;
            const int64_t first =
                (tile - (sp == 1 ? pc.tiles_e : 0)) * kLongTile + warp * kPart;
            int total = 0, records = 0;
            if (lepton) {
                if (first < pc.n[sp])
                    total = lepton_part<PREC, FK, R>(a, P, tm, sm, &sh.bar[0], lep_loaded, warp, sp,
                                                     first, pc.n[sp], sh.slots[warp],
                                                     part_stash(n), bs, records, next);
            } else {
                if (!ph_loaded) {
                    wait_tables(&sh.bar[1], a);
                    ph_loaded = true;
                }
                if (first < pc.n[2])
                    total = records = photon_part<PREC, FK, R>(a, P, tm, sm.T, first, pc.n[2],
                                                               part_stash(n), bs, next);
            }
            const int chain = lepton ? 0 : P.pairs ? 1 : 2;  // 2: appends nothing
            if (lane == 0) {
                part.chain = chain;
                part.last = lepton ? lt == pc.tiles_l - 1 : tile == pc.tiles_g - 1;
                part.sp = sp;
                part.n = records;
                part.tile = (unsigned)tile;
            }
            if (chain != 2)
                count_part(rec, warp, (n / (unsigned)kRing + 1u) * (unsigned)kWarps, total,
                           chain ? P.pho_words : P.lep_words, (unsigned)tile, epoch);
            else
                count_part_empty(rec);
            next.hand_over();
            __syncwarp();
        }
        // parts whose turn it is (all of them before a block leaves)
        const unsigned upto = leave ? n : n + 1u > (unsigned)kLag ? n + 1u - (unsigned)kLag : 0u;
#pragma unroll 1
        for (; lo < upto; ++lo)
            flush_part<PREC, FK>(a, P, tm, sh.pc, sh.ring.lng.part[warp][lo % kRing],
                             sh.ring.lng.rec[lo % kRing], lo, warp, epoch, bs, part_stash(lo));
        if (!leave) {
            ++n;
            continue;
        }
        leave_problem(a, P, cur, bs);
        if (!more) break;
        enter_problem<PREC, FK, R>(sh, table[b], true);
        cur = b;
    }
    // the copies of the tables land before the block leaves
    if (!lep_loaded) wait_tables(&sh.bar[0], a);
    if (!ph_loaded) wait_tables(&sh.bar[1], a);
}

// One launch = one step of every active problem of a batch, or one to
// kStepsPerLaunch steps of a single problem.  Persistent blocks take
// tiles by ticket (a block's first tile of a step is fixed in a cooperative
// launch, every other ticket comes from an atomic counter, fetched while the tile before it
// runs); tickets enumerate, problem after problem, its electron tiles,
// positron tiles and photon tiles, so within each problem's chains start
// order is tile order and the decoupled look-back only ever waits on tiles
// that are running.  Waits end: every wait of a warp is for an older tile than
// the one it works on (a prefix: smaller tiles of the chain; in a long tile
// also a record of the ring, a tile's count or prefix: its block's other
// warps, at tiles no younger than its own), and a block resolves the emitters
// of a tile before it waits for any prefix of a later one; so the smallest
// unpublished tile is never held up: what its warps wait for has published
// already.  BATCH = false: the single problem of the launch parameters (read
// in place, from the constant bank); BATCH = true: a device table of problems,
// each copied to shared memory for its tiles (every warp of a block goes
// through the same tiles, so they meet at a barrier where the problem
// changes), with time and step counters advanced on the device.
// Resident blocks of 128 per SM: FP64 4 (128 registers), mixed 7 (72).
template <int PREC, int FK>
constexpr int step_min_blocks()
{
    return PREC == kFP64 ? 4 : 7;
}

template <int PREC, int FK, bool BATCH>
__global__ void __launch_bounds__(kTile, step_min_blocks<PREC, FK>())
    k_step(const __grid_constant__ StepArgs a)
{
    using R = typename std::conditional<PREC == kFP64, double, float>::type;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    StepShared<FK, R> &sh = *reinterpret_cast<StepShared<FK, R> *>(smem_raw);
    Smem<FK, R> &sm = sh.sm;
    BlockStats &bs = sh.bs;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // Tickets.  A tile must belong to a running block (its successors' look-
    // backs wait on it).  A single problem on the mixed path, or of several
    // steps a launch, is launched cooperatively (launch_step): every block is
    // resident for the whole launch, so each has a fixed first tile (its own
    // number, or spread_ticket's in launches of several steps) and later
    // tickets come from the counter, offset by the grid; no block queues on
    // the contended counter before its first tile.  An FP64 launch of one step
    // and batches take every ticket from the counter, so a tile belongs to a
    // block only once that block runs (a batch's launches are captured in
    // graphs next to other streams' kernels; the FP64 path's one-launch-a-step
    // runs of small problems, 4096 e- on 608 blocks, took 75 -> 108 us a step
    // when launched cooperatively); the first atomic overlaps the reads of the
    // live counts below.  A block whose ticket is past the last tile leaves
    // without work.
    const int n_steps = BATCH ? 1 : single_steps(a.launch);
    const bool long_ok =
        has_long_tiles(FK) && (BATCH ? __ldcg(&a.batch->long_ok) != 0u : single_long(a.launch));
    const bool fixed_first = !BATCH && (PREC != kFP64 || n_steps > 1);
    const unsigned tbase = fixed_first ? gridDim.x : 0u;
    const int np = BATCH ? a.launch : 1;
    const Problem *table = BATCH ? a.problems : &a.single;
    double *const stash = (BATCH ? a.batch->stash : a.stash) + (size_t)blockIdx.x * stash_words(long_ok);
    unsigned epoch = __ldcg(&a.ctl->epoch);
    clear_stats(bs);
    // the lepton tiles' rate tables, staged from the start by a thread of
    // another warp than the ticket's and the counts' (their copy overlaps
    // the live counts' reads and the first tile's loads, gather and push),
    // and the photon tiles' table
    if (tid == 96) {
        stage_rate_tables<PREC, FK, R>(a, sm, &sh.bar[0]);
        stage_pair_table<PREC, FK, R>(a, sm, &sh.bar[1]);
    }

    const bool spread = !BATCH && n_steps > 1;
    long long first_ticket = blockIdx.x;
    if (spread && tid == 0)
        first_ticket = spread_ticket(a.ctl, a.spin_limit, a.status);

    bool lep_loaded = false, ph_loaded = false;
    // a launch of several steps (all of its blocks are resident) takes them
    // one after the other, the blocks meeting at the end of each
#pragma unroll 1
    for (int step = 0;; ++step) {
    if (tid == 0) {
        sh.ticket[0] = fixed_first ? first_ticket : atomicAdd(&a.ctl->ticket, 1u);
        sh.tdone = 1u;
        sh.tclaim = sh.claim = 0u;
    }
    if (!BATCH && tid == 97) set_time<PREC, FK>(sh.tm, a.single, (long long)a.single.step + step);
    if (tid >= 32 && tid < 64)
        for (int k = tid - 32; k < (int)(sizeof(sh.ring) / sizeof(int)); k += 32)
            reinterpret_cast<int *>(&sh.ring)[k] = 0;
    // the live slots of every problem, the kind of tile their sum calls for,
    // the tiles of every problem and the ticket offset of each (one thread a
    // problem from 64 on: not the ticket's or the tables' warp)
    ProbCounts mine{};
    const int pb = (tid + kTile - 64) % kTile;  // this thread's problem
    static_assert(kMaxProblems <= kTile, "one thread a problem");
    if (BATCH) {
        if (tid == 0) sh.subs = 0ull;
        __syncthreads();
    }
    if (pb < np) {
        mine = problem_counts(table[pb]);
        if (mine.bad && blockIdx.x == 0) raise_status(a.status, QP_ERR_INVALID_ARG);
        const unsigned long long subs =
            (unsigned long long)((mine.n[0] + 31) / 32 + (mine.n[1] + 31) / 32 +
                                 (mine.n[2] + 31) / 32);
        if (BATCH) {
            if (subs) atomicAdd(&sh.subs, subs);
        } else {
            sh.subs = subs;
            mine.set_tiles(long_ok && long_tiles((long long)subs, (int)gridDim.x));
            sh.off[0] = mine.tiles_l + mine.tiles_g;
            sh.tl[0] = (int)mine.tiles_l;
            sh.tg[0] = (int)mine.tiles_g;
            sh.pc = mine;
        }
    }
    __syncthreads();
    const bool lng = long_ok && long_tiles((long long)sh.subs, (int)gridDim.x);
    if (BATCH) {
        if (pb < np) {
            mine.set_tiles(lng);
            sh.off[pb] = mine.tiles_l + mine.tiles_g;
            sh.tl[pb] = (int)mine.tiles_l;
            sh.tg[pb] = (int)mine.tiles_g;
        }
        __syncthreads();
        scan_offsets(sh.off, np, sh.tmp);  // sh.off[b] = tickets of problems 0..b
    }
    const long long n_tickets = sh.off[np - 1];
    if (!lng) {
        int cur = BATCH ? -1 : 0;
        constexpr bool kHere = kEmitInPlace<FK, R>;
        // tiles of this block, counted from its first (uniform over the
        // block): q started, q_ev with their events resolved (q or q - 1),
        // q_lo written
        unsigned q = 0, q_ev = 0, q_lo = 0;
        for (int buf = 0;;) {
            const long long t = sh.ticket[buf];
            const bool more = t < n_tickets;
            const int b = BATCH && more ? problem_of(sh.off, np, t) : 0;
            const bool leave = !more || (BATCH && b != cur);  // the problem's last tile is done
            // a round without a tile empties the ring before the block leaves
            const bool drain = leave && q_lo != q;
            if (leave && !drain) {
                if (BATCH || step + 1 == n_steps)
                    leave_problem(a, BATCH ? sh.prob : a.single, cur, bs);
                if (!more) break;
                if constexpr (BATCH) {
                    enter_problem<PREC, FK, R>(sh, table[b], false);
                    cur = b;
                }
            }
            const Problem &P = BATCH ? sh.prob : a.single;
            const StepTime &tm = sh.tm;
            // fetch the next ticket while this tile runs, when another tile is
            // likely left for this block (else the atomic only adds contention)
            const bool early = !drain && t + (long long)gridDim.x < n_tickets;
            if (early && tid == 0) sh.ticket[buf ^ 1] = tbase + atomicAdd(&a.ctl->ticket, 1u);

            // ---- the new tile's physics
            bool tracked = true;  // the tile may append something
            if (!drain) {
                const ProbCounts &pc = sh.pc;
                const long long lt = t - (b > 0 ? sh.off[b - 1] : 0);  // tile within the problem
                ShortRec &rec = sh.ring.shrt[q % kRing];
                const bool lepton = lt < pc.tiles_l;
                const int sp = !lepton ? 2 : lt < pc.tiles_e ? 0 : 1;
                const long long tile = lepton ? lt : lt - pc.tiles_l;
                const int64_t first = (tile - (sp == 1 ? pc.tiles_e : 0)) * kTile;
                if (tid == 0) {
                    rec.chain = lepton ? 0 : 1;
                    rec.last = lepton ? lt == pc.tiles_l - 1 : tile == pc.tiles_g - 1;
                    rec.sp = sp;
                    rec.tile = (unsigned)tile;
                    rec.first = first;
                }
                double *const st = stash + (size_t)(q % kRing) * kStashFieldsHost * kTile;
                bool came_last;
                if (lepton) {
                    came_last = short_leptons<PREC, FK, R>(a, P, tm, sm, &sh.bar[0], lep_loaded, rec,
                                                           (q & 1u) * 32u, sp, first, pc.n[sp],
                                                           bs, st);
                } else {
                    if (!ph_loaded) {
                        wait_tables(&sh.bar[1], a);
                        ph_loaded = true;
                    }
                    came_last = short_photons<PREC, FK, R>(a, P, tm, sm.T, rec, first, pc.n[2], bs, st);
                    tracked = P.pairs != 0;  // without pairs a photon tile appends nothing
                }
                if (came_last && lane == 0) {
                    // the record's previous tile left the block at least a barrier ago
                    const int total = listed_total(rec);
                    rec.claimed = rec.resolved = 0u;
                    const int known = !lepton ? total : kHere ? *(volatile int *)&rec.made : 0;
                    rec.total = known;
                    rec.made = 0;  // for the record's next tile
                    if (!lepton || total == 0 || kHere)
                        publish_aggregate(lepton ? P.lep_words : P.pho_words, (unsigned)tile,
                                          known, epoch);
                }
            }

            // ---- the previous tile's emitters
            bool finished = false;  // this warp finished them
            if constexpr (!kHere) {
                if (q_ev != q) {
                    ShortRec &rec = sh.ring.shrt[q_ev % kRing];
                    if (rec.chain == 0)
                        finished = resolve_emitters<PREC, FK, R>(
                            a, P, tm, sm, rec, (q_ev & 1u) * 32u, drain, epoch, bs,
                            stash + (size_t)(q_ev % kRing) * kStashFieldsHost * kTile);
                }
            }

            // ---- during a problem the first warp to come here writes the
            // oldest tile of a full ring; in a round without a tile every
            // warp takes one of the tiles in flight (the last one goes to the
            // warp that finished its emitters)
            const bool due = !drain && q - q_lo == (unsigned)(kRing - 1);
            int now = -1, after = -1;
            if (due) {
                unsigned c = 0u;
                if (lane == 0) c = atomicAdd(&sh.claim, 1u);
                c = __shfl_sync(0xFFFFFFFFu, c, 0);
                if (c % (unsigned)kWarps == 0u) now = (int)(q_lo % kRing);
            } else if (drain) {
                const unsigned k = q_lo + (unsigned)warp;
                const ShortRec &r = sh.ring.shrt[k % kRing];
                if (k < q && (k != q_ev || kHere || r.chain != 0 || listed_total(r) == 0))
                    now = (int)(k % kRing);
                if (finished) after = (int)(q_ev % kRing);
            }
#pragma unroll 1
            for (;; now = after, after = -1) {
                if (now >= 0)
                    flush_short<PREC, FK, kHere>(a, P, sh.pc, sh.ring.shrt[now], tm, epoch, bs,
                                      stash + (size_t)now * kStashFieldsHost * kTile);
                if (after < 0) break;
            }
            if (!drain && !early && tid == 0)
                sh.ticket[buf ^ 1] = tbase + atomicAdd(&a.ctl->ticket, 1u);
            __syncthreads();  // this tile's lists and the next ticket are visible
            if (drain) {
                q_lo = q_ev = q;
            } else {
                if (due) ++q_lo;
                q_ev = q;
                if (tracked) ++q;
                buf ^= 1;
            }
        }
    } else if constexpr (has_long_tiles(FK)) {
        long_tile_loop<PREC, FK, BATCH>(a, table, np, tbase, epoch, stash);
        lep_loaded = ph_loaded = true;
    }

    // ---- the last block to finish publishes the step of every problem
    if (tid == 0) sh.last = last_block(a.ctl, step, n_steps);
    __syncthreads();
    if (sh.last) {
        // thread 0 acquired with its count; the other threads' reads (a
        // batch's problems) follow this fence
        if (BATCH) __threadfence();
#pragma unroll 1
        for (int b = tid; b < np; b += kTile) {
            const Problem &Q = table[b];
            if (Q.device_step && *((volatile long long *)Q.left_ctr) <= 0) continue;
            if (Q.device_step) {
                // slots this launch stepped (before the new counts are applied)
                const ProbCounts c = problem_counts(Q);
                *Q.work_ctr += c.n[0] + c.n[1] + c.n[2];
            }
            // the three counts read together, then written
            volatile long long *pend = Q.pending;
            const long long p0 = pend[0], p1 = pend[1], p2 = pend[2];
            if (sh.tl[b] > 0 && Q.sp[2].present) *Q.sp[2].n_live = p2;
            if (sh.tg[b] > 0 && Q.pairs && Q.sp[0].present && Q.sp[1].present) {
                *Q.sp[0].n_live = p0;
                *Q.sp[1].n_live = p1;
            }
            if (Q.device_step) {
                *Q.step_ctr += 1;
                *Q.left_ctr -= 1;
            }
        }
        __syncthreads();
        // every block has its first ticket: it has counted this step
        if (spread && step == 0) {
            for (int k = tid; k < kSpreadSms; k += kTile) a.ctl->sm_blocks[k] = 0u;
            if (tid < kSpreadRanks) a.ctl->rank_blocks[tid] = 0u;
            if (tid == 0) a.ctl->arrived = 0u;
        }
        if (tid == 0) end_step(a.ctl, epoch, step + 1 == n_steps);
    }
    if (BATCH || step + 1 == n_steps) break;
    if (tid == 0) sh.go = next_step(a.ctl, epoch, a.spin_limit, a.status);
    __syncthreads();
    if (!sh.go) break;  // given up: the status says so
    ++epoch;
    }
    // the copies of the tables land before the block leaves
    if (!lep_loaded) wait_tables(&sh.bar[0], a);
    if (!ph_loaded) wait_tables(&sh.bar[1], a);
}

// -------------------------------------------------------------------- fused steps
//
// K steps of every lepton in one launch, the particle held in registers
// from the first step to the last (analytic or fixed fields, pairs off: the
// leptons then never change in number and the photons only move).  The
// physics is lepton_push and lepton_events, the photon motion photon_move*: the same
// arithmetic as K launches of k_step, so the results are the same bits.
// New photons take provisional indices in arrival order (one atomic a warp
// and step) and are staged there with their order key: step, then emitter
// (tile, lane), then emission index, the slot order of K separate steps.
// The key sort (launch_fused_order) and k_fused_photons put them at those
// slots.  A tile of 32 leptons is one warp, or several of fewer lanes where
// the leptons leave the chip idle (launch_fused).

constexpr int kEmitBits = 3;
static_assert(QP_MAX_EMISSIONS <= (1 << kEmitBits), "emission index bits");

struct FusedArgs {
    StepArgs a;              // a.single: the problem at the window's first step
    int32_t K;               // steps in the window
    int32_t ob;              // bits of the emitter ordinal (tile * 32 + lane) in the key
    long long tiles_e, tiles; // lepton tiles of 32 slots (electron tiles first)
    int32_t split;           // a tile is 2^split warps of 32 / 2^split lanes
    FusedScratch fs;
    long long *win;          // [3] photons at the window start, stored and staged in it
};

// The append sink of a fused lepton: the state stays in registers, the
// emitted photons are kept for the warp's provisional indices.
struct FusedSink {
    LeptonState &cur;
    double chi_last, kx, ky, kz, ox, oy, oz;
    double gg[QP_MAX_EMISSIONS];
    unsigned what;  // 4 bits a photon: its emission
    template <int C>
    __device__ __forceinline__ void put(double v)
    {
        (&cur.x)[C] = v;
    }
    // (a species without z carries 0 along)
    __device__ __forceinline__ bool has_z() const { return true; }
    __device__ __forceinline__ void tables() {}
    __device__ __forceinline__ void chi(double c) { chi_last = c; }
    __device__ __forceinline__ void direction(double x, double y, double z)
    {
        kx = x;
        ky = y;
        kz = z;
    }
    __device__ __forceinline__ void photon(int j, double g, int k)
    {
        gg[j] = g;
        what |= (unsigned)k << (4 * j);
    }
    __device__ __forceinline__ void origin(double x, double y, double z)
    {
        ox = x;
        oy = y;
        oz = z;
    }
};

static_assert(offsetof(LeptonState, tau) == 6 * sizeof(double), "LeptonState layout");

// One warp a block, at most 64 registers a thread (32 resident warps an SM).
template <int PREC, int FK>
__global__ void __launch_bounds__(32, 32) k_fused(const __grid_constant__ FusedArgs f)
{
    using R = typename std::conditional<PREC == kFP64, double, float>::type;
    __shared__ __align__(16) Problem sP;
    __shared__ StepTime tm;
    const int lane = threadIdx.x;
    const StepArgs &a = f.a;
    const R *H, *G;
    if constexpr (PREC == kFP64) {
        H = a.tab.H;
        G = a.tab.Gs;
    } else {
        H = a.tab.Hf;
        G = a.tab.Gsf;
    }
    // photons at the window start; new photons are staged up to the capacity
    // (the key order decides which of them the free slots keep), the rest
    // dropped here
    long long stage_cap = 0;
    {
        const SpeciesDev &Ph = a.single.sp[2];
        long long base = 0;
        if (Ph.present) {
            base = *((volatile long long *)Ph.n_live);
            if (base < 0 || base > Ph.cap) {
                if (lane == 0 && blockIdx.x == 0) raise_status(a.status, QP_ERR_INVALID_ARG);
                base = base < 0 ? 0 : Ph.cap;
            }
            stage_cap = Ph.cap;
        }
        if (blockIdx.x == 0 && lane == 0) f.win[0] = base;
    }
    const int lanes = 32 >> f.split;
    for (long long t = blockIdx.x; t < f.tiles << f.split; t += gridDim.x) {
        const long long tile = t >> f.split;
        const int first_lane = lanes * (int)(t & ((1 << f.split) - 1));
        {
            const int *src = reinterpret_cast<const int *>(&a.single);
            int *dst = reinterpret_cast<int *>(&sP);
            for (int k = lane; k < (int)(sizeof(Problem) / sizeof(int)); k += 32) dst[k] = src[k];
            if (lane == 0) set_time<PREC, FK>(tm, a.single, (long long)a.single.step);
        }
        __syncwarp();
        const int sp = tile < f.tiles_e ? 0 : 1;
        const SpeciesDev &S = sP.sp[sp];
        const int64_t i = (tile - (sp ? f.tiles_e : 0)) * 32 + first_lane + lane;
        long long n = *((volatile long long *)S.n_live);
        if (n < 0 || n > S.cap) {
            if (lane == 0) raise_status(a.status, QP_ERR_INVALID_ARG);
            n = n < 0 ? 0 : S.cap;
        }
        const bool active = lane < lanes && i < n;
        LeptonState cur{};
        double w = 0.0;
        if (active) {
            cur = {S.x[i], S.y[i], S.z ? S.z[i] : 0.0, S.ux[i], S.uy[i], S.uz[i], S.tau[i]};
            w = S.w[i];
        }
        const unsigned long long ordinal = (unsigned long long)(tile * 32 + first_lane + lane)
                                           << kEmitBits;
        const uint64_t s0 = sP.step;
        unsigned c_emit = 0, c_sub = 0, c_cont = 0, c_sat = 0, c_clamp = 0, c_ph = 0, c_drop = 0;
        double e_sub = 0.0, e_drop = 0.0, chi_last = 0.0;
        for (int k = 0; k < f.K; ++k) {
            if (k > 0) {
                __syncwarp();
                if (lane == 0) set_time<PREC, FK>(tm, sP, (long long)(s0 + k));
                __syncwarp();
            }
            LeptonOut o{};
            FusedSink sink{cur};
            if (active) {
                const LeptonState in = cur;
                LeptonMid<R> mid;
                if (lepton_push<PREC, FK, R>(a, sP, tm, H, G, sp, in, mid, o, sink))
                    lepton_events<PREC, FK, R>(a, sP, tm, H, sp, S, i, in, mid, o, sink);
                else
                    lepton_finish<PREC, R>(sP, in, mid, sink);
                chi_last = sink.chi_last;
            }
            // provisional indices: the warp's total from one atomic, the
            // lanes in order after it
            int inc = o.nph;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int y = __shfl_up_sync(0xFFFFFFFFu, inc, d);
                if (lane >= d) inc += y;
            }
            const int tot = __shfl_sync(0xFFFFFFFFu, inc, 31);
            if (tot) {
                unsigned long long first = 0ull;
                if (lane == 31)
                    first = atomicAdd((unsigned long long *)f.fs.alloc, (unsigned long long)tot);
                first = __shfl_sync(0xFFFFFFFFu, first, 31) + (unsigned long long)(inc - o.nph);
                const unsigned long long kkey =
                    ((unsigned long long)k << (f.ob + kEmitBits)) | ordinal;
                for (int j = 0; j < o.nph; ++j) {
                    const long long pa = (long long)first + j;
                    const double g = sink.gg[j];
                    if (pa < stage_cap) {
                        f.fs.stage[0][pa] = sink.ox;
                        f.fs.stage[1][pa] = sink.oy;
                        f.fs.stage[2][pa] = sink.oz;
                        f.fs.stage[3][pa] = g * sink.kx;
                        f.fs.stage[4][pa] = g * sink.ky;
                        f.fs.stage[5][pa] = g * sink.kz;
                        f.fs.stage[6][pa] =
                            photon_depth<PREC>(sP, tm, sp, i, (int)(sink.what >> (4 * j) & 15u));
                        f.fs.stage[7][pa] = w;
                        f.fs.rkeys[pa] = kkey | (unsigned long long)j;
                        f.fs.moves_new[pa] = (unsigned short)(f.K - 1 - k);
                        ++c_ph;
                    } else {
                        ++c_drop;
                        e_drop += w * g;
                    }
                }
            }
            c_emit += (unsigned)o.n_emit;
            c_sub += (unsigned)o.n_sub;
            if (o.n_sub) e_sub += w * o.e_sub;
            c_cont += o.cont;
            c_sat += o.sat;
            c_clamp += o.clamped;
        }
        if (active) {
            S.x[i] = cur.x;
            S.y[i] = cur.y;
            if (S.z) S.z[i] = cur.z;
            S.ux[i] = cur.ux;
            S.uy[i] = cur.uy;
            S.uz[i] = cur.uz;
            S.tau[i] = cur.tau;
            if (S.chi) S.chi[i] = chi_last;
            if (c_emit && S.nemit) S.nemit[i] += (int)c_emit;
        }
        const unsigned t_emit = __reduce_add_sync(0xFFFFFFFFu, c_emit);
        const unsigned t_sub = __reduce_add_sync(0xFFFFFFFFu, c_sub);
        const unsigned t_cont = __reduce_add_sync(0xFFFFFFFFu, c_cont);
        const unsigned t_sat = __reduce_add_sync(0xFFFFFFFFu, c_sat);
        const unsigned t_clamp = __reduce_add_sync(0xFFFFFFFFu, c_clamp);
        const unsigned t_ph = __reduce_add_sync(0xFFFFFFFFu, c_ph);
        const unsigned t_drop = __reduce_add_sync(0xFFFFFFFFu, c_drop);
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            e_sub += __shfl_xor_sync(0xFFFFFFFFu, e_sub, d);
            e_drop += __shfl_xor_sync(0xFFFFFFFFu, e_drop, d);
        }
        if (lane == 0) {
            DevStats &st = a.stats[S.slot_stats];
            if (t_emit) atomicAdd(&st.n_emit, (unsigned long long)t_emit);
            if (t_sub) atomicAdd(&st.n_subthreshold, (unsigned long long)t_sub);
            if (t_cont) atomicAdd(&st.n_continuous, (unsigned long long)t_cont);
            if (t_sat) atomicAdd(&st.n_saturated, (unsigned long long)t_sat);
            if (t_clamp) {
                atomicAdd(&st.n_clamped, (unsigned long long)t_clamp);
                raise_status(a.status, QP_WARN_TABLE_CLAMPED);
            }
            if (t_ph) atomicAdd(&st.n_photon, (unsigned long long)t_ph);
            if (t_drop) atomicAdd(&st.n_photon_drop, (unsigned long long)t_drop);
            if (e_sub != 0.0) atomicAdd(&st.e_subthreshold, e_sub);
            if (e_drop != 0.0) atomicAdd(&st.e_dropped, e_drop);
        }
        __syncwarp();
    }
}

// The photons of the window moved ballistically: those that existed at its
// start over its K steps in place (decayed ones, tau < 0, stay), the new
// ones gathered from the staging in key order into the slots after them and
// moved over the steps left after the step that emitted them.  One thread
// a slot; the new live count.  Launched for any photon capacity > 0.
template <int PREC>
__global__ void __launch_bounds__(256) k_fused_photons(const __grid_constant__ FusedArgs f)
{
    const Problem &P = f.a.single;
    const SpeciesDev &Ph = P.sp[2];
    const long long base = f.win[0], n = base + f.win[1];
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        int moves;
        double x, y, z, ux, uy, uz, tau;
        long long pa = -1;
        if (i < base) {
            moves = f.K;
            tau = Ph.tau[i];
            if (!(tau >= 0.0)) continue;
            x = Ph.x[i];
            y = Ph.y[i];
            z = Ph.z ? Ph.z[i] : 0.0;
            ux = Ph.ux[i];
            uy = Ph.uy[i];
            uz = Ph.uz[i];
        } else {
            pa = f.fs.order[i - base];
            moves = f.fs.moves_new[pa];
            x = f.fs.stage[0][pa];
            y = f.fs.stage[1][pa];
            z = f.fs.stage[2][pa];
            ux = f.fs.stage[3][pa];
            uy = f.fs.stage[4][pa];
            uz = f.fs.stage[5][pa];
            tau = f.fs.stage[6][pa];
        }
        if (moves > 0 && tau >= 0.0) {
            if constexpr (PREC == kFP64) {
                const double u2 = photon_u64(ux, uy, uz);
                if (u2 > 0.0) {
                    const double ig = rsqrt64(u2);
                    x = repeat_step(x, moves, StepProduct{P.dt, __dmul_rn(ux, ig)});
                    y = repeat_step(y, moves, StepProduct{P.dt, __dmul_rn(uy, ig)});
                    z = repeat_step(z, moves, StepProduct{P.dt, __dmul_rn(uz, ig)});
                }
            } else {
                const float fx = hi_d(ux), fy = hi_d(uy), fz = hi_d(uz);
                const float g = photon_speed32(fx, fy, fz);
                if (g > 0.0f) {
                    const float c = P.mc.dt / g;
                    x = repeat_step(x, moves, StepFloat(c * fx));
                    y = repeat_step(y, moves, StepFloat(c * fy));
                    z = repeat_step(z, moves, StepFloat(c * fz));
                }
            }
        }
        Ph.x[i] = x;
        Ph.y[i] = y;
        if (Ph.z) Ph.z[i] = z;
        if (pa >= 0) {
            Ph.ux[i] = ux;
            Ph.uy[i] = uy;
            Ph.uz[i] = uz;
            Ph.tau[i] = tau;
            Ph.w[i] = f.fs.stage[7][pa];
            if (Ph.chi) Ph.chi[i] = 0.0;
            if (Ph.nemit) Ph.nemit[i] = 0;
        }
    }
    // staged photons past the free slots: dropped, in key order, on the
    // counters of the species that emitted them
    const long long staged = f.win[2];
    for (long long r = f.win[1] + (long long)blockIdx.x * blockDim.x + threadIdx.x; r < staged;
         r += stride) {
        const long long pa = f.fs.order[r];
        const unsigned long long tile =
            (f.fs.sorted_keys[r] >> kEmitBits & ((1ull << f.ob) - 1ull)) >> 5;
        const int sp = tile < (unsigned long long)f.tiles_e ? 0 : 1;
        const double ux = f.fs.stage[3][pa], uy = f.fs.stage[4][pa], uz = f.fs.stage[5][pa];
        DevStats &st = f.a.stats[P.sp[sp].slot_stats];
        atomicAdd(&st.n_photon, (unsigned long long)-1ll);
        atomicAdd(&st.n_photon_drop, 1ull);
        atomicAdd(&st.e_dropped, f.fs.stage[7][pa] * sqrt(ux * ux + uy * uy + uz * uz));
    }
    if (blockIdx.x == 0 && threadIdx.x == 0 && Ph.present) *Ph.n_live = n;
}

template <int PREC>
const void *fused_kernel_of(int fk)
{
    switch (fk) {
    case QP_FIELD_NONE: return (const void *)k_fused<PREC, QP_FIELD_NONE>;
    case QP_FIELD_PLANE: return (const void *)k_fused<PREC, QP_FIELD_PLANE>;
    case QP_FIELD_GAUSSIAN: return (const void *)k_fused<PREC, QP_FIELD_GAUSSIAN>;
    case QP_FIELD_YEE2D: return (const void *)k_fused<PREC, QP_FIELD_YEE2D>;
    case QP_FIELD_UNIFORM_B: return (const void *)k_fused<PREC, QP_FIELD_UNIFORM_B>;
    default: return nullptr;
    }
}

template <int PREC, bool BATCH>
const void *step_kernel_of(int fk)
{
    switch (fk) {
    case QP_FIELD_NONE: return (const void *)k_step<PREC, QP_FIELD_NONE, BATCH>;
    case QP_FIELD_PLANE: return (const void *)k_step<PREC, QP_FIELD_PLANE, BATCH>;
    case QP_FIELD_GAUSSIAN: return (const void *)k_step<PREC, QP_FIELD_GAUSSIAN, BATCH>;
    case QP_FIELD_YEE2D: return (const void *)k_step<PREC, QP_FIELD_YEE2D, BATCH>;
    case QP_FIELD_UNIFORM_B: return (const void *)k_step<PREC, QP_FIELD_UNIFORM_B, BATCH>;
    default: return nullptr;
    }
}

// Dynamic shared memory of a step kernel.
template <typename R>
size_t step_smem_of(int fk)
{
    switch (fk) {
    case QP_FIELD_YEE2D: return sizeof(StepShared<QP_FIELD_YEE2D, R>);
    case QP_FIELD_PLANE:
    case QP_FIELD_GAUSSIAN: return sizeof(StepShared<QP_FIELD_PLANE, R>);
    default: return sizeof(StepShared<QP_FIELD_NONE, R>);
    }
}

}  // namespace
}  // namespace qp
