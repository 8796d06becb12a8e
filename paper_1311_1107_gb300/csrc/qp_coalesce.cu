// Compaction and coalescence of super-photons (qp_compact_photons,
// qp_coalesce_photons), and the stable sort of a species by cell
// (qp_sort_species) on the same radix sort.
//
// The paper (section 3, last paragraph) names a coalescence of super-photons
// that conserves energy and momentum on average, without an algorithm.
// Here: the live photons are grouped by (cell of a box grid, log2-energy
// bin, direction bin on the faces of a cube); a group of at least
// min_group photons becomes two photons of half its weight each, at its
// mean energy E/W, with momenta P/W +- d (d perpendicular to P, |P/W|^2 +
// |d|^2 = (E/W)^2) in the plane of P and the group's first photon, at its
// weighted mean position, with fresh optical depths.  Weight, energy and
// momentum of every group are conserved to rounding; both photons stay
// massless.  Decayed photons (tau < 0) are removed; what remains keeps its
// slot order, a merged pair in place of its group's first photon.
//
// Pipeline (one stream, every kernel over the live count read on the
// device, grids of G blocks each owning one contiguous chunk of slots):
//   k_co_prepare   roles (1 alive, 0 decayed) and group keys;
//   radix passes   stable LSD sort of (key, slot), 8 bits a pass:
//                  k_co_hist, k_co_scan_rows, k_co_scatter;
//   k_co_groups    groups (runs of one key) cut into runs of at most
//                  max_group members in slot order; runs of >= min_group
//                  listed;
//   k_co_runs      eight lanes a run: its sums, its momentum checked, roles set (2 at
//                  the first member, 0 at the others);
//   role scan      k_co_chunk_sums, k_co_scan, k_co_offsets: the
//                  output slot of every survivor in slot order;
//   k_co_kept      survivors copied to the staging arrays;
//   k_co_pairs     merged pairs computed and written to the staging arrays;
//   k_co_copy_back staging -> species, new live count.
// Group sums run in slot order, one lane a sum, with the oracle's
// operations in the oracle's order; this unit is compiled without FMA
// contraction, so keys, sums and merged momenta are the oracle's bit for
// bit (the fresh optical depths -log(xi) differ by the last bit at most).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "qp_kernels.h"

namespace qp {
namespace {

constexpr int kCoThreads = 256;
constexpr int kRadix = 256;
constexpr int kCoWarps = kCoThreads / 32;
constexpr int kRngCoalesce = 5;
// Blocks of the kernels that stride over slots or runs, over those that own a
// chunk of slots (their number is the length of a digit's row).
constexpr int kWide = 2;

struct CoParams {
    double x0, y0, z0, dx, dy, dz;
    double idx, idy, idz;  // 1/dx, 1/dy, 1/dz
    long long nx, ny, nz;
    int lb;            // log2 of energy bins per octave
    int D;             // direction bins per face axis
    double half_D;     // D / 2
    int min_group;
    int max_group;     // longest run of one group merged into one pair
    int dims;
    unsigned long long seed;
    long long step;
    unsigned long long nomerge;  // the key of photons that are not merged
    int merge;
};

__device__ __forceinline__ long long live_count(const SpeciesDev &S, int *status)
{
    long long n = *((volatile long long *)S.n_live);
    if (n < 0 || n > S.cap) {
        if (threadIdx.x == 0 && blockIdx.x == 0) raise_status(status, QP_ERR_INVALID_ARG);
        n = n < 0 ? 0 : S.cap;
    }
    return n;
}

// The chunk of block b: contiguous, a multiple of kCoThreads long.
__device__ __forceinline__ void chunk_of(long long n, long long *beg, long long *end)
{
    long long per = (n + gridDim.x - 1) / gridDim.x;
    per = (per + kCoThreads - 1) / kCoThreads * kCoThreads;
    *beg = (long long)blockIdx.x * per;
    *end = *beg + per < n ? *beg + per : n;
    if (*beg > n) *beg = n;
}

// Square root rounded to nearest of x, within a half unit of the last place
// plus 2^-50 of one: a residual correction of x times 1/sqrt(x) (Markstein),
// nine FP64 instructions for an IEEE square root's more.
__device__ __forceinline__ double sqrt_rn(double x)
{
    return x > 0.0 ? root_of(x, rsqrt64(x)) : sqrt(x);
}

// 1/x rounded to nearest: the same correction of rcp64's reciprocal, exact but
// for a mantissa of ones.  group_key's bins depend on its last bit: one unit
// more or less moves a photon on the edge of two direction bins to the other,
// and a product |u| r above 1 out of the first.  (Both checked on the host for
// FP32 seeds within 2 units: 6e7 reciprocals, and 2e7 roots with the 14000
// nearest to a tie.)
__device__ __forceinline__ double rcp_rn(double x)
{
    const unsigned long long mantissa = (unsigned long long)__double_as_longlong(x) << 12;
    if (!in_fp32_range(x) || mantissa == ~0ull << 12) return rcp64_ieee(x);
    const double r = rcp64(x);
    return fma(fma(-x, r, 1.0), r, r);
}

// The cell of one axis: the offset times the reciprocal of the cell size
// (formed on the host), rounded down by the conversion; false outside the box
// (NaN converts to the lowest integer).
__device__ __forceinline__ bool cell_of(double x, double x0, double ix, long long n, long long &c)
{
    c = __double2ll_rd((x - x0) * ix);
    return c >= 0 && c < n;
}

__device__ __forceinline__ unsigned long long abs_bits(double x)
{
    return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}

// e: the photon's energy |u| (sqrt(ux ux + uy uy + uz uz), formed by the
// caller).  Comparisons and roundings are integer instructions or
// conversions: on the narrow FP64 pipe this is 30 instructions a photon.
__device__ unsigned long long group_key(const CoParams &C, double x, double y, double z, double ux,
                                        double uy, double uz, double e)
{
    long long cx, cy, cz = 0;
    if (!cell_of(x, C.x0, C.idx, C.nx, cx) || !cell_of(y, C.y0, C.idy, C.ny, cy) ||
        (C.dims == 3 && !cell_of(z, C.z0, C.idz, C.nz, cz)))
        return C.nomerge;
    const unsigned long long eb = (unsigned long long)__double_as_longlong(e);
    const unsigned long long ex = (eb >> 52) & 0x7FFull;
    if (ex == 0ull || ex == 0x7FFull) return C.nomerge;
    const unsigned long long ebin = (ex << C.lb) | ((eb & ((1ull << 52) - 1ull)) >> (52 - C.lb));
    // the dominant axis (the first of equals), the next two in cyclic order
    const bool y_dom = abs_bits(uy) > abs_bits(ux);
    const bool z_dom = abs_bits(uz) > abs_bits(y_dom ? uy : ux);
    const double d = z_dom ? uz : y_dom ? uy : ux;
    const double p = z_dom ? ux : y_dom ? uz : uy, q = z_dom ? uy : y_dom ? ux : uz;
    const int face = 2 * (z_dom ? 2 : y_dom ? 1 : 0) + (__double2hiint(d) < 0 ? 1 : 0);
    const double r = rcp_rn(fabs(d));  // p r and q r are in [-1, 1]
    const long long D = C.D;
    const long long ia = min((long long)__double2int_rd((p * r + 1.0) * C.half_D), D - 1);
    const long long ib = min((long long)__double2int_rd((q * r + 1.0) * C.half_D), D - 1);
    const unsigned long long dbin =
        ((unsigned long long)face * (unsigned long long)D + (unsigned long long)ia) *
            (unsigned long long)D +
        (unsigned long long)ib;
    const unsigned long long cell =
        ((unsigned long long)cx * (unsigned long long)C.ny + (unsigned long long)cy) *
            (unsigned long long)C.nz +
        (unsigned long long)cz;
    const unsigned long long n_e = 2048ull << C.lb, n_d = 6ull * (unsigned long long)(D * D);
    return (cell * n_e + ebin) * n_d + dbin;
}

// ---------------------------------------------------------------- prepare

// Doubles of a photon in the merge's copy: w, |u|, ux, uy, uz, x, y, z.
constexpr int kMember = 8;

__global__ void __launch_bounds__(kCoThreads) k_co_prepare(SpeciesDev S, CoParams C,
                                                           unsigned long long *keys,
                                                           unsigned *vals, unsigned char *role,
                                                           double *members, long long *counts,
                                                           int *status)
{
    const long long n = live_count(S, status);
    if (blockIdx.x == 0 && threadIdx.x == 0) counts[0] = n;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const bool alive = S.tau[i] >= 0.0;
        role[i] = alive ? 1 : 0;
        if (C.merge) {
            unsigned long long key = C.nomerge;
            if (alive) {
                const double ux = S.ux[i], uy = S.uy[i], uz = S.uz[i];
                const double x = S.x[i], y = S.y[i], z = S.z ? S.z[i] : 0.0, w = S.w[i];
                const double e = sqrt_rn(ux * ux + uy * uy + uz * uz);
                key = group_key(C, x, y, z, ux, uy, uz, e);
                // what the runs sum, side by side: they gather it in key order
                double2 *const m = reinterpret_cast<double2 *>(members + kMember * i);
                m[0] = make_double2(w, e);
                m[1] = make_double2(ux, uy);
                m[2] = make_double2(uz, x);
                m[3] = make_double2(y, z);
            }
            keys[i] = key;
            vals[i] = (unsigned)i;
        }
    }
}

// ---------------------------------------------------------------- radix sort

__global__ void __launch_bounds__(kCoThreads) k_co_hist(const unsigned long long *keys, int shift,
                                                        unsigned *hist, const long long *counts)
{
    __shared__ unsigned h[kRadix];
    h[threadIdx.x] = 0u;
    __syncthreads();
    long long beg, end;
    chunk_of(counts[0], &beg, &end);
    for (long long i = beg + threadIdx.x; i < end; i += kCoThreads)
        atomicAdd(&h[(unsigned)(keys[i] >> shift) & 255u], 1u);
    __syncthreads();
    hist[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = h[threadIdx.x];
}

// Exclusive scan of m entries (a sum a block) in place, by one block, with the
// sum of all entries in *total.
constexpr int kScanThreads = 1024;

__global__ void __launch_bounds__(kScanThreads) k_co_scan(unsigned *v, int m, long long *total)
{
    __shared__ unsigned s_warp[32];
    __shared__ unsigned s_tile;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    unsigned carry = 0u;
    for (int base = 0; base < m; base += kScanThreads) {
        const unsigned x = base + t < m ? v[base + t] : 0u;
        unsigned inc = x;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned y = __shfl_up_sync(0xFFFFFFFFu, inc, d);
            if (lane >= d) inc += y;
        }
        if (lane == 31) s_warp[w] = inc;
        __syncthreads();
        if (w == 0) {
            const unsigned sx = s_warp[lane];
            unsigned xi = sx;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const unsigned y = __shfl_up_sync(0xFFFFFFFFu, xi, d);
                if (lane >= d) xi += y;
            }
            s_warp[lane] = xi - sx;
            if (lane == 31) s_tile = xi;
        }
        __syncthreads();
        if (base + t < m) v[base + t] = carry + s_warp[w] + (inc - x);
        carry += s_tile;
        __syncthreads();  // s_warp and s_tile are reused by the next entries
    }
    if (t == 0) *total = (long long)carry;
}

// Exclusive scan over the blocks of every digit's counts, one block a digit,
// and the digit's total (k_co_scatter adds the smaller digits' totals).  One
// block over all kRadix x 304 counts took 19 us a pass; this takes 3.
constexpr int kRowThreads = 128;

__global__ void __launch_bounds__(kRowThreads) k_co_scan_rows(unsigned *hist, int blocks,
                                                              unsigned *total)
{
    __shared__ unsigned s_w[kRowThreads / 32];
    unsigned *row = hist + (size_t)blockIdx.x * blocks;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    unsigned run = 0u;
    for (int b0 = 0; b0 < blocks; b0 += kRowThreads) {
        const unsigned v = b0 + t < blocks ? row[b0 + t] : 0u;
        unsigned inc = v;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned y = __shfl_up_sync(0xFFFFFFFFu, inc, d);
            if (lane >= d) inc += y;
        }
        if (lane == 31) s_w[warp] = inc;
        __syncthreads();
        unsigned before = 0u, all = 0u;
#pragma unroll
        for (int w = 0; w < kRowThreads / 32; ++w) {
            if (w < warp) before += s_w[w];
            all += s_w[w];
        }
        if (b0 + t < blocks) row[b0 + t] = run + before + inc - v;
        run += all;
        __syncthreads();
    }
    if (t == 0) total[blockIdx.x] = run;
}

// Stable scatter: the block walks its chunk tile by tile; within a tile an
// element's rank among equal digits is its rank in its warp (match_any)
// plus the counts of the earlier warps.
__global__ void __launch_bounds__(kCoThreads) k_co_scatter(const unsigned long long *kin,
                                                           const unsigned *vin,
                                                           unsigned long long *kout,
                                                           unsigned *vout, int shift,
                                                           const unsigned *hist,
                                                           const unsigned *total,
                                                           const long long *counts)
{
    __shared__ unsigned base[kRadix];
    __shared__ unsigned wc[kCoWarps][kRadix];
    static_assert(kRadix == kCoThreads, "one thread a digit");
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    {
        // the digits below t, over all blocks, then t's of the earlier blocks
        const unsigned v = total[t];
        unsigned inc = v;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned y = __shfl_up_sync(0xFFFFFFFFu, inc, d);
            if (lane >= d) inc += y;
        }
        if (lane == 31) wc[0][warp] = inc;
        __syncthreads();
        unsigned before = 0u;
        for (int w = 0; w < warp; ++w) before += wc[0][w];
        base[t] = before + inc - v + hist[(size_t)t * gridDim.x + blockIdx.x];
        __syncthreads();
    }
    long long beg, end;
    chunk_of(counts[0], &beg, &end);
    const unsigned lt = (1u << lane) - 1u;
    for (long long t0 = beg; t0 < end; t0 += kCoThreads) {
        for (int w = 0; w < kCoWarps; ++w) wc[w][t] = 0u;
        __syncthreads();
        const long long i = t0 + t;
        const bool ok = i < end;
        unsigned long long k = 0ull;
        unsigned v = 0u;
        if (ok) {
            k = kin[i];
            v = vin[i];
        }
        const unsigned d = ok ? (unsigned)(k >> shift) & 255u : 256u + (unsigned)lane;
        const unsigned peers = __match_any_sync(0xFFFFFFFFu, d);
        const unsigned rank = (unsigned)__popc(peers & lt);
        if (ok && rank == 0u) wc[warp][d] = (unsigned)__popc(peers);
        __syncthreads();
        // per digit: exclusive prefix over the warps, and the tile's total
        unsigned run = 0u;
        for (int w = 0; w < kCoWarps; ++w) {
            const unsigned c = wc[w][t];
            wc[w][t] = run;
            run += c;
        }
        __syncthreads();
        if (ok) {
            const unsigned pos = base[d] + wc[warp][d] + rank;
            kout[pos] = k;
            vout[pos] = v;
        }
        __syncthreads();
        base[t] += run;
        __syncthreads();
    }
}

// ---------------------------------------------------------------- groups

// A run's sums over its members, and the momentum of the first.
struct GroupSums {
    double W, E, P[3], X[3], u[3];
};

// A merged group (run [j, end) of the sorted keys) starts at j; its end.
__device__ __forceinline__ bool group_start(const unsigned long long *keys, long long j,
                                            long long n, unsigned long long nomerge,
                                            long long *end)
{
    const unsigned long long k = keys[j];
    if (k == nomerge || (j > 0 && keys[j - 1] == k)) return false;
    // the first index past j with another key (the keys are sorted): steps
    // doubling from j until one lands past the group, then bisection
    long long lo = j, step = 1;  // keys[lo] == k
    long long hi = n;            // keys[hi] != k, or hi == n
    while (lo + step < n && keys[lo + step] == k) {
        lo += step;
        step <<= 1;
    }
    if (lo + step < n) hi = lo + step;
    while (hi - lo > 1) {
        const long long mid = lo + (hi - lo) / 2;
        if (keys[mid] == k)
            lo = mid;
        else
            hi = mid;
    }
    *end = hi;
    return true;
}

// Runs of the sorted keys: every group (one key) is cut into runs of at
// most max_group members in slot order; the runs of at least min_group go to
// the run list (one thread a group: it only walks the group's keys).
__global__ void __launch_bounds__(kCoThreads) k_co_groups(CoParams C,
                                                          const unsigned long long *keys,
                                                          long long *counts, uint2 *runs)
{
    const long long n = counts[0];
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += stride) {
        long long end;
        if (!group_start(keys, j, n, C.nomerge, &end)) continue;
        for (long long a = j; a < end; a += C.max_group) {
            const long long b = a + C.max_group < end ? a + C.max_group : end;
            if (b - a < C.min_group) continue;
            const unsigned long long r = atomicAdd((unsigned long long *)&counts[2], 1ull);
            runs[r] = make_uint2((unsigned)a, (unsigned)b);
        }
    }
}

// Eight lanes a run, one of its eight sums each, member by member in slot
// order; the sums are kept for k_co_pairs, with the first member's momentum.
// A run whose momentum vanishes is kept as it is, the others become pairs
// (role 2 at the first member, 0 at the others).  Bound by the gather in key
// order: a member is 64 consecutive bytes of the copy that k_co_prepare
// writes, one line for its eight lanes, where the species' eight arrays were
// eight sectors of 32 bytes (4e6 photons: a lane a run over the arrays 466 us,
// eight lanes over the arrays 524, over the copy 391).
constexpr int kRunLanes = kMember;

__global__ void __launch_bounds__(kCoThreads) k_co_runs(const double *members,
                                                        const unsigned *vals, const uint2 *runs,
                                                        unsigned char *role, GroupSums *rsum,
                                                        const long long *counts,
                                                        long long *stats)
{
    static_assert(sizeof(GroupSums) == 11 * sizeof(double), "eight sums, then the momentum");
    const long long nr = counts[2];
    const int c = threadIdx.x % kRunLanes, lane = threadIdx.x & 31;
    const unsigned team = 0xFFu << (lane & 24);
    const long long stride = (long long)gridDim.x * (kCoThreads / kRunLanes);
    for (long long r = (long long)blockIdx.x * (kCoThreads / kRunLanes) + threadIdx.x / kRunLanes;
         r < nr; r += stride) {
        const uint2 run = runs[r];
        const unsigned anchor = vals[run.x];
        // lane c sums W, E, P_x, P_y, P_z, X, Y, Z: w itself, or w times its double
        // four members in flight ahead of the four being added
        auto load = [&](unsigned k, double (&v)[4]) {
#pragma unroll
            for (unsigned m = 0; m < 4; ++m)
                v[m] = k + m < run.y ? members[(size_t)kMember * vals[k + m] + c] : 0.0;
        };
        double sum = 0.0, v[4];
        load(run.x, v);
        const double first = v[0];
        for (unsigned k = run.x; k < run.y; k += 4) {
            double next[4];
            load(k + 4, next);
#pragma unroll
            for (unsigned m = 0; m < 4; ++m) {
                if (k + m >= run.y) break;
                const double w = __shfl_sync(team, v[m], 0, kRunLanes);
                sum = sum + (c == 0 ? v[m] : w * v[m]);
            }
#pragma unroll
            for (int m = 0; m < 4; ++m) v[m] = next[m];
        }
        double *const out = &rsum[r].W;
        out[c] = sum;
        if (c >= 2 && c < 5) out[6 + c] = first;
        const double px = __shfl_sync(team, sum, 2, kRunLanes);
        const double py = __shfl_sync(team, sum, 3, kRunLanes);
        const double pz = __shfl_sync(team, sum, 4, kRunLanes);
        if (!(px * px + py * py + pz * pz > 0.0)) continue;
        // the sorted run is in slot order: its first member is the anchor
        for (unsigned m = run.x + c; m < run.y; m += kRunLanes)
            role[m == run.x ? anchor : vals[m]] = m == run.x ? 2 : 0;
        if (c == 0) {
            atomicAdd((unsigned long long *)&stats[0], 1ull);
            atomicAdd((unsigned long long *)&stats[1], (unsigned long long)(run.y - run.x));
        }
    }
}

// ---------------------------------------------------------------- role scan

__global__ void __launch_bounds__(kCoThreads) k_co_chunk_sums(const unsigned char *role,
                                                              unsigned *sums,
                                                              const long long *counts)
{
    __shared__ unsigned s[kCoWarps];
    long long beg, end;
    chunk_of(counts[0], &beg, &end);
    unsigned v = 0u;
    for (long long i = beg + threadIdx.x; i < end; i += kCoThreads) v += role[i];
    v = __reduce_add_sync(0xFFFFFFFFu, v);
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned t = 0u;
        for (int w = 0; w < kCoWarps; ++w) t += s[w];
        sums[blockIdx.x] = t;
    }
}

// Output slot of every survivor: the chunk's offset plus the exclusive scan
// of the roles within the chunk, tile after tile.
__global__ void __launch_bounds__(kCoThreads) k_co_offsets(const unsigned char *role,
                                                           const unsigned *chunk_off,
                                                           unsigned *off, const long long *counts)
{
    __shared__ unsigned s_w[kCoWarps];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    long long beg, end;
    chunk_of(counts[0], &beg, &end);
    unsigned run = chunk_off[blockIdx.x];
    for (long long t0 = beg; t0 < end; t0 += kCoThreads) {
        const long long i = t0 + t;
        const unsigned v = i < end ? role[i] : 0u;
        unsigned inc = v;
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned y = __shfl_up_sync(0xFFFFFFFFu, inc, d);
            if (lane >= d) inc += y;
        }
        if (lane == 31) s_w[warp] = inc;
        __syncthreads();
        unsigned before = 0u, tot = 0u;
        for (int w = 0; w < kCoWarps; ++w) {
            if (w < warp) before += s_w[w];
            tot += s_w[w];
        }
        if (i < end) off[i] = run + before + inc - v;
        run += tot;
        __syncthreads();
    }
}

// ---------------------------------------------------------------- outputs

struct Stage {
    double *f[9];  // x y z ux uy uz tau w chi
    int *nemit;
};

__global__ void __launch_bounds__(kCoThreads) k_co_kept(SpeciesDev S, const unsigned char *role,
                                                        const unsigned *off, Stage st,
                                                        const long long *counts)
{
    const long long n = counts[0];
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        if (role[i] != 1) continue;
        const unsigned o = off[i];
        st.f[0][o] = S.x[i];
        st.f[1][o] = S.y[i];
        if (S.z) st.f[2][o] = S.z[i];
        st.f[3][o] = S.ux[i];
        st.f[4][o] = S.uy[i];
        st.f[5][o] = S.uz[i];
        st.f[6][o] = S.tau[i];
        st.f[7][o] = S.w[i];
        if (S.chi) st.f[8][o] = S.chi[i];
        if (S.nemit) st.nemit[o] = S.nemit[i];
    }
}

__global__ void __launch_bounds__(kCoThreads) k_co_pairs(SpeciesDev S, CoParams C,
                                                         const unsigned *vals, const uint2 *runs,
                                                         const unsigned char *role,
                                                         const GroupSums *rsum,
                                                         const unsigned *off, Stage st,
                                                         const long long *counts)
{
    const long long nr = counts[2];
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < nr; q += stride) {
        const uint2 run = runs[q];
        const unsigned anchor = vals[run.x];
        if (role[anchor] != 2) continue;
        const GroupSums g = rsum[q];
        const double W = g.W, iW = __drcp_rn(W);
        const double eps = quotient64(g.E, W, iW);
        const double c[3] = {quotient64(g.P[0], W, iW), quotient64(g.P[1], W, iW),
                             quotient64(g.P[2], W, iW)};
        const double c2 = c[0] * c[0] + c[1] * c[1] + c[2] * c[2];
        const double d2 = eps * eps - c2;
        const double dm = d2 > 0.0 ? sqrt_rn(d2) : 0.0;
        const double cm = sqrt_rn(c2), icm = __drcp_rn(cm);
        const double ph[3] = {quotient64(c[0], cm, icm), quotient64(c[1], cm, icm),
                              quotient64(c[2], cm, icm)};
        const double r[3] = {g.u[0], g.u[1], g.u[2]};
        const double rp = r[0] * ph[0] + r[1] * ph[1] + r[2] * ph[2];
        double v[3] = {r[0] - rp * ph[0], r[1] - rp * ph[1], r[2] - rp * ph[2]};
        double vm = sqrt_rn(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
        const double rm = sqrt_rn(r[0] * r[0] + r[1] * r[1] + r[2] * r[2]);
        if (!(vm > 1e-12 * rm)) {
            // the first photon is parallel to P: the axis least aligned with P
            int a = 0;
            if (fabs(ph[1]) < fabs(ph[a])) a = 1;
            if (fabs(ph[2]) < fabs(ph[a])) a = 2;
            const double ap = ph[a];
            v[0] = (a == 0 ? 1.0 : 0.0) - ap * ph[0];
            v[1] = (a == 1 ? 1.0 : 0.0) - ap * ph[1];
            v[2] = (a == 2 ? 1.0 : 0.0) - ap * ph[2];
            vm = sqrt_rn(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
        }
        const double ivm = __drcp_rn(vm);
        const double dv[3] = {dm * quotient64(v[0], vm, ivm), dm * quotient64(v[1], vm, ivm),
                              dm * quotient64(v[2], vm, ivm)};
        const unsigned o = off[anchor];
        const long long id = particle_id(S, anchor);
        const double X[3] = {quotient64(g.X[0], W, iW), quotient64(g.X[1], W, iW),
                             quotient64(g.X[2], W, iW)};
        for (int s = 0; s < 2; ++s) {
            const double sg = s == 0 ? 1.0 : -1.0;
            const uint4 rr = draw(C.seed, QP_PHOTON, kRngCoalesce, id, (uint64_t)C.step, s);
            st.f[0][o + s] = X[0];
            st.f[1][o + s] = X[1];
            st.f[2][o + s] = X[2];
            st.f[3][o + s] = c[0] + sg * dv[0];
            st.f[4][o + s] = c[1] + sg * dv[1];
            st.f[5][o + s] = c[2] + sg * dv[2];
            st.f[6][o + s] = -log(u53(rr.x, rr.y));
            st.f[7][o + s] = 0.5 * W;
            st.f[8][o + s] = 0.0;
            st.nemit[o + s] = 0;
        }
    }
}

__global__ void __launch_bounds__(kCoThreads) k_co_copy_back(SpeciesDev S, Stage st,
                                                             const long long *counts,
                                                             long long *stats)
{
    const long long n_after = counts[1];
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n_after;
         k += stride) {
        S.x[k] = st.f[0][k];
        S.y[k] = st.f[1][k];
        if (S.z) S.z[k] = st.f[2][k];
        S.ux[k] = st.f[3][k];
        S.uy[k] = st.f[4][k];
        S.uz[k] = st.f[5][k];
        S.tau[k] = st.f[6][k];
        S.w[k] = st.f[7][k];
        if (S.chi) S.chi[k] = st.f[8][k];
        if (S.nemit) S.nemit[k] = st.nemit[k];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        stats[2] = counts[0];
        stats[3] = n_after;
        *S.n_live = n_after;
    }
}

// ---------------------------------------------------------------- sort by cell

// Cell keys of the live slots (row-major; outside the grid: nx ny, after
// every cell) and the identity order.
__global__ void __launch_bounds__(kCoThreads) k_sort_prepare(SpeciesDev S, YeeGrid g,
                                                             double idx, double idy,
                                                             unsigned long long *keys,
                                                             unsigned *vals, long long *counts,
                                                             int *status)
{
    const long long n = live_count(S, status);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        counts[0] = n;
        counts[1] = n;
    }
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        // (the quotients' bits, without the divisions' loops: 11.7 -> 8.6 us for 131072 slots)
        const double gx = floor(quotient64(S.x[i] - g.x0, g.dx, idx));
        const double gy = floor(quotient64(S.y[i] - g.y0, g.dy, idy));
        unsigned long long key = (unsigned long long)g.nx * (unsigned long long)g.ny;
        if (gx >= 0.0 && gy >= 0.0 && gx < (double)g.nx && gy < (double)g.ny)
            key = (unsigned long long)gy * (unsigned long long)g.nx + (unsigned long long)gx;
        keys[i] = key;
        vals[i] = (unsigned)i;
    }
}

// Every array of the sorted slot k from its source slot, into the staging arrays.
__global__ void __launch_bounds__(kCoThreads) k_sort_gather(SpeciesDev S, const unsigned *vals,
                                                            Stage st, const long long *counts)
{
    const long long n = counts[0];
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += stride) {
        const unsigned i = vals[k];
        st.f[0][k] = S.x[i];
        st.f[1][k] = S.y[i];
        if (S.z) st.f[2][k] = S.z[i];
        st.f[3][k] = S.ux[i];
        st.f[4][k] = S.uy[i];
        st.f[5][k] = S.uz[i];
        st.f[6][k] = S.tau[i];
        st.f[7][k] = S.w[i];
        if (S.chi) st.f[8][k] = S.chi[i];
        if (S.nemit) st.nemit[k] = S.nemit[i];
    }
}

}  // namespace

size_t coalesce_scratch_bytes(int64_t cap, int grid)
{
    const size_t c = (size_t)(cap > 0 ? cap : 1);
    return 2 * c * 8 + 2 * c * 4 + c + c * 4 + c * 9 * 8 + c * 4 +
           ((size_t)kRadix * grid + kRadix + grid + 64) * 4 + 16 * 8 + (c / 3 + 1) * 8 +
           (c / 3 + 1) * sizeof(GroupSums) + 32 * 256;
}

namespace {

// The scratch of qp_coalesce_photons, qp_sort_species and the fused steps'
// photon order, carved in one layout (every piece 256-byte aligned).
struct CoScratch {
    unsigned long long *keys[2];
    unsigned *vals[2];
    unsigned char *role;
    unsigned *off;
    Stage stg;
    unsigned *hist, *total, *chunk;  // counts of a pass by digit and block, by digit; chunk sums
    long long *counts;
    uint2 *runs;
    GroupSums *rsum;  // the sums of each run (k_co_runs, for k_co_pairs)
};

CoScratch carve(void *scratch, int64_t cap, int grid)
{
    const size_t c = (size_t)(cap > 0 ? cap : 1);
    unsigned char *p = (unsigned char *)scratch;
    auto take = [&](size_t bytes) {
        unsigned char *q = p;
        p += (bytes + 255) / 256 * 256;
        return q;
    };
    CoScratch s;
    s.keys[0] = (unsigned long long *)take(c * 8);
    s.keys[1] = (unsigned long long *)take(c * 8);
    s.vals[0] = (unsigned *)take(c * 4);
    s.vals[1] = (unsigned *)take(c * 4);
    s.role = take(c);
    s.off = (unsigned *)take(c * 4);
    for (int f = 0; f < 9; ++f) s.stg.f[f] = (double *)take(c * 8);
    s.stg.nemit = (int *)take(c * 4);
    s.hist = (unsigned *)take((size_t)kRadix * grid * 4);
    s.total = (unsigned *)take((size_t)kRadix * 4);
    s.chunk = (unsigned *)take((size_t)grid * 4 + 64);
    s.counts = (long long *)take(16 * 8);
    s.runs = (uint2 *)take((c / 3 + 1) * sizeof(uint2));
    s.rsum = (GroupSums *)take((c / 3 + 1) * sizeof(GroupSums));
    return s;
}

// `passes` passes of the stable sort of the counts[0] (key, value) pairs in
// keys[0] and vals[0], 8 bits each from the lowest; the sorted pairs are in
// keys[r] and vals[r] of the returned r.
int radix_sort(const CoScratch &cs, int passes, int grid, cudaStream_t st)
{
    int cur = 0;
    for (int ps = 0; ps < passes; ++ps, cur ^= 1) {
        k_co_hist<<<grid, kCoThreads, 0, st>>>(cs.keys[cur], 8 * ps, cs.hist, cs.counts);
        k_co_scan_rows<<<kRadix, kRowThreads, 0, st>>>(cs.hist, grid, cs.total);
        k_co_scatter<<<grid, kCoThreads, 0, st>>>(cs.keys[cur], cs.vals[cur], cs.keys[cur ^ 1],
                                                   cs.vals[cur ^ 1], 8 * ps, cs.hist, cs.total,
                                                   cs.counts);
    }
    return cur;
}

}  // namespace

cudaError_t launch_coalesce(const SpeciesDev &S, const qp_coalesce_params *P, void *scratch,
                            int grid, long long *stats, int *status, cudaStream_t st)
{
    const CoScratch cs = carve(scratch, S.cap, grid);
    unsigned long long *const *keys = cs.keys;
    unsigned *const *vals = cs.vals;
    unsigned char *role = cs.role;
    unsigned *off = cs.off;
    const Stage stg = cs.stg;
    unsigned *chunk = cs.chunk;
    long long *counts = cs.counts;
    uint2 *runs = cs.runs;
    // the merge's copy of the photons (k_co_prepare to k_co_runs) takes the
    // place of the staging arrays, which k_co_kept and k_co_pairs write after
    static_assert(kMember <= 9, "the copy fits the nine staging arrays");
    double *members = stg.f[0];

    CoParams C{};
    int passes = 0;
    if (P) {
        C.x0 = P->x0;
        C.y0 = P->y0;
        C.z0 = P->z0;
        C.dx = P->dx;
        C.dy = P->dy;
        C.dz = P->dz;
        C.idx = 1.0 / P->dx;
        C.idy = 1.0 / P->dy;
        C.idz = P->dz > 0.0 ? 1.0 / P->dz : 0.0;  // used with dims 3 only
        C.nx = P->nx;
        C.ny = P->ny;
        C.nz = P->nz;
        int lb = 0;
        while ((1 << lb) < P->energy_bins_per_octave) ++lb;
        C.lb = lb;
        C.D = P->direction_bins;
        C.half_D = 0.5 * C.D;
        C.min_group = P->min_group;
        C.max_group = P->max_group > 0 ? P->max_group : 256;
        C.dims = S.z ? 3 : 2;
        C.seed = P->seed;
        C.step = P->step;
        C.merge = 1;
        const unsigned long long n_e = 2048ull << lb;
        const unsigned long long n_d = 6ull * (unsigned long long)C.D * (unsigned long long)C.D;
        C.nomerge = (unsigned long long)P->nx * (unsigned long long)P->ny *
                    (unsigned long long)P->nz * n_e * n_d;
        int bits = 0;
        while (bits < 64 && (C.nomerge >> bits) != 0ull) ++bits;
        passes = (bits + 7) / 8;
    }
    cudaError_t e = cudaMemsetAsync(counts, 0, 16 * 8, st);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(stats, 0, 4 * 8, st);
    if (e != cudaSuccess) return e;
    k_co_prepare<<<kWide * grid, kCoThreads, 0, st>>>(S, C, keys[0], vals[0], role, members, counts,
                                                          status);
    const int cur = radix_sort(cs, passes, grid, st);
    if (passes) {
        k_co_groups<<<kWide * grid, kCoThreads, 0, st>>>(C, keys[cur], counts, runs);
        k_co_runs<<<kWide * grid, kCoThreads, 0, st>>>(members, vals[cur], runs, role, cs.rsum, counts,
                                                stats);
    }
    k_co_chunk_sums<<<grid, kCoThreads, 0, st>>>(role, chunk, counts);
    k_co_scan<<<1, kScanThreads, 0, st>>>(chunk, grid, counts + 1);
    k_co_offsets<<<grid, kCoThreads, 0, st>>>(role, chunk, off, counts);
    k_co_kept<<<kWide * grid, kCoThreads, 0, st>>>(S, role, off, stg, counts);
    if (passes) {
        k_co_pairs<<<kWide * grid, kCoThreads, 0, st>>>(S, C, vals[cur], runs, role, cs.rsum, off, stg,
                                                 counts);
    }
    k_co_copy_back<<<kWide * grid, kCoThreads, 0, st>>>(S, stg, counts, stats);
    return cudaGetLastError();
}

cudaError_t launch_sort_cells(const SpeciesDev &S, const YeeGrid &g, void *scratch, int grid,
                              long long *stats, int *status, cudaStream_t st)
{
    const CoScratch cs = carve(scratch, S.cap, grid);
    unsigned long long *const *keys = cs.keys;
    unsigned *const *vals = cs.vals;
    const Stage stg = cs.stg;
    long long *counts = cs.counts;
    const unsigned long long top = (unsigned long long)g.nx * (unsigned long long)g.ny;
    int bits = 0;
    while (bits < 64 && (top >> bits) != 0ull) ++bits;
    const int passes = (bits + 7) / 8;
    cudaError_t e = cudaMemsetAsync(stats, 0, 4 * 8, st);
    if (e != cudaSuccess) return e;
    k_sort_prepare<<<kWide * grid, kCoThreads, 0, st>>>(S, g, 1.0 / g.dx, 1.0 / g.dy, keys[0], vals[0], counts, status);
    const int cur = radix_sort(cs, passes, grid, st);
    k_sort_gather<<<kWide * grid, kCoThreads, 0, st>>>(S, vals[cur], stg, counts);
    k_co_copy_back<<<kWide * grid, kCoThreads, 0, st>>>(S, stg, counts, stats);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- fused photon order

namespace {

// counts[3]: photons the fused window allocated; counts[0] and win[2]:
// those it staged (the capacity bounds them), sorted next; win[1]: those it
// stores (the free slots bound them); identity order to sort.
__global__ void __launch_bounds__(kCoThreads) k_fo_prepare(SpeciesDev Ph, long long *counts,
                                                           long long *win, unsigned *vals,
                                                           int *status)
{
    const long long base = win[0];
    const long long cap = Ph.present ? Ph.cap : 0;
    const long long alloc = counts[3];
    const long long staged = alloc < cap ? alloc : cap;
    const long long stored = staged < cap - base ? staged : cap - base;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        counts[0] = staged;
        win[1] = stored;
        win[2] = staged;
        if (alloc > stored) raise_status(status, QP_WARN_BUFFER_FULL);
    }
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long a = (long long)blockIdx.x * blockDim.x + threadIdx.x; a < staged; a += stride)
        vals[a] = (unsigned)a;
}

}  // namespace

FusedScratch fused_scratch(void *scratch, int64_t photon_cap, int grid, int key_bits)
{
    const CoScratch cs = carve(scratch, photon_cap, grid);
    FusedScratch f;
    for (int c = 0; c < 8; ++c) f.stage[c] = cs.stg.f[c];
    f.rkeys = cs.keys[0];
    f.moves_new = (unsigned short *)cs.off;
    f.alloc = cs.counts + 3;
    f.order = cs.vals[((key_bits + 7) / 8) & 1];
    f.sorted_keys = cs.keys[((key_bits + 7) / 8) & 1];
    return f;
}

cudaError_t launch_fused_order(const SpeciesDev &Ph, void *scratch, int grid, int key_bits,
                               long long *win, int *status, cudaStream_t st)
{
    const CoScratch cs = carve(scratch, Ph.present ? Ph.cap : 0, grid);
    k_fo_prepare<<<kWide * grid, kCoThreads, 0, st>>>(Ph, cs.counts, win, cs.vals[0], status);
    radix_sort(cs, (key_bits + 7) / 8, grid, st);
    return cudaGetLastError();
}

}  // namespace qp
