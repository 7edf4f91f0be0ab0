// dat_step_pipelined: Steps 7, 9 and 12 of Algorithm A1 in ONE launch of ordinary (non-persistent)
// CTAs (and, further down, the two other forms of a step: one launch per phase, and one launch whose CTAs keep their
// pieces; see p_phases and p_resident).  Codes, integer sums and g_hat never reach memory; the gradients are read twice (for the norm, then
// for the levels), the second time from L2 only where a layer is small enough to still be there.
//
// The quantizer norm of a layer (Eq. rand_q) must be known before the first level of that layer
// (Eq. xi) can be drawn, and the two layer norms of Eq. 3 before the first parameter moves: three
// phases per layer, each needing the previous one complete for the whole layer.  The flat vector is
// cut into per-layer tiles, and the host lays three streams of tiles side by side in one list of
// work items: item s holds (at most) one tile for each phase,
//     N  sums of squares of the gradients of a tile          (gradients from HBM, L2 evict-first),
//     Q  levels, signed sum, g_hat, m', layer sums of a tile  (the same gradients once more: from L2 for
//                                                             small layers, from HBM for the others),
//     U  theta update of a tile                               (theta and m' kept in L2 with evict-last),
// where the Q stream runs behind the N stream, and the U stream behind the Q stream, by the size of
// the layer plus a fixed number of items.  A CTA takes the next item by an atomic ticket, so items
// start in list order, and does its N part first: the sums a later item waits for are produced by
// CTAs that started earlier and never wait themselves.  The last CTA to finish a layer's N (or Q)
// tiles reduces the layer's partial sums in a fixed order and publishes the layer's factors with the
// call's epoch; a Q (or U) part whose layer is not published yet polls that word, with a limit.
//
// Two-sided quantisation (Algorithm A1 Step 10) adds a fourth stream between Q and U: the Q part then
// stops at g_hat (stored, with the tile's sum of squares), the layer's last Q tile publishes
// nu^_l = ||g_hat_l||_2, and the R part of a later item draws the server's levels of its tile on the
// random stream of index M, forms the receiver's value and goes on with m' and the layer sums.
#include <algorithm>
#include <new>
#include <vector>

#include "dat_internal.cuh"

#ifndef DAT_P_THREADS
#define DAT_P_THREADS 256
#endif
#ifndef DAT_P_GROUPS                              // groups of eight consecutive elements per thread and tile
#define DAT_P_GROUPS 2
#endif
#define DAT_P_TILE (DAT_P_THREADS * 8 * DAT_P_GROUPS)   // elements per tile, tiles start on multiples of 8
#ifndef DAT_P_MINB
#define DAT_P_MINB (1024 / DAT_P_THREADS)         // 64 registers per thread
#endif
#ifndef DAT_P_LAG                                 // items between the last N tile of a layer and its first Q tile
#define DAT_P_LAG 256
#endif
#ifndef DAT_P_LAG_U                               // items between the last Q tile of a layer and its first U tile
#define DAT_P_LAG_U 512
#endif
#ifndef DAT_P_KEEP_T                              // layers of at most this many tiles: the first reads stay in L2 for the second
#define DAT_P_KEEP_T 72
#endif
#ifndef DAT_P_KEEP_TAIL                           // of a larger layer, the first reads of this many last tiles stay in L2 too
#define DAT_P_KEEP_TAIL 64
#endif
#ifndef DAT_P_REVERSE_FROM                        // layers of at least this many tiles: Q walks back from the last tile
#define DAT_P_REVERSE_FROM (DAT_P_KEEP_T + 1)
#endif
#define DAT_P_WAIT_CYCLES (4000000000ll)          // about two seconds

// which form a step takes (see p_resident, p_phases); the last one for tests: the resident form as if most of its CTAs were late
enum { P_BY_RULE = 0, P_ONE_LAUNCH = 1, P_PHASES = 2, P_RESIDENT = 3, P_RESIDENT_LATE = 4 };
enum { P_MODE_SHARED = 0, P_MODE_PER_WORKER = 1, P_MODE_IDENTITY = 2 };
enum { P_OPT_MOMENTUM = 0, P_OPT_LAMB = 1 };     // the descent direction u of Eq. 3: heavy-ball momentum, or Algorithm A2

struct PipePart {                                 // one tile of one layer; layer < 0: none
    int64_t lo, hi;                               // the layer's element range
    int32_t tb, T;                                // first tile of the layer in the partial-sum tables, tiles of the layer
    int32_t layer, tile;
};
struct PipeItem {
    PipePart n, q, u, r;                          // r: the server's quantizer (two-sided schedules only)
};

// A contiguous range of layers as a list of its own (dat_step_host: the step range by range, as the data arrives).
struct PipeGroup {
    int64_t e0, e1;                               // elements
    int64_t first, n_items;                       // in d_group_items
};

struct PipeSchedule {
    char *mem = nullptr;                          // one device allocation, carved up
    size_t mem_bytes = 0;
    PipeItem *d_items = nullptr;                  // the three streams N, Q, U
    int64_t n_items = 0;
    PipePart *d_parts = nullptr;                  // n_tiles: every tile once, in slot order (the phases)
    PipePart *d_pieces = nullptr;                 // the half tiles that hold elements, numbered as such (tb, T, tile), then each layer's
                                                  // first once more; small problems with b < 32 only
    int64_t n_pieces = 0;
    PipeItem *d_items2 = nullptr;                 // the four streams N, Q, R, U of the two-sided step
    int64_t n_items2 = 0;
    double *d_partR = nullptr;                    // 1 per half tile
    float *d_server = nullptr;                    // 2h: S / nu^_l and nu^_l / S
    double *d_partN = nullptr;                    // n_tiles * M (with pieces twice that)
    double *d_partQ = nullptr;                    // 2 per half tile
    uint32_t *d_sync = nullptr;                   // [0] ticket, [1] abort epoch, then cntN[h], cntQ[h], readyN[h], readyQ[h], cntR[h], readyR[h] and
                                                  // claim[n_pieces], the epoch of the call in which a piece was last taken
    size_t sync_bytes = 0;
    int64_t n_tiles = 0, largest = 0;             // elements of the largest layer
    std::vector<int64_t> tile_base;               // h + 1
    std::vector<PipeGroup> groups;                // built by the first dat_step_host that goes in groups
    PipeItem *d_group_items = nullptr;
    uint32_t epoch = 0;                           // calls made so far
    int form = P_BY_RULE;                         // of the calls that leave it to the rule (test hooks)
    long long wait_cycles = DAT_P_WAIT_CYCLES;
};

struct PArgs {
    GradPtrs gp;
    PhiloxKeys keys;
    PhiloxWorkers workers;
    const PipeItem *items;
    const PipePart *parts;
    float *theta, *mom, *var;                     // var: second moment (LAMB only)
    LambConst lamb;
    double *partN, *partQ, *partR;
    uint32_t *ticket, *abort_epoch, *cntN, *cntQ, *readyN, *readyQ, *cntR, *readyR, *claim, *status;
    float *worker_norms, *scales, *qmul, *dq, *step_a;
    float *ghat, *qmul2, *dq2;                    // two-sided: g_hat / the receiver's value (d), the server's factors (h each)
    float *norms_out, *scales_out, *server_scales_out;
    int32_t *code_sum;
    long long wait_cycles;
    float S_f, SM_f, M_f, mu, wd, lr, c_l, c_u;
    uint32_t epoch, n_items, n_whole;             // n_whole: of a phase's tiles, those that a CTA takes whole
    int M, h;
    bool wide;                                    // every bulk buffer starts on a 32-byte boundary
    int64_t d, n_tiles;
};

// ---- memory access helpers ---------------------------------------------------------------------------
// Bulk data goes past L1 (another CTA of the same launch may have written it) with an L2 eviction hint.
__device__ __forceinline__ uint32_t p_ld_acquire(const uint32_t *p)
{
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void p_st_release(uint32_t *p, uint32_t v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" :: "l"(p), "r"(v) : "memory");
}
// theta / m at a layer's ragged ends: element loads from L2 (never from L1, see above)
__device__ __forceinline__ void p_load4_cg(const float *__restrict__ p, int64_t e0, int64_t lo, int64_t hi, float v[4])
{
    if (e0 >= lo && e0 + 4 <= hi) {
        const float4 f = __ldcg(reinterpret_cast<const float4 *>(p + e0));
        v[0] = f.x; v[1] = f.y; v[2] = f.z; v[3] = f.w;
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = (e0 + j >= lo && e0 + j < hi) ? __ldcg(p + e0 + j) : 0.0f;
    }
}

// Eight consecutive elements with an L2 eviction priority where the group lies inside the layer, element accesses
// (no priority) at a layer's ragged ends.
template <int EV>
__device__ __forceinline__ void p_ld8(const float *p, bool wide, int64_t e0, int64_t lo, int64_t hi, float v[8])
{
    if (e0 >= lo && e0 + 8 <= hi) {
        dat_ld8<EV>(p + e0, wide, v);
    } else {
        p_load4_cg(p, e0, lo, hi, v);
        p_load4_cg(p, e0 + 4, lo, hi, v + 4);
    }
}
template <int EV>
__device__ __forceinline__ void p_st8(float *p, bool wide, int64_t e0, int64_t lo, int64_t hi, const float v[8])
{
    if (e0 >= lo && e0 + 8 <= hi) {
        dat_st8<EV>(p + e0, wide, v);
    } else {
        dat_store4(p, e0, lo, hi, v);
        dat_store4(p, e0 + 4, lo, hi, v + 4);
    }
}

// One thread: waits until `word` carries this call's epoch.  Bounded: when the limit runs out the status
// word gets DAT_STATUS_TIMEOUT and the call's abort word is set, which ends every other wait at once.
// Returns false if the part that needs the word must be skipped.
template <int SLEEP = 128>
__device__ __forceinline__ bool p_poll(const PArgs &a, const uint32_t *word)
{
    if (p_ld_acquire(word) == a.epoch) return true;
    const long long t0 = clock64();
    for (;;) {
        __nanosleep(SLEEP);
        if (p_ld_acquire(word) == a.epoch) return true;
        if (p_ld_acquire(a.abort_epoch) == a.epoch) return false;
        if (clock64() - t0 > a.wait_cycles) {
            atomicOr(a.status, DAT_STATUS_TIMEOUT);
            p_st_release(a.abort_epoch, a.epoch);
            return false;
        }
    }
}

// Self-checking build (-DDAT_SELFCHECK): what an item says about its tiles is checked before it is used;
// a violation sets DAT_STATUS_BOUNDS and the item is skipped, nothing faults.
#ifdef DAT_SELFCHECK
#define P_CHECK(a, cond) ((cond) ? true : (atomicOr((a).status, DAT_STATUS_BOUNDS), false))
__device__ __forceinline__ bool p_part_valid(const PArgs &a, const PipePart &p)
{
    return p.layer >= 0 && p.layer < a.h && p.tile >= 0 && p.tile < p.T && p.tb >= 0 && (int64_t)p.tb + p.tile < a.n_tiles &&
           p.lo >= 0 && p.lo < p.hi && p.hi <= a.d && (p.lo & ~(int64_t)7) + (int64_t)p.tile * DAT_P_TILE < p.hi;
}
#else
#define P_CHECK(a, cond) true
#endif

__device__ __forceinline__ int64_t p_tile_begin(const PipePart &pt)
{
    return (pt.lo & ~(int64_t)7) + (int64_t)pt.tile * DAT_P_TILE;
}
__device__ __forceinline__ bool p_tile_inside(const PipePart &pt)
{
    const int64_t begin = p_tile_begin(pt);
    return begin >= pt.lo && begin + DAT_P_TILE <= pt.hi;
}

// ---- N: sums of squares of one tile, every worker ------------------------------------------------
// A tile is cut into 4M units (worker, quarter tile); warp w of W takes the units [w*4M/W, (w+1)*4M/W),
// lane j the 32-byte pieces j, j+32, ... of a unit, four pieces in flight.  Units of the same worker
// are summed per lane before the warp reduction; the structure depends on M only, so the sums are the
// same from run to run.  Leaves one sum per run of units in s_unit (zero elsewhere).
template <int EV>
__device__ __forceinline__ void p_norm_units(const PArgs &a, int64_t begin, int u0, int u1, int &run, double &acc, double *s_unit)
{
    constexpr int QUARTER = DAT_P_TILE / 4, LPU = QUARTER / 256, UPB = 4 / LPU;   // units per batch of 4 loads
    static_assert(LPU >= 1 && LPU <= 4 && UPB * LPU == 4, "quarter tiles of 256 .. 1024 elements");
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (int ub = u0; ub < u1; ub += UPB) {
        float v[4][8];
#pragma unroll
        for (int k = 0; k < UPB; ++k) {
            const int u = ub + k;
            if (u < u1) {
                const float *g = a.gp.p[u >> 2] + begin + (u & 3) * QUARTER + 8 * lane;
#pragma unroll
                for (int b = 0; b < LPU; ++b) dat_ld8<EV>(g + 256 * b, a.wide, v[k * LPU + b]);
            }
        }
#pragma unroll
        for (int k = 0; k < UPB; ++k) {
            const int u = ub + k;
            if (u < u1) {
                if ((u >> 2) != (run >> 2)) {
                    acc = dat_warp_sum(acc);
                    if (lane == 0) s_unit[run] = acc;
                    acc = 0.0;
                    run = u;
                }
#pragma unroll
                for (int b = 0; b < LPU; ++b)
#pragma unroll
                    for (int j = 0; j < 8; ++j) acc = fma((double)v[k * LPU + b][j], (double)v[k * LPU + b][j], acc);
            }
        }
    }
}

__device__ __forceinline__ void p_norm_sums(const PArgs &a, const PipePart &pt, double *s_unit)
{
    constexpr int W = DAT_P_THREADS / 32, QUARTER = DAT_P_TILE / 4;
    const int M = a.M;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int U = 4 * M;
    const int u0 = warp * U / W, u1 = (warp + 1) * U / W;
    const int64_t begin = p_tile_begin(pt);
    double acc = 0.0;
    int run = u0;
    if (p_tile_inside(pt)) {
        // A small layer's lines are still in L2 when the Q part of a later item reads them again, and so are those of
        // a larger layer's last tiles, which the Q stream (walking back from the last tile) reads first; the rest of a
        // large layer is gone by then anyway: better it leaves first than push out those lines, theta and m'.
        if (pt.T <= DAT_P_KEEP_T || pt.tile >= pt.T - DAT_P_KEEP_TAIL) p_norm_units<EV_NORMAL>(a, begin, u0, u1, run, acc, s_unit);
        else p_norm_units<EV_FIRST>(a, begin, u0, u1, run, acc, s_unit);
    } else {
#pragma unroll 1
        for (int u = u0; u < u1; ++u) {
            if ((u >> 2) != (run >> 2)) {
                acc = dat_warp_sum(acc);
                if (lane == 0) s_unit[run] = acc;
                acc = 0.0;
                run = u;
            }
            const float *__restrict__ g = a.gp.p[u >> 2];
#pragma unroll
            for (int b = 0; b < QUARTER / 128; ++b) {
                const int64_t e = begin + (u & 3) * QUARTER + 4 * lane + 128 * b;
                float t[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                if (e < pt.hi) dat_load4(g, e, pt.lo, pt.hi, t);
#pragma unroll
                for (int k = 0; k < 4; ++k) acc = fma((double)t[k], (double)t[k], acc);
            }
        }
    }
    if (u1 > u0) {
        acc = dat_warp_sum(acc);
        if (lane == 0) s_unit[run] = acc;
    }
}

// Warp 0, after the barrier that follows the N sums: writes the tile's M partial sums and counts the tile
// in.  Returns (in lane 0) whether this was the layer's last tile.
__device__ __forceinline__ bool p_norm_publish(const PArgs &a, const PipePart &pt, const double *s_unit)
{
    const int M = a.M, lane = threadIdx.x & 31;
    for (int i = lane; i < M; i += 32) {
        const double *s = s_unit + 4 * i;
        a.partN[((int64_t)pt.tb + pt.tile) * M + i] = ((s[0] + s[1]) + s[2]) + s[3];
    }
    __syncwarp();
    return lane == 0 && dat_count_in(a.cntN + pt.layer, (uint32_t)pt.T);
}

// The CTA that counted in the layer's last N tile (every thread): nu_{i,l} = sqrt(sum over the tiles),
// nu_l = max_i, and the layer's two factors, published with the call's epoch.
template <int MODE>
__device__ __forceinline__ void p_norm_finish(const PArgs &a, const PipePart &pt, float *s_norm)
{
    const int M = a.M, layer = pt.layer;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t tb = pt.tb;
    const uint32_t T = (uint32_t)pt.T;
    for (int i = warp; i < M; i += DAT_P_THREADS / 32) {
        double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
        uint32_t t = lane;
        for (; t + 96 < T; t += 128) {            // four loads in flight per lane
            const double x0 = __ldcg(a.partN + (tb + t) * M + i), x1 = __ldcg(a.partN + (tb + t + 32) * M + i);
            const double x2 = __ldcg(a.partN + (tb + t + 64) * M + i), x3 = __ldcg(a.partN + (tb + t + 96) * M + i);
            s0 += x0; s1 += x1; s2 += x2; s3 += x3;
        }
        for (; t < T; t += 32) s0 += __ldcg(a.partN + (tb + t) * M + i);
        const double s = dat_warp_sum((s0 + s1) + (s2 + s3));
        if (lane == 0) {
            const float nrm = (float)sqrt(s);
            s_norm[i] = nrm;
            a.worker_norms[(int64_t)i * a.h + layer] = nrm;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        float nu = s_norm[0];
        bool bad = !isfinite(nu);
        for (int i = 1; i < M; ++i) {
            bad |= !isfinite(s_norm[i]);
            nu = (s_norm[i] > nu) ? s_norm[i] : nu;
        }
        if (MODE == P_MODE_PER_WORKER) {
            // every worker keeps its own norm (Eq. rand_q as written): index i*h + l; nu_{i,l} itself is in worker_norms
            for (int i = 0; i < M; ++i) {
                a.qmul[(int64_t)i * a.h + layer] = dat_level_factor(s_norm[i], a.S_f, isfinite(s_norm[i]));
                if (a.scales_out) a.scales_out[(int64_t)i * a.h + layer] = s_norm[i];
            }
        } else {
            a.scales[layer] = nu;
            a.qmul[layer] = dat_level_factor(nu, a.S_f, !bad);
            a.dq[layer] = (nu == 0.0f) ? 0.0f : nu / a.SM_f;
            if (a.scales_out) a.scales_out[layer] = nu;
        }
        if (bad) atomicOr(a.status, DAT_STATUS_NONFINITE);
        a.cntN[layer] = 0u;
        p_st_release(a.readyN + layer, a.epoch);
    }
}

// ---- the layer's step length from the partial sums of theta^2 and m'^2 (Eq. 3), by the CTA that counted
// in the layer's last Q tile (every thread) ----------------------------------------------------------
// U: sums in flight per thread and quantity (the order of the additions is the same).
template <int U = 1>
__device__ __forceinline__ void p_quant_finish(const PArgs &a, const PipePart &pt, double *scratch)
{
    const int layer = pt.layer;
    const int64_t tb = pt.tb;
    const uint32_t T = (uint32_t)pt.T;
    double x = 0.0, y = 0.0;
    uint32_t t = threadIdx.x;
    if (U > 1)
        for (; t + (U - 1) * DAT_P_THREADS < T; t += U * DAT_P_THREADS) {
            double vx[U], vy[U];
#pragma unroll
            for (int k = 0; k < U; ++k) {
                vx[k] = __ldcg(a.partQ + 2 * (tb + t + k * DAT_P_THREADS));
                vy[k] = __ldcg(a.partQ + 2 * (tb + t + k * DAT_P_THREADS) + 1);
            }
#pragma unroll
            for (int k = 0; k < U; ++k) { x += vx[k]; y += vy[k]; }
        }
    for (; t < T; t += DAT_P_THREADS) {
        x += __ldcg(a.partQ + 2 * (tb + t));
        y += __ldcg(a.partQ + 2 * (tb + t) + 1);
    }
    x = dat_warp_sum(x);
    y = dat_warp_sum(y);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) { scratch[2 * (threadIdx.x >> 5)] = x; scratch[2 * (threadIdx.x >> 5) + 1] = y; }
    __syncthreads();
    if (threadIdx.x == 0) {
        x = 0.0; y = 0.0;
#pragma unroll
        for (int w = 0; w < DAT_P_THREADS / 32; ++w) { x += scratch[2 * w]; y += scratch[2 * w + 1]; }
        const float n_theta = (float)sqrt(x), n_u = (float)sqrt(y);
        const float tau = fminf(fmaxf(n_theta, a.c_l), a.c_u);
        const float ratio = (n_u == 0.0f) ? 0.0f : tau / n_u;
        a.step_a[layer] = a.lr * ratio;
        if (a.norms_out) { a.norms_out[2 * layer] = n_theta; a.norms_out[2 * layer + 1] = n_u; }
        if (!isfinite(n_theta) || !isfinite(n_u)) atomicOr(a.status, DAT_STATUS_NONFINITE);
        a.cntQ[layer] = 0u;
        p_st_release(a.readyQ + layer, a.epoch);
    }
}

// Eq. grad_agg as written, every worker on its own grid: acc = sum_i nu_{i,l} * (signed level_i), in fp32
// with one fused multiply-add per worker, ascending; the caller divides by S*M.  Levels by the scaled form (see
// qu_rows) with the worker's own S/nu_{i,l}; by the plain form of Eq. xi at a layer's ragged ends and where the scaled
// form does not apply to some worker (one path for all workers of a group: the sum is ordered).
template <bool RNG16, int UNROLL>
__device__ __noinline__ float4 p_rows_per_worker_slow4(const PArgs &a, const float2 *s_fac, int64_t e0, int64_t lo, int64_t hi)
{
    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll UNROLL
    for (int i = 0; i < a.M; ++i) {
        float v[4], u1[4];
        if (UNROLL > 1) dat_load4_masked(a.gp.p[i], e0, lo, hi, v);
        else dat_load4(a.gp.p[i], e0, lo, hi, v);
        dat_u1x4((uint64_t)e0, (uint32_t)i, a.keys, RNG16, u1);
        const float2 fac = s_fac[i];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float lf = (float)dat_level_u1(v[j], fac.x, a.S_f + 1.0f, u1[j]);
            acc[j] = __fmaf_rn(fac.y, (v[j] < 0.0f) ? -lf : lf, acc[j]);
        }
    }
    return make_float4(acc[0], acc[1], acc[2], acc[3]);
}
// A ragged group by its whole warp (see qu_rows_ragged4): a lane draws a worker's levels, every lane forms the ordered
// sums from the lanes' levels.
template <bool RNG16>
__device__ __noinline__ float4 p_rows_per_worker_ragged4(const PArgs &a, const float2 *s_fac, int64_t e0, int64_t lo, int64_t hi)
{
    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    for (int i0 = 0; i0 < a.M; i0 += 32) {
        const int i = i0 + (threadIdx.x & 31), n = min(32, a.M - i0);
        int lev[4] = {0, 0, 0, 0};
        if (i < a.M) dat_signed_levels4<RNG16>(a.gp.p[i], (uint32_t)i, a.keys, s_fac[i].x, a.S_f + 1.0f, e0, lo, hi, lev);
        __syncwarp();
        for (int k = 0; k < n; ++k) {
            const float nu = s_fac[i0 + k].y;
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[j] = __fmaf_rn(nu, (float)__shfl_sync(0xFFFFFFFFu, lev[j], k), acc[j]);
        }
    }
    return make_float4(acc[0], acc[1], acc[2], acc[3]);
}
// The group's sums for its own thread, in shared memory (a layer's first or last group, drawn before the others).
template <bool RNG16, int MODE>
__device__ __forceinline__ void p_ragged(const PArgs &a, const QuConst &qc, const float2 *s_fac, int64_t e0, int64_t lo, int64_t hi, float *s_out)
{
#pragma unroll 1
    for (int p = 0; p < 2; ++p) {
        const float4 x = MODE == P_MODE_PER_WORKER ? p_rows_per_worker_ragged4<RNG16>(a, s_fac, e0 + 4 * p, lo, hi)
                                                   : qu_rows_ragged4<RNG16>(a.gp, a.keys, qc.t, qc.two_b, a.M, e0 + 4 * p, lo, hi);
        if ((threadIdx.x & 31) == 0) { s_out[4 * p] = x.x; s_out[4 * p + 1] = x.y; s_out[4 * p + 2] = x.z; s_out[4 * p + 3] = x.w; }
    }
}
template <bool RNG16, int UNROLL>
__device__ __forceinline__ void p_rows_per_worker(const PArgs &a, const QuConst &qc, const float2 *s_fac, bool fast, int64_t e0, int64_t lo, int64_t hi, float acc[8])
{
    if (!fast) {
        const float4 x = p_rows_per_worker_slow4<RNG16, UNROLL>(a, s_fac, e0, lo, hi), y = p_rows_per_worker_slow4<RNG16, UNROLL>(a, s_fac, e0 + 4, lo, hi);
        acc[0] = x.x; acc[1] = x.y; acc[2] = x.z; acc[3] = x.w; acc[4] = y.x; acc[5] = y.y; acc[6] = y.z; acc[7] = y.w;
        return;
    }
    const PhiloxGroup<RNG16> pg = dat_philox_group<RNG16>((uint64_t)e0, a.keys);
#pragma unroll 2
    for (int i = 0; i < a.M; ++i) {
        float v[8];
        dat_ld8<EV_FIRST>(a.gp.p[i] + e0, a.wide, v);
        const float2 fac = s_fac[i];                // S/nu_{i,l} and nu_{i,l}
        const float ts = fac.x * qc.inv_two_b;
        uint32_t w[8];
        dat_group_words<RNG16>(pg, a.workers.w[i], a.keys, w);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float ys = __saturatef(__fmaf_rn(fabsf(v[j]), ts, dat_u1_scaled<RNG16>(w, j, qc.ubits)));
            const float lf = __fmaf_rz(ys, qc.two_b, 8388607.0f) - 8388608.0f;
            acc[j] = __fmaf_rn(__uint_as_float((__float_as_uint(v[j]) & 0x80000000u) | __float_as_uint(fac.y)), lf, acc[j]);
        }
    }
}

// ---- m' (or m', v') and the layer sums of Eq. 3, pass 1, for one thread's group of eight elements whose
// g_hat is in registers: theta and m are loaded only now (registers limit the resident warps here).
template <int OPT>
__device__ __forceinline__ void p_direction(const PArgs &a, int64_t e0, int64_t lo, int64_t hi, const float ghat[8],
                                            double &ss_theta, double &ss_u)
{
    // what the U part reads again (theta, m', v') is kept in L2 (evict-last); the old m is dead (evict-first)
    float th[8], m[8];
    p_ld8<EV_LAST>(a.theta, a.wide, e0, lo, hi, th);
    p_ld8<EV_FIRST>(a.mom, a.wide, e0, lo, hi, m);
    if (OPT == P_OPT_LAMB) {
        // Algorithm A2: both moments are stored, the direction is formed on the fly for the layer sums
        float v[8];
        p_ld8<EV_LAST>(a.var, a.wide, e0, lo, hi, v);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            m[j] = __fmaf_rn(a.lamb.beta1, m[j], __fmul_rn(a.lamb.om1, ghat[j]));
            v[j] = __fmaf_rn(a.lamb.beta2, v[j], __fmul_rn(a.lamb.om2, __fmul_rn(ghat[j], ghat[j])));
            const bool inside = (e0 + j >= lo && e0 + j < hi);
            const float u = inside ? dat_lamb_direction(a.lamb, m[j], v[j], th[j]) : 0.0f;
            ss_theta = fma((double)th[j], (double)th[j], ss_theta);
            ss_u = fma((double)u, (double)u, ss_u);
        }
        p_st8<EV_LAST>(a.var, a.wide, e0, lo, hi, v);
    } else {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            m[j] = __fmaf_rn(a.mu, m[j], __fmaf_rn(a.wd, th[j], ghat[j]));
            ss_theta = fma((double)th[j], (double)th[j], ss_theta);
            ss_u = fma((double)m[j], (double)m[j], ss_u);
        }
    }
    p_st8<EV_LAST>(a.mom, a.wide, e0, lo, hi, m);
}

// ---- Q: levels (Eq. xi), signed sum over the workers and g_hat (Eq. grad_agg), m' and the layer sums
// (Eq. 3, pass 1) of one tile; codes, sums and g_hat stay in registers.  Leaves the tile's two sums per
// warp in scratch[2w], scratch[2w + 1].  TWO (Algorithm A1 Step 10 follows): stops at g_hat, which is
// stored, and leaves the tile's sum of g_hat^2 per warp in scratch[2w]. ----------------------------
// G: groups of eight per thread, from the tile's piece `piece` on (G = 2: the whole tile, piece 0; G = 1: half a tile; with
// G = 2 a call may ask for one group: half a tile too).
// ENDS: the groups at the layer's two ends by whole warps.  One or two workers are drawn sooner by the group's own lane than
// handed out (own lane / warp, by phases: 1.5 million elements in 300 layers, M = 1, 26.1 / 27.2 us, M = 2, 30.8 / 32.6, M = 3,
// 34.5 / 34.9, M = 4, 39.3 / 38.1, M = 5, 43.9 / 41.3): half tiles leave it to the number, whole tiles have a kernel without the
// warps' code, beside which 64 registers are tight (16 million elements, M = 1, 108.3 / 106.7 us, two-sided 149.6 / 147.0, M = 2,
// 168.3 / 165.3), and the resident form always does it (there both take the same: 300 thousand in 150 layers, M = 1, 20.6 / 20.3).
enum { P_ENDS_NONE = 0, P_ENDS_ALL = 1, P_ENDS_BY_M = 2 };
#define P_ENDS_FROM 3
template <bool RNG16, int MODE, int OPT, bool TWO, int G, int ENDS>
__device__ __forceinline__ void p_part_quant(const PArgs &a, const PipePart &pt, int piece, double *scratch, float2 *s_fac, int groups = G)
{
    const int M = a.M, layer = pt.layer;
    const int64_t lo = pt.lo, hi = pt.hi;
    float t = 0.0f, f = 0.0f;
    if (MODE == P_MODE_SHARED) { t = __ldcg(a.qmul + layer); f = __ldcg(a.dq + layer); }
    const QuConst qc = dat_qu_const(t, a.S_f, a.wide);
    bool plain = dat_qu_plain<RNG16>(qc, p_tile_begin(pt), DAT_P_TILE);
    if (MODE == P_MODE_PER_WORKER) {               // S/nu and nu of every worker: the layer's, for the whole tile
        bool out = false;
        for (int i = threadIdx.x; i < M; i += DAT_P_THREADS) {
            const float ti = __ldcg(a.qmul + (int64_t)i * a.h + layer);
            s_fac[i] = make_float2(ti, __ldcg(a.worker_norms + (int64_t)i * a.h + layer));
            out |= dat_qu_plain<RNG16>(dat_qu_const(ti, a.S_f, a.wide), 0, 8);
        }
        plain |= __syncthreads_or(out);
    }
    double ss_theta = 0.0, ss_u = 0.0;
    const int64_t begin = p_tile_begin(pt) + (int64_t)piece * (8 * DAT_P_THREADS);
    __shared__ float s_ends[ENDS ? 2 : 1][8];
    const bool ends = ENDS != P_ENDS_NONE && !plain && (ENDS == P_ENDS_ALL || M >= P_ENDS_FROM);
    if (ends && begin < hi) {
        const int64_t last = min(begin + 8 * (groups * DAT_P_THREADS - 1), (hi - 1) & ~(int64_t)7);
        if ((threadIdx.x >> 5) == 0 && (begin < lo || begin + 8 > hi)) p_ragged<RNG16, MODE>(a, qc, s_fac, begin, lo, hi, s_ends[0]);
        if ((threadIdx.x >> 5) == (unsigned)((last - begin) / 256) % (DAT_P_THREADS / 32) && last > begin && last + 8 > hi)
            p_ragged<RNG16, MODE>(a, qc, s_fac, last, lo, hi, s_ends[ENDS ? 1 : 0]);
        __syncwarp();                              // (read by a lane of the warp that drew it)
    }
#pragma unroll 1
    for (int k = 0; k < groups; ++k) {
        const int64_t e0 = begin + 8 * (int64_t)(k * DAT_P_THREADS + threadIdx.x);
        if (e0 >= hi) continue;
        const bool full = (e0 >= lo && e0 + 8 <= hi);
        float acc[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[j] = 0.0f;
        if (MODE == P_MODE_IDENTITY) {
#pragma unroll 4
            for (int i = 0; i < M; ++i) {           // Q is the identity: the ordered fp32 sum of the workers' gradients
                float v[8];
                p_ld8<EV_FIRST>(a.gp.p[i], a.wide, e0, lo, hi, v);
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[j] += v[j];
            }
        } else if (ends && !full) {
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[j] = s_ends[e0 != begin][j];
        } else if (MODE == P_MODE_PER_WORKER) p_rows_per_worker<RNG16, G == 1 ? 4 : 1>(a, qc, s_fac, full && !plain, e0, lo, hi, acc);
        else if (full && !plain) qu_rows<RNG16, G == 1 ? 4 : 2>(a.gp, a.keys, a.workers, qc, M, e0, acc);       // nearly always
        else qu_rows_slow<RNG16, G == 1 ? 4 : 1>(a.gp, a.keys, qc, M, e0, lo, hi, acc);
        if (TWO) {
            if (MODE == P_MODE_SHARED && a.code_sum) {
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (e0 + j >= lo && e0 + j < hi) a.code_sum[e0 + j] = (int)acc[j];
            }
#pragma unroll
            for (int j = 0; j < 8; ++j)
                acc[j] = (MODE == P_MODE_IDENTITY) ? acc[j] / a.M_f : (MODE == P_MODE_PER_WORKER) ? acc[j] / a.SM_f : acc[j] * f;
            p_st8<EV_LAST>(a.ghat, a.wide, e0, lo, hi, acc);   // the R part of a later item reads it again
#pragma unroll
            for (int j = 0; j < 8; ++j) ss_theta = fma((double)acc[j], (double)acc[j], ss_theta);
            continue;
        }
        // theta and m only now: registers are what limits the number of resident warps here.  (The same
        // arithmetic as p_direction, spelled out so that the loads are issued before g_hat is scaled: the step
        // is 3 % slower with the call.)
        float th[8], m[8];
        p_ld8<EV_LAST>(a.theta, a.wide, e0, lo, hi, th);       // read again by the U part
        p_ld8<EV_FIRST>(a.mom, a.wide, e0, lo, hi, m);         // dead
        if (MODE == P_MODE_SHARED && a.code_sum) {
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (e0 + j >= lo && e0 + j < hi) a.code_sum[e0 + j] = (int)acc[j];
        }
        if (OPT == P_OPT_LAMB) {
            // Algorithm A2: both moments are stored, the direction is formed on the fly for the layer sums
            float v[8];
            p_ld8<EV_LAST>(a.var, a.wide, e0, lo, hi, v);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float ghat = (MODE == P_MODE_IDENTITY) ? acc[j] / a.M_f : (MODE == P_MODE_PER_WORKER) ? acc[j] / a.SM_f : acc[j] * f;
                m[j] = __fmaf_rn(a.lamb.beta1, m[j], __fmul_rn(a.lamb.om1, ghat));
                v[j] = __fmaf_rn(a.lamb.beta2, v[j], __fmul_rn(a.lamb.om2, __fmul_rn(ghat, ghat)));
                const bool inside = (e0 + j >= lo && e0 + j < hi);
                const float u = inside ? dat_lamb_direction(a.lamb, m[j], v[j], th[j]) : 0.0f;
                ss_theta = fma((double)th[j], (double)th[j], ss_theta);
                ss_u = fma((double)u, (double)u, ss_u);
            }
            p_st8<EV_LAST>(a.var, a.wide, e0, lo, hi, v);
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float ghat = (MODE == P_MODE_IDENTITY) ? acc[j] / a.M_f : (MODE == P_MODE_PER_WORKER) ? acc[j] / a.SM_f : acc[j] * f;
                m[j] = __fmaf_rn(a.mu, m[j], __fmaf_rn(a.wd, th[j], ghat));
                ss_theta = fma((double)th[j], (double)th[j], ss_theta);
                ss_u = fma((double)m[j], (double)m[j], ss_u);
            }
        }
        p_st8<EV_LAST>(a.mom, a.wide, e0, lo, hi, m);          // the U part of a later item reads m' again
    }
    ss_theta = dat_warp_sum(ss_theta);
    ss_u = dat_warp_sum(ss_u);
    if ((threadIdx.x & 31) == 0) {
        scratch[2 * (threadIdx.x >> 5)] = ss_theta;
        scratch[2 * (threadIdx.x >> 5) + 1] = ss_u;
    }
}

// ---- R: Algorithm A1 Step 10 on one tile.  g_hat <- nu^_l * sign * level / S with the level of Eq. xi
// drawn on the random stream of index M (the first one no worker uses), then m' and the layer sums as in
// the Q part of the one-sided step. ------------------------------------------------------------------
template <bool RNG16, int OPT, int G>
__device__ __forceinline__ void p_part_requant(const PArgs &a, const PipePart &pt, int piece, double *scratch, int groups = G)
{
    const int64_t lo = pt.lo, hi = pt.hi;
    const float t = __ldcg(a.qmul2 + pt.layer), f = __ldcg(a.dq2 + pt.layer);
    const float two_b = a.S_f + 1.0f;
    double ss_theta = 0.0, ss_u = 0.0;
    const int64_t begin = p_tile_begin(pt) + (int64_t)piece * (8 * DAT_P_THREADS);
#pragma unroll 1
    for (int k = 0; k < groups; ++k) {
        const int64_t e0 = begin + 8 * (int64_t)(k * DAT_P_THREADS + threadIdx.x);
        if (e0 >= hi) continue;
        float v[8];
        p_ld8<EV_FIRST>(a.ghat, a.wide, e0, lo, hi, v);
        uint32_t w[8];
        if (RNG16) {
            dat_random_words((uint64_t)e0 >> 3, (uint32_t)a.M, a.keys, w);
        } else {
            dat_random_words((uint64_t)e0 >> 2, (uint32_t)a.M, a.keys, w);
            dat_random_words(((uint64_t)e0 >> 2) + 1, (uint32_t)a.M, a.keys, w + 4);
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float u1 = RNG16 ? dat_u1_from_half((j & 1) ? (w[j >> 1] >> 16) : (w[j >> 1] & 0xFFFFu)) : dat_u1_from_word(w[j]);
            const int lev = (int)dat_level_u1(v[j], t, two_b, u1);
            v[j] = (float)((v[j] < 0.0f) ? -lev : lev) * f;
        }
        p_st8<EV_FIRST>(a.ghat, a.wide, e0, lo, hi, v);        // the receiver's value
        p_direction<OPT>(a, e0, lo, hi, v, ss_theta, ss_u);
    }
    ss_theta = dat_warp_sum(ss_theta);
    ss_u = dat_warp_sum(ss_u);
    if ((threadIdx.x & 31) == 0) {
        scratch[2 * (threadIdx.x >> 5)] = ss_theta;
        scratch[2 * (threadIdx.x >> 5) + 1] = ss_u;
    }
}

// One thread: a part's sums from its warps', in index order -- the even places, and both into the part's slot.
__device__ __forceinline__ double p_warps_sum(const double *scratch)
{
    double x = 0.0;
#pragma unroll
    for (int w = 0; w < DAT_P_THREADS / 32; ++w) x += scratch[2 * w];
    return x;
}
__device__ __forceinline__ void p_quant_sums(const PArgs &a, int64_t slot, const double *scratch)
{
    a.partQ[2 * slot] = p_warps_sum(scratch);
    a.partQ[2 * slot + 1] = p_warps_sum(scratch + 1);
}

// Two-sided step, one thread after the barrier that follows the Q part: the tile's sum of g_hat^2 (warps in
// index order), counted in.  Returns whether this was the layer's last tile.
__device__ __forceinline__ bool p_server_publish(const PArgs &a, const PipePart &pt, const double *scratch)
{
    a.partR[(int64_t)pt.tb + pt.tile] = p_warps_sum(scratch);
    return dat_count_in(a.cntR + pt.layer, (uint32_t)pt.T);
}

// The CTA that counted in the layer's last Q tile of a two-sided step (every thread): the server's norm
// nu^_l = ||g_hat_l||_2 from the tiles' sums in index order, and its two factors, published with the epoch.
template <int U = 1>
__device__ __forceinline__ void p_server_finish(const PArgs &a, const PipePart &pt, double *scratch)
{
    const int layer = pt.layer;
    const int64_t tb = pt.tb;
    const uint32_t T = (uint32_t)pt.T;
    double x = 0.0;
    uint32_t t = threadIdx.x;
    if (U > 1)
        for (; t + (U - 1) * DAT_P_THREADS < T; t += U * DAT_P_THREADS) {
            double v[U];
#pragma unroll
            for (int k = 0; k < U; ++k) v[k] = __ldcg(a.partR + tb + t + k * DAT_P_THREADS);
#pragma unroll
            for (int k = 0; k < U; ++k) x += v[k];
        }
    for (; t < T; t += DAT_P_THREADS) x += __ldcg(a.partR + tb + t);
    x = dat_warp_sum(x);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
        x = 0.0;
#pragma unroll
        for (int w = 0; w < DAT_P_THREADS / 32; ++w) x += scratch[w];
        const float nu = (float)sqrt(x);
        a.qmul2[layer] = (nu == 0.0f) ? 0.0f : a.S_f / nu;
        a.dq2[layer] = (nu == 0.0f) ? 0.0f : nu / a.S_f;
        if (a.server_scales_out) a.server_scales_out[layer] = nu;
        if (!isfinite(nu)) atomicOr(a.status, DAT_STATUS_NONFINITE);
        a.cntR[layer] = 0u;
        p_st_release(a.readyR + layer, a.epoch);
    }
}

// One thread, after the barrier that follows the Q part: the tile's two sums (warps in index order),
// counted in.  Returns whether this was the layer's last tile.
__device__ __forceinline__ bool p_quant_publish(const PArgs &a, const PipePart &pt, const double *scratch)
{
    p_quant_sums(a, (int64_t)pt.tb + pt.tile, scratch);
    return dat_count_in(a.cntQ + pt.layer, (uint32_t)pt.T);      // releases m' (and v', or g_hat) of the whole CTA too
}

// ---- U: theta' = theta - a_l m' (Eq. 3, pass 2) of one tile ---------------------------------------
template <int OPT, int G>
__device__ __forceinline__ void p_part_update(const PArgs &a, const PipePart &pt, int piece, int groups = G)
{
    const int64_t lo = pt.lo, hi = pt.hi;
    const float na = -__ldcg(a.step_a + pt.layer);
    const int64_t begin = p_tile_begin(pt) + (int64_t)piece * (8 * DAT_P_THREADS);
#pragma unroll
    for (int k = 0; k < G; ++k) {
        const int64_t e0 = begin + 8 * (int64_t)(k * DAT_P_THREADS + threadIdx.x);
        if (e0 >= hi || k >= groups) continue;
        float th[8], m[8];
        if (OPT == P_OPT_LAMB) {
            // the direction once more from the stored moments: the same fp32 operations give the same bits
            float v[8];
            p_ld8<EV_FIRST>(a.theta, a.wide, e0, lo, hi, th);
            p_ld8<EV_FIRST>(a.mom, a.wide, e0, lo, hi, m);
            p_ld8<EV_FIRST>(a.var, a.wide, e0, lo, hi, v);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const bool inside = (e0 + j >= lo && e0 + j < hi);
                const float u = inside ? dat_lamb_direction(a.lamb, m[j], v[j], th[j]) : 0.0f;
                th[j] = __fmaf_rn(na, u, th[j]);
            }
        } else {
            p_ld8<EV_FIRST>(a.theta, a.wide, e0, lo, hi, th);
            p_ld8<EV_FIRST>(a.mom, a.wide, e0, lo, hi, m);
#pragma unroll
            for (int j = 0; j < 8; ++j) th[j] = __fmaf_rn(na, m[j], th[j]);
        }
        p_st8<EV_FIRST>(a.theta, a.wide, e0, lo, hi, th);
    }
}

// Resident CTAs per SM: four, at 64 registers.  Without a quantizer there are fewer live values than that and only
// loads to wait for, so five (ResNet-50, M = 8, b = 32: 240 us with four, 222 with five, 218 with six, which costs 8 million
// elements, M = 16, 131 instead of 124).
template <bool RNG16, int MODE, int OPT, bool TWO>
__global__ void __launch_bounds__(DAT_P_THREADS, MODE == P_MODE_IDENTITY ? 5 : DAT_P_MINB)
k_step_pipelined(const __grid_constant__ PArgs a)
{
    __shared__ double s_unit[4 * DAT_MAX_WORKERS];
    __shared__ float s_norm[DAT_MAX_WORKERS];
    __shared__ float2 s_fac[MODE == P_MODE_PER_WORKER ? DAT_MAX_WORKERS : 1];
    __shared__ __align__(16) PipeItem s_item;
    __shared__ int s_ctl[4];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // items are taken in the order in which CTAs start, whatever order the hardware starts them in
    if (warp == 0) {
        uint32_t tk = 0;
        if (lane == 0) {
            tk = atomicAdd(a.ticket, 1u);
            if (tk == a.n_items - 1u) *a.ticket = 0u;  // every ticket of this call is out: ready for the next call
        }
        tk = __shfl_sync(0xFFFFFFFFu, tk, 0);
        if (!P_CHECK(a, tk < a.n_items)) tk = 0;
        if (lane < (int)((TWO ? sizeof(PipeItem) : 3 * sizeof(PipePart)) / 16))
            reinterpret_cast<uint4 *>(&s_item)[lane] = __ldg(reinterpret_cast<const uint4 *>(a.items + tk) + lane);
    }
    for (int u = threadIdx.x; u < 4 * a.M; u += DAT_P_THREADS) s_unit[u] = 0.0;
    __syncthreads();
    const PipePart pn = s_item.n, pq = s_item.q, pu = s_item.u;
    PipePart pm = pq;                               // the part that leaves m' and the tile's two sums of Eq. 3
#ifdef DAT_SELFCHECK
    {
        const PipePart pr = TWO ? s_item.r : pq;
        const PipePart *pp[4] = {&pn, &pq, &pu, &pr};
        bool ok = true;
        for (int k = 0; k < 4; ++k) ok = ok && (pp[k]->layer < 0 || p_part_valid(a, *pp[k]));
        if (!P_CHECK(a, ok)) return;
    }
#endif
    // The CTA meets at five barriers: item read; N sums in shared memory; (A) tile counted in and the Q part's
    // layer known to be published; Q sums in shared memory; (B) tile counted in and the U part's layer
    // published.  Between them warp 0 does the publishing and the polling.
    if (pn.layer >= 0) p_norm_sums(a, pn, s_unit);
    __syncthreads();
    if (warp == 0) {
        bool n_last = false, q_go = true;
        if (pn.layer >= 0) n_last = p_norm_publish(a, pn, s_unit);
        if (lane == 0) {
            if (pq.layer >= 0 && MODE != P_MODE_IDENTITY) q_go = p_poll(a, a.readyN + pq.layer);
            s_ctl[0] = n_last;
            s_ctl[1] = q_go;
        }
    }
    __syncthreads();                               // (A)
    if (s_ctl[0]) p_norm_finish<MODE>(a, pn, s_norm);
    bool alive = (s_ctl[1] != 0);
    // (the groups at a layer's ends by their own lanes: the wait is hidden here, and the code beside the long loop is not --
    // with whole warps ResNet-50 takes 336 us instead of 330, 1 billion parameters 13.9 ms instead of 13.7)
    if (alive && pq.layer >= 0) p_part_quant<RNG16, MODE, OPT, TWO, DAT_P_GROUPS, P_ENDS_NONE>(a, pq, 0, s_unit, s_fac);
    __syncthreads();
    if (TWO) {
        // Step 10: the tile's sum of g_hat^2 counted in; the layer's last tile publishes the server's norm;
        // then the R part of this item (a tile of an earlier layer) once that layer's norm is published
        pm = s_item.r;
        if (threadIdx.x == 0) s_ctl[2] = (alive && pq.layer >= 0) ? (int)p_server_publish(a, pq, s_unit) : 0;
        __syncthreads();
        if (s_ctl[2]) p_server_finish(a, pq, s_unit);
        if (threadIdx.x == 0) s_ctl[1] = (alive && pm.layer >= 0) ? (int)p_poll(a, a.readyR + pm.layer) : (int)alive;
        __syncthreads();
        alive = (s_ctl[1] != 0);
        if (alive && pm.layer >= 0) p_part_requant<RNG16, OPT, DAT_P_GROUPS>(a, pm, 0, s_unit);
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        bool q_last = false, u_go = alive;
        if (alive && pm.layer >= 0) q_last = p_quant_publish(a, pm, s_unit);
        if (alive && pu.layer >= 0) u_go = p_poll(a, a.readyQ + pu.layer);
        s_ctl[2] = q_last;
        s_ctl[3] = u_go;
    }
    __syncthreads();                               // (B)
    if (s_ctl[2]) p_quant_finish(a, pm, s_unit);
    if (s_ctl[3] && pu.layer >= 0) p_part_update<OPT, DAT_P_GROUPS>(a, pu, 0);
}

// ---- the step as separate launches, one per phase: N (k_sumsq), Q, R (two-sided), U ---------------------------------
// The same parts on one tile per CTA, without tickets and polls: a launch ends when the layers' results are there.  The
// next phase's CTAs are set up under the last ones of the phase before (programmatic dependent launch) and walk the tiles
// the other way, so that they find in L2 what was touched last.
__device__ __forceinline__ PipePart p_part_of(const PArgs &a, uint32_t tile)
{
    PipePart pt;
    if (!P_CHECK(a, tile < a.n_tiles)) tile = 0;
    const uint4 *src = reinterpret_cast<const uint4 *>(a.parts + tile);
    reinterpret_cast<uint4 *>(&pt)[0] = __ldg(src);
    reinterpret_cast<uint4 *>(&pt)[1] = __ldg(src + 1);
    return pt;
}
// What a CTA of a phase does: `groups` halves of a tile from `piece` on.  A phase's CTAs take whole tiles as long as those
// fill waves; the tiles of a last wave that is at most half full go by halves (a.n_whole whole ones), in half the time (see
// p_whole).
struct PhaseShare {
    PipePart pt, slot;                             // the tile; the first half as the partial sums see it, a slot per half tile
    int piece, groups;
};
template <int G>
__device__ __forceinline__ PhaseShare p_share(const PArgs &a, uint32_t cta, bool back)
{
    uint32_t tile, half = 0;
    int groups = G;
    if (G == 1) {
        tile = cta / 2;
        half = cta & 1;
    } else if (cta < a.n_whole) {
        tile = cta;
    } else {
        tile = a.n_whole + (cta - a.n_whole) / 2;
        half = (cta - a.n_whole) & 1;
        groups = 1;
    }
    if (back) tile = (uint32_t)a.n_tiles - 1u - tile;
    PhaseShare x;
    x.pt = p_part_of(a, tile);
    x.slot = x.pt;
    x.slot.tb *= 2;
    x.slot.T *= 2;
    x.slot.tile = 2 * x.slot.tile + (int)half;
    x.piece = (int)half;
    x.groups = groups;
    return x;
}
// One thread: the share's sums (of a whole tile in its first half's slot, 0 in the other), counted in by halves.  Returns
// whether it was the layer's last.
template <bool TWO>
__device__ __forceinline__ bool p_share_publish(const PArgs &a, const PhaseShare &x, const double *scratch)
{
    const int64_t slot = (int64_t)x.slot.tb + x.slot.tile;
    if (TWO) {
        a.partR[slot] = p_warps_sum(scratch);
        if (x.groups == 2) a.partR[slot + 1] = 0.0;
    } else {
        p_quant_sums(a, slot, scratch);
        if (x.groups == 2) a.partQ[2 * slot + 2] = a.partQ[2 * slot + 3] = 0.0;
    }
    return dat_count_in((TWO ? a.cntR : a.cntQ) + x.pt.layer, (uint32_t)x.slot.T, (uint32_t)x.groups);
}

// A phase ends with the largest layer's last CTA, which adds a slot per half tile: four in flight per thread (60 million
// elements in one layer, M = 1: 395 -> 387 us, two-sided 550 -> 531; eight are no better there, and 8 million, one layer half of
// them, two-sided, M = 4, take 116.1 instead of 113.6).
#define P_FINISH 4

// G = 2: whole tiles (see p_share).  G = 1: half a tile (see p_halves): twice the CTAs, and four workers' loads in flight
// per thread, which then has the registers (300 thousand elements, M = 64: 166 us with G = 2, 121 with G = 1).
template <bool RNG16, int MODE, int OPT, bool TWO, int G, int ENDS>
__global__ void __launch_bounds__(DAT_P_THREADS, G == 1 ? 3 : DAT_P_MINB)
k_phase_quant(const __grid_constant__ PArgs a)
{
    __shared__ double s_red[2 * (DAT_P_THREADS / 32)];
    __shared__ float2 s_fac[MODE == P_MODE_PER_WORKER ? DAT_MAX_WORKERS : 1];
    __shared__ bool s_last;
    const PhaseShare x = p_share<G>(a, blockIdx.x, true);
    cudaTriggerProgrammaticLaunchCompletion();
    cudaGridDependencySynchronize();
    if (!P_CHECK(a, p_part_valid(a, x.pt))) return;
    p_part_quant<RNG16, MODE, OPT, TWO, G, ENDS>(a, x.pt, x.piece, s_red, s_fac, x.groups);
    __syncthreads();
    if (threadIdx.x == 0) s_last = p_share_publish<TWO>(a, x, s_red);
    __syncthreads();
    if (!s_last) return;
    if (TWO) p_server_finish<P_FINISH>(a, x.slot, s_red);
    else p_quant_finish<P_FINISH>(a, x.slot, s_red);
}

template <bool RNG16, int OPT, int G>
__global__ void __launch_bounds__(DAT_P_THREADS, DAT_P_MINB)
k_phase_requant(const __grid_constant__ PArgs a)
{
    __shared__ double s_red[2 * (DAT_P_THREADS / 32)];
    __shared__ bool s_last;
    const PhaseShare x = p_share<G>(a, blockIdx.x, false);
    cudaTriggerProgrammaticLaunchCompletion();
    cudaGridDependencySynchronize();
    if (!P_CHECK(a, p_part_valid(a, x.pt))) return;
    p_part_requant<RNG16, OPT, G>(a, x.pt, x.piece, s_red, x.groups);
    __syncthreads();
    if (threadIdx.x == 0) s_last = p_share_publish<false>(a, x, s_red);
    __syncthreads();
    if (s_last) p_quant_finish<P_FINISH>(a, x.slot, s_red);
}

template <int OPT, bool BACK, int G>
__global__ void __launch_bounds__(DAT_P_THREADS, DAT_P_MINB)
k_phase_update(const __grid_constant__ PArgs a)
{
    const PhaseShare x = p_share<G>(a, blockIdx.x, BACK);
    cudaGridDependencySynchronize();
    if (!P_CHECK(a, p_part_valid(a, x.pt))) return;
    p_part_update<OPT, G>(a, x.pt, x.piece, x.groups);
}

#include "dat_resident.cuh"

// ---- host: the item list -----------------------------------------------------------------------------
void dat_pipe_destroy(dat_plan_t *plan)
{
    if (!plan->pipe) return;
    if (plan->pipe->mem) cudaFree(plan->pipe->mem);
    if (plan->pipe->d_group_items) cudaFree(plan->pipe->d_group_items);
    delete plan->pipe;
    plan->pipe = nullptr;
}

static size_t p_align(size_t x) { return (x + 255) / 256 * 256; }

// The items of the layers [l0, l1).
static std::vector<PipeItem> p_items(const dat_plan_t *plan, const std::vector<int64_t> &tb, int l0, int l1, bool two)
{
    const bool identity = (plan->bits == 32);
    const int h = l1 - l0;
    // layers smallest first (ties in index order): the distance between the N and the Q stream is the
    // size of the layer being worked on, so it grows slowly and the streams stay paired to the end
    std::vector<int> order((size_t)h);
    for (int l = 0; l < h; ++l) order[l] = l0 + l;
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
        return plan->offsets[x + 1] - plan->offsets[x] < plan->offsets[y + 1] - plan->offsets[y];
    });
    // slot of every tile in each of the three streams (four with the server's quantizer between Q and U)
    const PipePart nopart = {0, 1, 0, 1, -1, 0};
    const PipeItem none = {nopart, nopart, nopart, nopart};
    auto part = [&](int l, int64_t t) {
        PipePart pp = {plan->offsets[l], plan->offsets[l + 1], (int32_t)tb[l], (int32_t)(tb[l + 1] - tb[l]), l, (int32_t)t};
        return pp;
    };
    std::vector<PipeItem> items;
    items.reserve(2 * (size_t)(tb[l1] - tb[l0]) + 4096);
    auto at = [&](int64_t slot) -> PipeItem & {
        if ((int64_t)items.size() <= slot) items.resize((size_t)slot + 1, none);
        return items[(size_t)slot];
    };
    std::vector<int64_t> done_n((size_t)l1, -1 - (int64_t)DAT_P_LAG), done_q((size_t)l1, 0), done_r((size_t)l1, 0);
    int64_t slot = 0;
    if (!identity)
        for (int k = 0; k < h; ++k) {
            const int l = order[k];
            for (int64_t t = 0; t < tb[l + 1] - tb[l]; ++t) { at(slot).n = part(l, t); done_n[l] = slot++; }
        }
    slot = 0;
    for (int k = 0; k < h; ++k) {
        const int l = order[k];
        const int64_t T = tb[l + 1] - tb[l];
        slot = std::max(slot, done_n[l] + DAT_P_LAG + 1);
        // a layer that L2 cannot hold next to what streams in meanwhile is walked back from its last
        // tile (what N read last, and marked to stay, is read first); the others in N's order
        const bool reverse = T >= DAT_P_REVERSE_FROM;
        for (int64_t t = 0; t < T; ++t) { at(slot).q = part(l, reverse ? T - 1 - t : t); done_q[l] = slot++; }
    }
    if (two) {
        slot = 0;
        for (int k = 0; k < h; ++k) {
            const int l = order[k];
            slot = std::max(slot, done_q[l] + DAT_P_LAG_U + 1);
            for (int64_t t = 0; t < tb[l + 1] - tb[l]; ++t) { at(slot).r = part(l, t); done_r[l] = slot++; }
        }
    }
    slot = 0;
    for (int k = 0; k < h; ++k) {
        const int l = order[k];
        slot = std::max(slot, (two ? done_r[l] : done_q[l]) + DAT_P_LAG_U + 1);
        for (int64_t t = 0; t < tb[l + 1] - tb[l]; ++t) { at(slot).u = part(l, t); ++slot; }
    }
    return items;
}

// Called by dat_plan_create (device current).  Allocates the schedule's tables (synchronous).
int dat_pipe_build(dat_plan_t *plan)
{
    PipeSchedule *g = new (std::nothrow) PipeSchedule();
    if (!g) return DAT_ERR_NOMEM;
    plan->pipe = g;
    const int h = (int)plan->h, M = plan->M;
    const bool identity = (plan->bits == 32);
    try {
        std::vector<int64_t> tb((size_t)h + 1);
        int64_t nt = 0;
        for (int l = 0; l < h; ++l) {
            tb[l] = nt;
            g->largest = std::max(g->largest, plan->offsets[l + 1] - plan->offsets[l]);
            nt += (plan->offsets[l + 1] - (plan->offsets[l] & ~(int64_t)7) + DAT_P_TILE - 1) / DAT_P_TILE;
        }
        tb[h] = nt;
        g->n_tiles = nt;
        if (nt > ((int64_t)1 << 30)) return DAT_ERR_UNSUPPORTED;
        const std::vector<PipeItem> items = p_items(plan, tb, 0, h, false);
        const std::vector<PipeItem> items2 = identity ? std::vector<PipeItem>() : p_items(plan, tb, 0, h, true);
        g->tile_base = tb;
        g->n_items2 = (int64_t)items2.size();
        g->n_items = (int64_t)items.size();

        size_t off = 0;
        auto take = [&](size_t bytes) { size_t o = off; off = p_align(off + bytes); return o; };
        const size_t o_items = take(items.size() * sizeof(PipeItem)), o_items2 = take(items2.size() * sizeof(PipeItem));
        std::vector<PipePart> parts;
        parts.reserve((size_t)nt);
        for (int l = 0; l < h; ++l)
            for (int64_t t = 0; t < tb[l + 1] - tb[l]; ++t)
                parts.push_back(PipePart{plan->offsets[l], plan->offsets[l + 1], (int32_t)tb[l], (int32_t)(tb[l + 1] - tb[l]), l, (int32_t)t});
        const size_t o_parts = take(parts.size() * sizeof(PipePart));
        std::vector<PipePart> pieces;
        const int64_t most = std::min<int64_t>(R_MOST, (int64_t)R_CTAS * plan->sm_count);
        if (!identity && nt <= most) {
            pieces.reserve((size_t)(2 * nt + h));
            for (int l = 0; l < h; ++l) {
                const int64_t lo = plan->offsets[l], hi = plan->offsets[l + 1], n = (hi - (lo & ~(int64_t)7) + R_PIECE - 1) / R_PIECE;
                const int32_t first = (int32_t)pieces.size();
                for (int64_t t = 0; t < n; ++t) pieces.push_back(PipePart{lo, hi, first, (int32_t)n, l, (int32_t)t});
            }
        }
        if ((int64_t)pieces.size() > most) pieces.clear();
        g->n_pieces = (int64_t)pieces.size();
        for (int64_t k = 0; k < g->n_pieces; ++k) {
            const PipePart piece = pieces[(size_t)k];
            if (piece.tile == 0) pieces.push_back(piece);
        }
        const size_t o_pieces = take(pieces.size() * sizeof(PipePart));
        const size_t o_pn = take((size_t)nt * (size_t)M * (pieces.empty() ? 8 : 16)), o_pq = take((size_t)nt * 32), o_pr = take((size_t)nt * 16);
        const size_t o_server = take(2 * (size_t)h * 4);
        g->sync_bytes = (2 + 6 * (size_t)h + (size_t)g->n_pieces) * 4;
        const size_t o_sync = take(g->sync_bytes);
        g->mem_bytes = off;
        cudaError_t e;
        e = cudaMalloc((void **)&g->mem, off);
        if (e != cudaSuccess) { g->mem = nullptr; plan->last_cuda = (int)e; (void)cudaGetLastError(); return DAT_ERR_NOMEM; }
        g->d_items = (PipeItem *)(g->mem + o_items);
        g->d_items2 = (PipeItem *)(g->mem + o_items2);
        g->d_partR = (double *)(g->mem + o_pr);
        g->d_server = (float *)(g->mem + o_server);
        g->d_parts = (PipePart *)(g->mem + o_parts);
        g->d_pieces = (PipePart *)(g->mem + o_pieces);
        g->d_partN = (double *)(g->mem + o_pn);
        g->d_partQ = (double *)(g->mem + o_pq);
        g->d_sync = (uint32_t *)(g->mem + o_sync);
        e = cudaMemset(g->mem + o_pn, 0, off - o_pn);
        if (e == cudaSuccess) e = cudaMemcpy(g->d_items, items.data(), items.size() * sizeof(PipeItem), cudaMemcpyHostToDevice);
        if (e == cudaSuccess && !items2.empty())
            e = cudaMemcpy(g->d_items2, items2.data(), items2.size() * sizeof(PipeItem), cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaMemcpy(g->d_parts, parts.data(), parts.size() * sizeof(PipePart), cudaMemcpyHostToDevice);
        if (e == cudaSuccess && !pieces.empty())
            e = cudaMemcpy(g->d_pieces, pieces.data(), pieces.size() * sizeof(PipePart), cudaMemcpyHostToDevice);
        if (e != cudaSuccess) return dat_cuda_fail(plan, e);
    } catch (...) {
        return DAT_ERR_NOMEM;
    }
    return DAT_OK;
}

// The plan's layers cut into at most `most` contiguous groups of about equal size, each with a list of items of its own
// (built and uploaded by the first call; synchronous).
int dat_pipe_groups(dat_plan_t *plan, int most)
{
    PipeSchedule *g = plan->pipe;
    if (!g || !g->mem) return DAT_ERR_ARG;
    if (g->d_group_items) return DAT_OK;
    std::vector<PipeItem> all;
    try {
        g->groups.clear();
        for (int64_t l0 = 0, l1; l0 < plan->h; l0 = l1) {
            const int64_t left = most - (int64_t)g->groups.size();
            const int64_t want = plan->offsets[l0] + (plan->d - plan->offsets[l0] + left - 1) / left;
            for (l1 = l0 + 1; left > 1 && l1 < plan->h && plan->offsets[l1] < want; ++l1) {}
            if (left <= 1) l1 = plan->h;
            const std::vector<PipeItem> list = p_items(plan, g->tile_base, (int)l0, (int)l1, false);
            g->groups.push_back(PipeGroup{plan->offsets[l0], plan->offsets[l1], (int64_t)all.size(), (int64_t)list.size()});
            all.insert(all.end(), list.begin(), list.end());
        }
    } catch (...) {
        return DAT_ERR_NOMEM;
    }
    PipeItem *mem = nullptr;
    cudaError_t e = cudaMalloc((void **)&mem, all.size() * sizeof(PipeItem));
    if (e != cudaSuccess) { plan->last_cuda = (int)e; (void)cudaGetLastError(); return DAT_ERR_NOMEM; }
    e = cudaMemcpy(mem, all.data(), all.size() * sizeof(PipeItem), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) { cudaFree(mem); return dat_cuda_fail(plan, e); }
    g->d_group_items = mem;
    return DAT_OK;
}

int dat_pipe_group_count(const dat_plan_t *plan) { return (int)plan->pipe->groups.size(); }

void dat_pipe_group_range(const dat_plan_t *plan, int k, int64_t *e0, int64_t *e1)
{
    *e0 = plan->pipe->groups[(size_t)k].e0;
    *e1 = plan->pipe->groups[(size_t)k].e1;
}

// After a call that timed out the arrival counters and the ticket are left mid-way: clear them
// (enqueued on `s`; called by dat_get_status when it finds DAT_STATUS_TIMEOUT).
cudaError_t dat_pipe_reset(dat_plan_t *plan, cudaStream_t s)
{
    PipeSchedule *g = plan->pipe;
    if (!g || !g->mem) return cudaSuccess;
    return cudaMemsetAsync(g->d_sync, 0, g->sync_bytes, s);
}

// Which form a step takes (both sides measured over sizes, shares and workers; the figures here are us of the momentum step,
// b = 8, where nothing else is said).
//
// The one launch keeps its streams 256 and 512 items apart, so a small problem runs through waves of nearly empty CTAs; the
// phases have a launch's set-up and last wave each.  And the streams of the largest layer, which come last, overlap with
// nothing: where one layer has a good part of the elements the phases win at every measured size (one launch / phases; the
// largest 0.28 of 10 million elements, M = 2, 94 / 83, M = 8, 178 / 158, of 30 million 232 / 216, 463 / 433; LAMB two-sided,
// M = 3, 163 / 156, 430 / 419; 0.3 of 100 million 737 / 695, 1463 / 1447; a smaller share than 0.27 may gain too, but ResNet-18,
// 0.21, M = 6, 123 / 139, and ResNet-50, 0.09, M = 8, 309 / 358, do not).  Two-sided momentum steps of more than 24 tiles per SM
// have less to gain below 16 workers: the largest 0.28 of 30 million, M = 4, 359 / 365, 0.33: 360 / 370, 0.4: 375 / 371.
// One worker: by phases (60 million elements: 409 / 359), but two-sided momentum steps of more than 14 tiles per SM only where
// a layer is large (30 million, the largest 0.06: 235 / 256, 0.15: 247 / 257, 0.2: 256 / 259; LAMB 330 / 335, 342 / 337, 351 / 337).
// b = 32 has no norms: 1 million, M = 8, 22 / 18, but 2.8 million 28 / 34, 16 million 153 / 159.
#define P_PHASES_WAVE 4                           // tiles per SM: one wave of a phase's CTAs
#define P_PHASES_MOST 9
#define P_PHASES_SHARE 0.27                       // of the elements, in the largest layer
#define P_TWO_LARGE 24                            // tiles per SM
#define P_TWO_SHARE 0.38
#define P_TWO_LARGE_1 14                          // with one worker
#define P_TWO_SHARE_1 0.16
static bool p_phases(const dat_plan_t *plan, bool two, bool lamb)
{
    const int64_t n = plan->pipe->n_tiles, sm = plan->sm_count;
    if (n <= P_PHASES_WAVE * sm) return true;
    if (plan->bits == 32) return false;
    if (n <= P_PHASES_MOST * sm) return true;
    const double share = (double)plan->pipe->largest / (double)plan->d;
    const bool two_large = two && !lamb && n > (plan->M == 1 ? P_TWO_LARGE_1 : P_TWO_LARGE) * sm;
    if (plan->M == 1) return !two_large || share >= P_TWO_SHARE_1;
    return share >= (two_large && plan->M < 16 ? P_TWO_SHARE : P_PHASES_SHARE);
}

// The resident form: one piece of 2048 elements per CTA, up to 0.9 million elements.  Phases / resident in us, 40 odd layers:
//   elements       M = 1          4            8           16          64         two-sided: M = 4     16
//   20 thousand  16.4 / 16.4  18.5 / 16.7  18.5 / 18.5  21.6 / 22.6  47.2 / 47.3      22.8 / 21.0  26.6 / 26.7
//   150          16.4 / 16.4  18.5 / 17.1  20.5 / 18.5  26.9 / 22.6  62.1 / 51.5      23.6 / 21.7  31.8 / 26.8
//   300          16.4 / 17.8  18.5 / 18.8  22.1 / 20.2  29.8 / 24.7  70.6 / 63.0      23.9 / 23.3  35.2 / 29.9
//   850          20.4 / 20.6  24.6 / 21.1  29.3 / 23.7  39.2 / 33.0  95.1 / 94.7      30.8 / 26.8  47.1 / 39.5
// With several pieces per CTA it loses to the phases (1 million, M = 32: 70 / 85).  b = 32, two phases without norms, gains nothing.
//
// Not where a few CTAs would read many workers' gradients one after the other, which the phases' norms spread over the chip (20
// thousand elements in one layer, M = 16, 17.4 / 18.5, M = 64, 30.9 / 41.2; two-sided M = 64, 35.3 / 45.3, but M = 16, 22.5 / 20.6
// at 5 thousand); nor with so many workers on nearly all places (850 thousand in one layer, M = 64: 92.7 / 99.4); nor where one
// or two workers have hardly anything to read and most pieces end a layer (150 layers, 20 to 300 thousand elements, M = 1, 16.4 /
// 18.5 to 16.6 / 20.3, LAMB 20.5 / 22.1 to 21.3 / 22.7, two-sided 21.8 / 23.5 to 22.6 / 24.9); nor for the momentum step of two
// workers on up to half of the chip (150 thousand in 40 layers 16.4 / 17.3, 300 thousand 16.6 / 17.9).
static bool p_resident(const dat_plan_t *plan, bool two, bool lamb)
{
    const int64_t n = plan->pipe->n_pieces;
    const int M = plan->M;
    if (n == 0) return false;
    if (M >= (two ? 32 : 16) && n <= 48) return false;
    if (M >= 48 && n > 400) return false;
    if (M <= 2 && n >= 100 && n <= 2 * plan->h) return false;
    return !(M == 2 && !two && !lamb && n > 48 && n < 250);
}

// Half a tile per CTA: in one wave, and with many workers (a long loop per CTA, so that a last wave of whole tiles costs
// much: 2.5 million elements, 617 tiles, M = 32: 185 / 156 us; 4 million, M = 3: 51.1 / 53.5).
static bool p_halves(const dat_plan_t *plan)
{
    const int64_t n = plan->pipe->n_tiles, sm = plan->sm_count;
    return n <= P_PHASES_WAVE * sm || (n <= P_PHASES_MOST * sm && plan->M >= 8);
}

// The tiles that a phase's CTAs take whole, where not all go by halves: full waves of them, if the rest fits 0.4 of a wave, of LAMB
// steps half a wave.
// All whole / the rest by halves, in us, 592 CTAs a wave: 2.5 million elements in 40 odd layers, M = 1, 4, 6: 29.8 / 29.0, 41.0 / 39.8,
// 47.6 / 45.8, LAMB 47.5 / 43.2, 54.9 / 50.8, 61.9 / 56.5, two-sided 39.6 / 38.9, 51.8 / 49.5, 58.3 / 56.0; 5.2 million, LAMB, M = 4, 86.5 / 83.4.  A rest of 0.3 of a wave, M = 1, 4, 6: 27.5 / 26.7, 42.1 / 41.0,
// 51.0 / 48.8; 0.4: 28.8 / 28.5, 43.3 / 43.1, 52.9 / 51.7, two-sided 41.0 / 40.5, 56.0 / 55.5, 66.0 / 65.0; but 0.5: 29.9 / 30.7, 45.5 / 45.6, 55.2 / 55.0,
// two-sided 41.7 / 42.0, 58.8 / 59.3, 69.0 / 68.4; LAMB 45.2 / 43.6, 61.1 / 59.4, 70.3 / 67.9.
static uint32_t p_whole(const dat_plan_t *plan, bool lamb)
{
    const int64_t n = plan->pipe->n_tiles, wave = DAT_P_MINB * (int64_t)plan->sm_count, rest = n % wave;
    return (uint32_t)((lamb ? 2 * rest <= wave : 5 * rest <= 2 * wave) ? n - rest : n);
}

// A launch that may be set up while the one before it ends (its kernel waits for that end itself).
template <class K>
static cudaError_t p_launch_after(K kernel, unsigned grid, cudaStream_t s, const PArgs &a)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(DAT_P_THREADS);
    cfg.stream = s;
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, a);
}

// One launch of the step.  lamb == nullptr: the momentum direction with hp; else Algorithm A2 with *lamb.
// g_hat != nullptr: the two-sided step (Algorithm A1 Step 10 between the aggregation and the update).
static int p_launch(dat_plan_t *plan, float *theta, float *mom, float *var, const float *const *grads,
                    uint64_t seed, uint64_t step, const dat_hparams_t *hp, const LambConst *lamb, float lr, float c_l, float c_u,
                    int32_t *code_sum_out, float *layer_norms_out, float *scales_out, void *stream,
                    float *g_hat = nullptr, float *server_scales_out = nullptr, const PipeGroup *group = nullptr, int how = P_BY_RULE)
{
    if (step >> 32) return DAT_ERR_ARG;
    if (plan->elem_base || plan->worker_base) return DAT_ERR_UNSUPPORTED;     // a slice of a larger problem: separate calls only
    if (!dat_aligned16(theta) || !dat_aligned16(mom) || (var && !dat_aligned16(var)) || (code_sum_out && !dat_aligned16(code_sum_out)) ||
        (layer_norms_out && !dat_aligned16(layer_norms_out)) || (scales_out && !dat_aligned16(scales_out)) ||
        (g_hat && !dat_aligned16(g_hat)) || (server_scales_out && !dat_aligned16(server_scales_out)))
        return DAT_ERR_ALIGN;
    const bool two = (g_hat != nullptr);
    if (how != P_PHASES) {   // the call's epoch and the Philox key are launch parameters: a captured graph would replay them unchanged
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing((cudaStream_t)stream, &cap) != cudaSuccess) { (void)cudaGetLastError(); return DAT_ERR_CUDA; }
        if (cap != cudaStreamCaptureStatusNone) return DAT_ERR_UNSUPPORTED;
    }
    if (two && plan->bits == 32) return DAT_ERR_BITS;      // nothing to quantize with
    PArgs a;
    int rc = dat_check_grads(plan, grads, &a.gp);
    if (rc != DAT_OK) return rc;
    PipeSchedule *g = plan->pipe;
    if (!g || !g->mem) return DAT_ERR_ARG;
    const bool identity = (plan->bits == 32);
    const bool per_worker = !identity && plan->scale_mode == DAT_SCALE_PER_WORKER;
    const size_t h = (size_t)plan->h;
    a.keys = dat_make_keys(seed, step);
    dat_make_worker_table(a.keys, plan->M, &a.workers);
    a.wide = dat_grads_wide(plan, grads) && (((uintptr_t)theta | (uintptr_t)mom | (uintptr_t)var | (uintptr_t)g_hat) & 31u) == 0;
    a.items = group ? g->d_group_items + group->first : two ? g->d_items2 : g->d_items;
    a.parts = g->d_parts;
    a.theta = theta;
    a.mom = mom;
    a.var = var;
    if (lamb) a.lamb = *lamb;
    else a.lamb = LambConst{};
    a.partN = g->d_partN;
    a.partQ = g->d_partQ;
    a.partR = g->d_partR;
    a.ticket = g->d_sync;
    a.abort_epoch = g->d_sync + 1;
    a.cntN = g->d_sync + 2;
    a.cntQ = a.cntN + h;
    a.readyN = a.cntQ + h;
    a.readyQ = a.readyN + h;
    a.cntR = a.readyQ + h;
    a.readyR = a.cntR + h;
    a.claim = a.readyR + h;
    a.ghat = g_hat;
    a.qmul2 = g->d_server;
    a.dq2 = g->d_server + h;
    a.server_scales_out = server_scales_out;
    a.status = plan->d_status;
    a.worker_norms = plan->d_worker_norms;
    a.scales = plan->d_scales;
    a.qmul = plan->d_qmul;
    a.dq = plan->d_dq;
    a.step_a = plan->d_step_a;
    a.norms_out = layer_norms_out;
    a.scales_out = identity ? nullptr : scales_out;
    a.code_sum = (identity || per_worker) ? nullptr : code_sum_out;
    a.wait_cycles = g->wait_cycles;
    a.S_f = (float)plan->S;
    a.SM_f = (float)((uint64_t)plan->S * (uint64_t)plan->M);
    a.M_f = (float)plan->M;
    a.mu = hp ? hp->momentum : 0.0f;
    a.wd = hp ? hp->weight_decay : 0.0f;
    a.lr = lr;
    a.c_l = c_l;
    a.c_u = c_u;
    if (++g->epoch == 0u) ++g->epoch;              // 0 is what the words hold before the first call
    a.epoch = g->epoch;
    a.n_items = (uint32_t)(group ? group->n_items : two ? g->n_items2 : g->n_items);
    a.M = plan->M;
    a.h = (int)plan->h;
    a.d = plan->d;
    a.n_tiles = g->n_tiles;
    cudaStream_t s = (cudaStream_t)stream;
    const bool rng16 = (plan->rng_bits == 16);
    int form = group ? P_ONE_LAUNCH : how == P_BY_RULE ? g->form : how;
    if (form == P_BY_RULE) form = p_resident(plan, two, lamb != nullptr) ? P_RESIDENT : p_phases(plan, two, lamb != nullptr) ? P_PHASES : P_ONE_LAUNCH;
    if (form == P_RESIDENT || form == P_RESIDENT_LATE) {
        a.parts = form == P_RESIDENT ? g->d_pieces : g->d_pieces + g->n_pieces;
        const unsigned ctas = form == P_RESIDENT ? (unsigned)g->n_pieces : (unsigned)plan->h;
#define P_RES(R, MODE, OPT, TWO) k_step_resident<R, MODE, OPT, TWO><<<ctas, DAT_P_THREADS, 0, s>>>(a)
#define P_RES_OPT(R, MODE)                                                                                          \
    do {                                                                                                            \
        if (two) { if (lamb) P_RES(R, MODE, P_OPT_LAMB, true); else P_RES(R, MODE, P_OPT_MOMENTUM, true); }         \
        else if (lamb) P_RES(R, MODE, P_OPT_LAMB, false);                                                           \
        else P_RES(R, MODE, P_OPT_MOMENTUM, false);                                                                 \
    } while (0)
        if (per_worker && rng16) P_RES_OPT(true, P_MODE_PER_WORKER);
        else if (per_worker) P_RES_OPT(false, P_MODE_PER_WORKER);
        else if (rng16) P_RES_OPT(true, P_MODE_SHARED);
        else P_RES_OPT(false, P_MODE_SHARED);
#undef P_RES_OPT
#undef P_RES
        DAT_LAUNCHED(plan);
        return DAT_OK;
    }
    const bool phases = form == P_PHASES;
    const bool halves = phases && p_halves(plan);
    a.n_whole = phases && !halves ? p_whole(plan, lamb != nullptr) : 0u;
    const unsigned grid = phases ? 2u * (unsigned)g->n_tiles - a.n_whole : a.n_items;
    if (phases && !identity) {
        rc = dat_norm_phase(plan, a.gp, a.scales_out, s);
        if (rc != DAT_OK) return rc;
    }
#define P_PHASES_GO(R, MODE, OPT, TWO, G, ENDS)                                                                     \
    do {                                                                                                            \
        if (MODE == P_MODE_IDENTITY) k_phase_quant<R, MODE, OPT, TWO, G, ENDS><<<grid, DAT_P_THREADS, 0, s>>>(a);   \
        else DAT_CUDA(plan, p_launch_after(k_phase_quant<R, MODE, OPT, TWO, G, ENDS>, grid, s, a));                 \
        DAT_LAUNCHED(plan);                                                                                         \
        if (TWO) {                                                                                                  \
            DAT_CUDA(plan, p_launch_after(k_phase_requant<R, OPT, G>, grid, s, a));                                 \
            DAT_LAUNCHED(plan);                                                                                     \
        }                                                                                                           \
        DAT_CUDA(plan, p_launch_after(k_phase_update<OPT, TWO, G>, grid, s, a));                                    \
    } while (0)
#define P_GO(R, MODE, OPT, TWO)                                                                                     \
    do {                                                                                                            \
        if (!phases) k_step_pipelined<R, MODE, OPT, TWO><<<grid, DAT_P_THREADS, 0, s>>>(a);                         \
        else if (halves) P_PHASES_GO(R, MODE, OPT, TWO, 1, MODE != P_MODE_IDENTITY ? P_ENDS_BY_M : P_ENDS_NONE);    \
        else if (plan->M >= P_ENDS_FROM) P_PHASES_GO(R, MODE, OPT, TWO, 2, MODE != P_MODE_IDENTITY ? P_ENDS_ALL : P_ENDS_NONE); \
        else P_PHASES_GO(R, MODE, OPT, TWO, 2, P_ENDS_NONE);                                                        \
    } while (0)
#define P_GO_OPT(R, MODE)                                                                                           \
    do {                                                                                                            \
        if (two) { if (lamb) P_GO(R, MODE, P_OPT_LAMB, true); else P_GO(R, MODE, P_OPT_MOMENTUM, true); }           \
        else if (lamb) P_GO(R, MODE, P_OPT_LAMB, false);                                                            \
        else P_GO(R, MODE, P_OPT_MOMENTUM, false);                                                                  \
    } while (0)
    if (identity) { if (lamb) P_GO(true, P_MODE_IDENTITY, P_OPT_LAMB, false); else P_GO(true, P_MODE_IDENTITY, P_OPT_MOMENTUM, false); }
    else if (per_worker && rng16) P_GO_OPT(true, P_MODE_PER_WORKER);
    else if (per_worker) P_GO_OPT(false, P_MODE_PER_WORKER);
    else if (rng16) P_GO_OPT(true, P_MODE_SHARED);
    else P_GO_OPT(false, P_MODE_SHARED);
#undef P_GO_OPT
#undef P_GO
    DAT_LAUNCHED(plan);
    return DAT_OK;
}

// dat_step on the layers of one group.
int dat_pipe_step_group(dat_plan_t *plan, int k, float *theta, float *mom, const float *const *grads, uint64_t seed, uint64_t step,
                        const dat_hparams_t *hp, cudaStream_t s)
{
    return p_launch(plan, theta, mom, nullptr, grads, seed, step, hp, nullptr, hp->lr, hp->c_l, hp->c_u, nullptr, nullptr, nullptr, s,
                    nullptr, nullptr, &plan->pipe->groups[(size_t)k]);
}

extern "C" int dat_step_pipelined(dat_plan_t *plan, float *theta, float *mom, const float *const *grads,
                                  uint64_t seed, uint64_t step, const dat_hparams_t *hp,
                                  int32_t *code_sum_out, float *layer_norms_out, float *scales_out, void *stream)
{
    int rc = dat_check_plan(plan);
    if (rc != DAT_OK) return rc;
    if (!theta || !mom || !hp) return DAT_ERR_ARG;
    return p_launch(plan, theta, mom, nullptr, grads, seed, step, hp, nullptr, hp->lr, hp->c_l, hp->c_u, code_sum_out,
                    layer_norms_out, scales_out, stream, nullptr, nullptr, nullptr, P_ONE_LAUNCH);
}

// dat_step: Steps 7, 9 and 12 in the form that p_resident and p_phases choose.
extern "C" int dat_step(dat_plan_t *plan, float *theta, float *mom, const float *const *grads,
                        uint64_t seed, uint64_t step, const dat_hparams_t *hp,
                        int32_t *code_sum_out, float *layer_norms_out, float *scales_out, void *stream)
{
    int rc = dat_check_plan(plan);
    if (rc != DAT_OK) return rc;
    if (!theta || !mom || !hp) return DAT_ERR_ARG;
    return p_launch(plan, theta, mom, nullptr, grads, seed, step, hp, nullptr, hp->lr, hp->c_l, hp->c_u, code_sum_out,
                    layer_norms_out, scales_out, stream);
}

// dat_step_passes: the same as one launch per phase, which wait for no epoch: the call can be recorded into a graph.
extern "C" int dat_step_passes(dat_plan_t *plan, float *theta, float *mom, const float *const *grads,
                               uint64_t seed, uint64_t step, const dat_hparams_t *hp,
                               int32_t *code_sum_out, float *layer_norms_out, float *scales_out, void *stream)
{
    int rc = dat_check_plan(plan);
    if (rc != DAT_OK) return rc;
    if (!theta || !mom || !hp) return DAT_ERR_ARG;
    if (plan->bits == 32 || plan->scale_mode != DAT_SCALE_SHARED_MAX) return DAT_ERR_UNSUPPORTED;
    return p_launch(plan, theta, mom, nullptr, grads, seed, step, hp, nullptr, hp->lr, hp->c_l, hp->c_u, code_sum_out,
                    layer_norms_out, scales_out, stream, nullptr, nullptr, nullptr, P_PHASES);
}

extern "C" int dat_step_lamb(dat_plan_t *plan, float *theta, float *mom, float *var, const float *const *grads,
                             uint64_t seed, uint64_t step, const dat_lamb_hparams_t *hp, int64_t t,
                             int32_t *code_sum_out, float *layer_norms_out, float *scales_out, void *stream)
{
    int rc = dat_check_plan(plan);
    if (rc != DAT_OK) return rc;
    if (!theta || !mom || !var || !hp || t < 1) return DAT_ERR_ARG;
    if (!(hp->beta1 > 0.0f && hp->beta1 < 1.0f && hp->beta2 > 0.0f && hp->beta2 < 1.0f)) return DAT_ERR_ARG;
    const LambConst c = dat_lamb_const(hp, t);
    return p_launch(plan, theta, mom, var, grads, seed, step, nullptr, &c, hp->lr, hp->c_l, hp->c_u, code_sum_out,
                    layer_norms_out, scales_out, stream);
}

extern "C" int dat_step_two_sided(dat_plan_t *plan, float *theta, float *mom, const float *const *grads,
                                  uint64_t seed, uint64_t step, const dat_hparams_t *hp, float *g_hat,
                                  int32_t *code_sum_out, float *layer_norms_out, float *scales_out,
                                  float *server_scales_out, void *stream)
{
    int rc = dat_check_plan(plan);
    if (rc != DAT_OK) return rc;
    if (!theta || !mom || !hp || !g_hat) return DAT_ERR_ARG;
    return p_launch(plan, theta, mom, nullptr, grads, seed, step, hp, nullptr, hp->lr, hp->c_l, hp->c_u, code_sum_out,
                    layer_norms_out, scales_out, stream, g_hat, server_scales_out);
}

extern "C" int dat_step_lamb_two_sided(dat_plan_t *plan, float *theta, float *mom, float *var, const float *const *grads,
                                       uint64_t seed, uint64_t step, const dat_lamb_hparams_t *hp, int64_t t, float *g_hat,
                                       int32_t *code_sum_out, float *layer_norms_out, float *scales_out,
                                       float *server_scales_out, void *stream)
{
    int rc = dat_check_plan(plan);
    if (rc != DAT_OK) return rc;
    if (!theta || !mom || !var || !hp || !g_hat || t < 1) return DAT_ERR_ARG;
    if (!(hp->beta1 > 0.0f && hp->beta1 < 1.0f && hp->beta2 > 0.0f && hp->beta2 < 1.0f)) return DAT_ERR_ARG;
    const LambConst c = dat_lamb_const(hp, t);
    return p_launch(plan, theta, mom, var, grads, seed, step, nullptr, &c, hp->lr, hp->c_l, hp->c_u, code_sum_out,
                    layer_norms_out, scales_out, stream, g_hat, server_scales_out);
}

// Test hook (see dat.h): the form of the plan's steps, whatever the rule says.
extern "C" int dat_plan_test_form(dat_plan_t *plan, int form)
{
    int rc = dat_check_plan(plan);
    if (rc != DAT_OK) return rc;
    if (!plan->pipe || form < P_BY_RULE || form > P_RESIDENT_LATE) return DAT_ERR_ARG;
    if (form >= P_RESIDENT && plan->bits == 32) form = P_PHASES;            // (no norms to wait for: no resident form)
    if (form >= P_RESIDENT && !plan->pipe->n_pieces) return DAT_ERR_ARG;
    plan->pipe->form = form;
    return DAT_OK;
}

// Test hook (see dat.h): a short wait limit, and a layer whose norm never completes in the next call.
extern "C" int dat_plan_test_stall(dat_plan_t *plan, int64_t wait_cycles, int64_t layer, void *stream)
{
    int rc = dat_check_plan(plan);
    if (rc != DAT_OK) return rc;
    PipeSchedule *g = plan->pipe;
    if (!g || !g->mem || wait_cycles < 0 || layer >= plan->h) return DAT_ERR_ARG;
    g->wait_cycles = wait_cycles ? (long long)wait_cycles : DAT_P_WAIT_CYCLES;
    g->form = (wait_cycles || layer >= 0) ? P_ONE_LAUNCH : P_BY_RULE;        // (the phases, which the rule may choose, do not wait)
    if (layer >= 0) {
        // a count that the layer's tiles cannot bring to T - 1: nobody becomes the layer's last tile
        static const uint32_t far = 0x40000000u;
        DAT_CUDA(plan, cudaMemcpyAsync(g->d_sync + 2 + layer, &far, sizeof far, cudaMemcpyHostToDevice, (cudaStream_t)stream));
        DAT_CUDA(plan, cudaStreamSynchronize((cudaStream_t)stream));
    }
    return DAT_OK;
}
