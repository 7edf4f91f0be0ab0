// The step in one launch whose CTAs stay: a CTA owns a piece of the vector (half a tile) through the phases N, Q, (R,)
// U and waits between them for its piece's layer.  Included by dat_pipeline.cu.
//
// A small problem is bound by latency: as a launch per phase each has its set-up and its first reads from cold, as items 256
// and 512 places apart its streams run through waves of nearly empty CTAs.  Here a phase ends with a count and a flag
// per layer, and theta and the moments are fetched into L2 under the norms.
//
// A CTA waits for CTAs of the same launch, and nothing promises that those have started: kernels of other streams may
// hold the SMs they need.  So a piece belongs to whom claims it: a CTA claims its own when it starts, and one that has
// waited R_PATIENCE for its layer's norms claims the layer's pieces that no CTA has begun, one after the other, and takes
// them along through all phases (a CTA that starts later finds its piece gone and ends).  Whoever claims a piece sums its
// norms before it waits again, and its levels before it waits for the levels of others.  So what a CTA waits for is always
// under way in CTAs that run, any number of running CTAs finish the step, and the limit of a wait is only spent on them.
// A CTA that is late has a body of its own: loops over a CTA's pieces around the one body cost registers there (150 thousand elements in 8 layers, M = 16: 24.7 us instead of 22.6).
#pragma once

#define R_CTAS 3                                  // per SM
#define R_MOST 512                                // pieces of a problem, at most: R_CTAS on each of 148 SMs are 444
#define R_PIECE (8 * DAT_P_THREADS)               // elements of a piece
#define R_PATIENCE 200000                         // cycles, about 100 us: the CTAs of an idle GPU start within 2
enum { R_GO = -1, R_STOP = -2, R_LATE = -3 };

// The sums of squares of a piece: 2 M units (worker, half piece), consecutive ones per warp, four 32-byte loads in
// flight per lane.  Units of one worker are added per lane first; the structure depends on M only.
__device__ __forceinline__ void r_norm_sums(const PArgs &a, const PipePart &pc, int64_t begin, double *s_unit)
{
    constexpr int W = DAT_P_THREADS / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, U = 2 * a.M;
    const int u0 = warp * U / W, u1 = (warp + 1) * U / W;
    const int64_t lo = pc.lo, hi = pc.hi;
    const bool inside = begin >= lo && begin + R_PIECE <= hi;
    double acc = 0.0;
    int run = u0;
#pragma unroll 1
    for (int u = u0; u < u1; ++u) {
        const float *g = a.gp.p[u >> 1];
        const int64_t e = begin + (u & 1) * (R_PIECE / 2) + 8 * lane;
        float v[4][8];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int64_t e0 = e + 256 * b;
            if (inside || (e0 >= lo && e0 + 8 <= hi)) {
                dat_ld8<EV_NORMAL>(g + e0, a.wide, v[b]);
            } else if (e0 < hi) {
                dat_load4_masked(g, e0, lo, hi, v[b]);
                dat_load4_masked(g, e0 + 4, lo, hi, v[b] + 4);
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j) v[b][j] = 0.0f;
            }
        }
        if ((u >> 1) != (run >> 1)) {
            acc = dat_warp_sum(acc);
            if (lane == 0) s_unit[run] = acc;
            acc = 0.0;
            run = u;
        }
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc = fma((double)v[b][j], (double)v[b][j], acc);
    }
    if (u1 > u0) {
        acc = dat_warp_sum(acc);
        if (lane == 0) s_unit[run] = acc;
    }
}

__device__ __forceinline__ int64_t r_begin(const PipePart &pc, int tile) { return (pc.lo & ~(int64_t)7) + (int64_t)tile * R_PIECE; }

// A piece as the parts of a tile know it (beside tile & 1, the half).
__device__ __forceinline__ PipePart r_tile(const PipePart &pc, int tile)
{
    PipePart pt = pc;
    pt.tile = tile >> 1;
    return pt;
}

// One thread: waits until the norms of the layer are published.  R_GO; R_STOP if the call has been given up; R_LATE after
// R_PATIENCE.
__device__ __forceinline__ int r_wait_norms(const PArgs &a, int layer)
{
    if (p_ld_acquire(a.readyN + layer) == a.epoch) return R_GO;
    const long long t0 = clock64();
    for (;;) {
        __nanosleep(32);
        if (p_ld_acquire(a.readyN + layer) == a.epoch) return R_GO;
        if (p_ld_acquire(a.abort_epoch) == a.epoch) return R_STOP;
        if (clock64() - t0 > R_PATIENCE) return R_LATE;
    }
}

// A warp: a piece of the layer that no CTA had begun, now the caller's, or -1.  The first `seen` pieces from the CTA's own
// on are known to be claimed.
__device__ __forceinline__ int r_take(const PArgs &a, const PipePart &pc, int &seen)
{
    const int lane = threadIdx.x & 31;
    while (seen < pc.T) {
        const bool in = seen + lane < pc.T;
        int t = pc.tile + (in ? seen + lane : 0);
        if (t >= pc.T) t -= pc.T;
        const unsigned some = __ballot_sync(0xFFFFFFFFu, in && __ldcg(a.claim + pc.tb + t) != a.epoch);
        if (!some) { seen += 32; continue; }
        const int first = __ffs(some) - 1;
        uint32_t had = 0;
        if (lane == first) had = atomicExch(a.claim + pc.tb + t, a.epoch);
        had = __shfl_sync(0xFFFFFFFFu, had, first);
        t = __shfl_sync(0xFFFFFFFFu, t, first);
        seen += first + 1;
        if (had != a.epoch) return t;
    }
    return -1;
}

// The rest of the step of a CTA that has waited for R_PATIENCE, its own piece's norms being counted in: takes the pieces of
// its layer that no CTA has begun, and goes through the phases with them and its own one.
template <bool RNG16, int MODE, int OPT, bool TWO>
__device__ __forceinline__ void r_late(const PArgs &a, const PipePart &pc, double *s_unit, float *s_norm, double *s_red, float2 *s_fac, int16_t *s_own,
                                       int *s_ctl)
{
    const int warp = threadIdx.x >> 5;
    int n = 1, seen = 1;
    if (threadIdx.x == 0) s_own[0] = (int16_t)pc.tile;
#pragma unroll 1
    for (;;) {
        __syncthreads();
        if (warp == 0) {
            const int t = r_take(a, pc, seen);
            if (threadIdx.x == 0) s_own[n] = (int16_t)t;
        }
        for (int u = threadIdx.x; u < 2 * a.M; u += DAT_P_THREADS) s_unit[u] = 0.0;
        __syncthreads();
        const int tile = s_own[n];
        if (tile < 0) break;
        ++n;
        r_norm_sums(a, pc, r_begin(pc, tile), s_unit);
        __syncthreads();
        if (warp == 0) {
            for (int i = threadIdx.x; i < a.M; i += 32) a.partN[((int64_t)pc.tb + tile) * a.M + i] = s_unit[2 * i] + s_unit[2 * i + 1];
            __syncwarp();
            if (threadIdx.x == 0) s_ctl[0] = dat_count_in(a.cntN + pc.layer, (uint32_t)pc.T);
        }
        __syncthreads();
        if (s_ctl[0]) p_norm_finish<MODE>(a, pc, s_norm);
    }
    // Thread 0: waits for the layer; every thread: whether to go on.
    auto go = [&](const uint32_t *ready) -> bool {
        if (threadIdx.x == 0) s_ctl[1] = p_poll<32>(a, ready + pc.layer);
        __syncthreads();
        return s_ctl[1] != 0;
    };
    if (!go(a.readyN)) return;
#pragma unroll 1
    for (int phase = 0; phase < (TWO ? 2 : 1); ++phase) {        // Q, R
        const bool server = TWO && phase == 0;
#pragma unroll 1
        for (int k = 0; k < n; ++k) {
            const int tile = s_own[k];
            if (!TWO || server) p_part_quant<RNG16, MODE, OPT, TWO, 1, P_ENDS_ALL>(a, r_tile(pc, tile), tile & 1, s_red, s_fac);
            else p_part_requant<RNG16, OPT, 1>(a, r_tile(pc, tile), tile & 1, s_red);
            __syncthreads();
            if (threadIdx.x == 0) {
                if (server) a.partR[pc.tb + tile] = p_warps_sum(s_red);
                else p_quant_sums(a, pc.tb + tile, s_red);
                s_ctl[0] = dat_count_in((server ? a.cntR : a.cntQ) + pc.layer, (uint32_t)pc.T);
            }
            __syncthreads();
            if (s_ctl[0]) { if (server) p_server_finish(a, pc, s_red); else p_quant_finish(a, pc, s_red); }
        }
        if (!go(server ? a.readyR : a.readyQ)) return;
    }
#pragma unroll 1
    for (int k = 0; k < n; ++k) p_part_update<OPT, 1>(a, r_tile(pc, s_own[k]), s_own[k] & 1);
}

template <bool RNG16, int MODE, int OPT, bool TWO>
__global__ void __launch_bounds__(DAT_P_THREADS, R_CTAS)
k_step_resident(const __grid_constant__ PArgs a)
{
    __shared__ double s_unit[2 * DAT_MAX_WORKERS], s_red[2 * (DAT_P_THREADS / 32)];
    __shared__ float s_norm[DAT_MAX_WORKERS];
    __shared__ float2 s_fac[MODE == P_MODE_PER_WORKER ? DAT_MAX_WORKERS : 1];
    __shared__ int16_t s_own[R_MOST + 1];          // (r_late) the CTA's pieces by their number in the layer
    __shared__ int s_ctl[2];
    const int warp = threadIdx.x >> 5, M = a.M;
    PipePart pc;
    {
        const uint4 *src = reinterpret_cast<const uint4 *>(a.parts + blockIdx.x);
        reinterpret_cast<uint4 *>(&pc)[0] = __ldg(src);
        reinterpret_cast<uint4 *>(&pc)[1] = __ldg(src + 1);
    }
    const int64_t begin = r_begin(pc, pc.tile), e0 = begin + 8 * threadIdx.x, slot = (int64_t)pc.tb + pc.tile;
    if (!P_CHECK(a, pc.layer >= 0 && pc.layer < a.h && pc.tile >= 0 && pc.tile < pc.T && pc.T <= R_MOST && pc.tb >= 0 &&
                        (int64_t)pc.tb + pc.T <= 2 * a.n_tiles && pc.lo >= 0 && pc.lo < pc.hi && pc.hi <= a.d && r_begin(pc, pc.T - 1) < pc.hi)) return;
    // asked for before the norms are read, looked at after them (compared at once, the first warp waits for the answer)
    uint32_t claimed = 0;
    if (threadIdx.x == 0) claimed = atomicExch(a.claim + slot, a.epoch);
    // The piece's sums being written, thread 0 counts it in; the layer's last one finishes the layer.  Then the CTA waits until
    // the layer is published.
    auto phase_end = [&](uint32_t *count, const uint32_t *ready, auto &&finish) -> bool {
        if (threadIdx.x == 0) s_ctl[0] = dat_count_in(count + pc.layer, (uint32_t)pc.T);
        __syncthreads();
        if (s_ctl[0]) finish();
        if (threadIdx.x == 0) s_ctl[1] = p_poll<32>(a, ready + pc.layer);
        __syncthreads();
        return s_ctl[1] != 0;
    };

    if (e0 < pc.hi) {                              // what the next phase reads beside the gradients
        asm volatile("prefetch.global.L2 [%0];" :: "l"(a.theta + e0));
        asm volatile("prefetch.global.L2 [%0];" :: "l"(a.mom + e0));
        if (OPT == P_OPT_LAMB) asm volatile("prefetch.global.L2 [%0];" :: "l"(a.var + e0));
    }
    for (int u = threadIdx.x; u < 2 * M; u += DAT_P_THREADS) s_unit[u] = 0.0;
    __syncthreads();
    r_norm_sums(a, pc, begin, s_unit);
    __syncthreads();
    if (warp == 0) {
        const bool mine = __shfl_sync(0xFFFFFFFFu, claimed, 0) != a.epoch;
        if (mine)
            for (int i = threadIdx.x; i < M; i += 32) a.partN[slot * M + i] = s_unit[2 * i] + s_unit[2 * i + 1];
        __syncwarp();
        if (threadIdx.x == 0) s_ctl[0] = mine ? (int)dat_count_in(a.cntN + pc.layer, (uint32_t)pc.T) : R_STOP;
    }
    __syncthreads();
    if (s_ctl[0] == R_STOP) return;                // the piece is another CTA's
    if (s_ctl[0]) p_norm_finish<MODE>(a, pc, s_norm);
    if (threadIdx.x == 0) s_ctl[1] = r_wait_norms(a, pc.layer);
    __syncthreads();
    if (s_ctl[1] == R_STOP) return;
    if (s_ctl[1] == R_LATE) {
        r_late<RNG16, MODE, OPT, TWO>(a, pc, s_unit, s_norm, s_red, s_fac, s_own, s_ctl);
        return;
    }

    p_part_quant<RNG16, MODE, OPT, TWO, 1, P_ENDS_ALL>(a, r_tile(pc, pc.tile), pc.tile & 1, s_red, s_fac);
    __syncthreads();
    if (TWO) {
        if (threadIdx.x == 0) a.partR[slot] = p_warps_sum(s_red);
        if (!phase_end(a.cntR, a.readyR, [&] { p_server_finish(a, pc, s_red); })) return;
        p_part_requant<RNG16, OPT, 1>(a, r_tile(pc, pc.tile), pc.tile & 1, s_red);
        __syncthreads();
    }
    if (threadIdx.x == 0) p_quant_sums(a, slot, s_red);
    if (!phase_end(a.cntQ, a.readyQ, [&] { p_quant_finish(a, pc, s_red); })) return;
    p_part_update<OPT, 1>(a, r_tile(pc, pc.tile), pc.tile & 1);
}
