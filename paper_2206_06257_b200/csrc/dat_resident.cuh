// The step in one launch whose CTAs all stay: a CTA owns a piece of the vector (half a tile) through the phases N, Q, (R,)
// U and waits between them for its piece's layer.  Included by dat_pipeline.cu.
//
// A small problem is bound by latency: as a launch per phase each has its set-up and its first reads from cold, as items 256
// and 512 places apart its streams run through waves of nearly empty CTAs.  Here a phase ends with a count and a flag
// per layer, theta and the moments are fetched into L2 under the norms, and what a thread reads again (g_hat, m', theta) it has
// written itself, so the update's reads are under way while it waits.
//
// A CTA waits for CTAs of the same launch, so all of them must be resident: the launch is a cooperative one, of no more
// than R_CTAS per SM, which the launch bounds guarantee.
#pragma once

#define R_CTAS 3
#define R_PIECE (8 * DAT_P_THREADS)               // elements of a piece

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

template <bool RNG16, int MODE, int OPT, bool TWO>
__global__ void __launch_bounds__(DAT_P_THREADS, R_CTAS)
k_step_resident(const __grid_constant__ PArgs a)
{
    __shared__ double s_unit[2 * DAT_MAX_WORKERS], s_red[2 * (DAT_P_THREADS / 32)];
    __shared__ float s_norm[DAT_MAX_WORKERS];
    __shared__ float2 s_fac[MODE == P_MODE_PER_WORKER ? DAT_MAX_WORKERS : 1];
    __shared__ bool s_last, s_go;
    const int warp = threadIdx.x >> 5, M = a.M;
    PipePart pc;
    {
        const uint4 *src = reinterpret_cast<const uint4 *>(a.parts + blockIdx.x);
        reinterpret_cast<uint4 *>(&pc)[0] = __ldg(src);
        reinterpret_cast<uint4 *>(&pc)[1] = __ldg(src + 1);
    }
    const int64_t begin = (pc.lo & ~(int64_t)7) + (int64_t)pc.tile * R_PIECE, e0 = begin + 8 * threadIdx.x, slot = (int64_t)pc.tb + pc.tile;
    if (!P_CHECK(a, pc.layer >= 0 && pc.layer < a.h && pc.tile >= 0 && pc.tile < pc.T && pc.tb >= 0 && slot < 2 * a.n_tiles && pc.lo >= 0 &&
                        pc.lo < pc.hi && pc.hi <= a.d && begin < pc.hi)) return;
    PipePart pt = pc;                              // the piece as the parts of a tile know it
    pt.tile = pc.tile >> 1;
    const int half = pc.tile & 1;
    // Thread 0, the piece's sums being written: counts the piece in; the layer's last one finishes the layer.  Then the CTA
    // waits until the layer is published.
    auto phase_end = [&](uint32_t *count, const uint32_t *ready, auto &&finish) -> bool {
        if (threadIdx.x == 0) s_last = dat_count_in(count + pc.layer, (uint32_t)pc.T);
        __syncthreads();
        if (s_last) finish();
        if (threadIdx.x == 0) s_go = p_poll<32>(a, ready + pc.layer);
        __syncthreads();
        return s_go;
    };

    if (e0 < pc.hi) {                          // what the next phase reads beside the gradients
        asm volatile("prefetch.global.L2 [%0];" :: "l"(a.theta + e0));
        asm volatile("prefetch.global.L2 [%0];" :: "l"(a.mom + e0));
        if (OPT == P_OPT_LAMB) asm volatile("prefetch.global.L2 [%0];" :: "l"(a.var + e0));
    }
    for (int u = threadIdx.x; u < 2 * M; u += DAT_P_THREADS) s_unit[u] = 0.0;
    __syncthreads();
    r_norm_sums(a, pc, begin, s_unit);
    __syncthreads();
    if (warp == 0) {
        for (int i = threadIdx.x; i < M; i += 32) a.partN[slot * M + i] = s_unit[2 * i] + s_unit[2 * i + 1];
        __syncwarp();
    }
    if (!phase_end(a.cntN, a.readyN, [&] { p_norm_finish<MODE>(a, pc, s_norm); })) return;
    p_part_quant<RNG16, MODE, OPT, TWO, 1>(a, pt, half, s_red, s_fac);
    __syncthreads();
    if (TWO) {
        if (threadIdx.x == 0) a.partR[slot] = p_warps_sum(s_red);
        if (!phase_end(a.cntR, a.readyR, [&] { p_server_finish(a, pc, s_red); })) return;
        p_part_requant<RNG16, OPT, 1>(a, pt, half, s_red);
        __syncthreads();
    }
    if (threadIdx.x == 0) p_quant_sums(a, slot, s_red);
    if (!phase_end(a.cntQ, a.readyQ, [&] { p_quant_finish(a, pc, s_red); })) return;
    p_part_update<OPT, 1>(a, pt, half);
}
